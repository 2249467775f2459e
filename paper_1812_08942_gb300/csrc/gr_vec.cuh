// Row-chunk access to row-major n x K vector blocks of double, float or
// bfloat16.  A row is split into G chunks of E elements; one lane owns one
// chunk and moves it with a single 16-byte (or 8-byte) access.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

namespace gr {

template <typename T>
struct AccOf { using type = float; };
template <>
struct AccOf<double> { using type = double; };

// FP64 <-> FP32 conversions on the integer pipe.  The conversion unit runs at
// the FP64 pipe's rate (measured: 626 G a second against 530 G FP64
// operations and about 20 T integer ones), and a conversion in a branch costs
// its time even where no lane takes the branch, so every range is handled
// with integer operations.  Results are the hardware's, bit for bit (NaN: some NaN).
// To nearest even: the 53-bit significand is cut to FP32's 24 bits (fewer for
// a subnormal result) and the remainder's carry added.
__device__ __forceinline__ float f64_to_f32(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned ex = (hi >> 20) & 0x7ffu, sign = hi & 0x80000000u;
    unsigned b;
    if (ex - 897u <= 253u) {
        b = ((ex - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
        b += ((lo & 0x1fffffffu) + 0x0fffffffu + (b & 1u)) >> 29;
    } else if (ex > 896u) {  // too large, infinite or NaN
        b = 0x7f800000u | ((ex == 0x7ffu && ((hi & 0xfffffu) | lo)) ? 0x400000u : 0u);
    } else if (ex >= 872u) {  // subnormal result: the significand in units of 2^-149
        const unsigned long long m = (1ull << 52) | ((unsigned long long)(hi & 0xfffffu) << 32) | lo;
        const int sh = 29 + (int)(897u - ex);  // 30 .. 54
        const unsigned long long rem = m & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
        b = (unsigned)(m >> sh);
        b += (rem > half || (rem == half && (b & 1u))) ? 1u : 0u;
    } else {
        b = 0u;
    }
    return __int_as_float((int)(b | sign));
}
// exact: the exponent rebiased, a subnormal number scaled to a normal one first
__device__ __forceinline__ double f32_to_f64(float x) {
    const unsigned bx = (unsigned)__float_as_int(x), ex = (bx >> 23) & 0xffu, sign = bx & 0x80000000u;
    const unsigned b = (ex ? bx : (unsigned)__float_as_int(x * 0x1p64f)) & 0x7fffffffu;
    const unsigned bias = ex ? (ex == 0xffu ? 0x70000000u : 0x38000000u) : 0x34000000u;
    return __hiloint2double((int)(sign | (b ? (b >> 3) + bias : 0u)), (int)(b << 29));
}

constexpr int next_pow2_c(int x) { return x <= 1 ? 1 : 2 * next_pow2_c((x + 1) / 2); }

template <typename T, int K>
struct RowLayout {
    static constexpr int RB = K * (int)sizeof(T);           // row bytes
    static constexpr int CB = (RB % 16 == 0) ? 16 : 8;       // chunk bytes
    static constexpr int E = CB / (int)sizeof(T);            // elements per chunk
    static constexpr int G = K / E;                          // chunks per row
    static constexpr int GP = next_pow2_c(G);                // lanes reserved per row
    static_assert(RB % 8 == 0, "row must be a multiple of 8 bytes");
    static_assert(G <= 32, "row too wide");
};

template <typename T, int E>
__device__ __forceinline__ void load_chunk(const T* __restrict__ p, typename AccOf<T>::type (&x)[E]);

template <>
__device__ __forceinline__ void load_chunk<float, 4>(const float* __restrict__ p, float (&x)[4]) {
    float4 v = __ldg(reinterpret_cast<const float4*>(p));
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
}
template <>
__device__ __forceinline__ void load_chunk<float, 2>(const float* __restrict__ p, float (&x)[2]) {
    float2 v = __ldg(reinterpret_cast<const float2*>(p));
    x[0] = v.x; x[1] = v.y;
}
template <>
__device__ __forceinline__ void load_chunk<double, 2>(const double* __restrict__ p, double (&x)[2]) {
    double2 v = __ldg(reinterpret_cast<const double2*>(p));
    x[0] = v.x; x[1] = v.y;
}
template <>
__device__ __forceinline__ void load_chunk<double, 1>(const double* __restrict__ p, double (&x)[1]) {
    x[0] = __ldg(p);
}
template <>
__device__ __forceinline__ void load_chunk<__nv_bfloat16, 8>(const __nv_bfloat16* __restrict__ p,
                                                            float (&x)[8]) {
    uint4 v = __ldg(reinterpret_cast<const uint4*>(p));
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float2 f = __bfloat1622float2(h[i]);
        x[2 * i] = f.x;
        x[2 * i + 1] = f.y;
    }
}
template <>
__device__ __forceinline__ void load_chunk<__nv_bfloat16, 4>(const __nv_bfloat16* __restrict__ p,
                                                            float (&x)[4]) {
    uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        float2 f = __bfloat1622float2(h[i]);
        x[2 * i] = f.x;
        x[2 * i + 1] = f.y;
    }
}

// Round to storage, store, and hand back the stored value in the accumulator
// type (so statistics describe exactly what the next sweep reads).
template <typename T, int E>
__device__ __forceinline__ void store_chunk(T* __restrict__ p, typename AccOf<T>::type (&x)[E]);

template <>
__device__ __forceinline__ void store_chunk<float, 4>(float* __restrict__ p, float (&x)[4]) {
    *reinterpret_cast<float4*>(p) = make_float4(x[0], x[1], x[2], x[3]);
}
template <>
__device__ __forceinline__ void store_chunk<float, 2>(float* __restrict__ p, float (&x)[2]) {
    *reinterpret_cast<float2*>(p) = make_float2(x[0], x[1]);
}
template <>
__device__ __forceinline__ void store_chunk<double, 2>(double* __restrict__ p, double (&x)[2]) {
    *reinterpret_cast<double2*>(p) = make_double2(x[0], x[1]);
}
template <>
__device__ __forceinline__ void store_chunk<double, 1>(double* __restrict__ p, double (&x)[1]) {
    *p = x[0];
}
template <>
__device__ __forceinline__ void store_chunk<__nv_bfloat16, 8>(__nv_bfloat16* __restrict__ p,
                                                             float (&x)[8]) {
    uint4 v;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        h[i] = __floats2bfloat162_rn(x[2 * i], x[2 * i + 1]);
        float2 f = __bfloat1622float2(h[i]);
        x[2 * i] = f.x;
        x[2 * i + 1] = f.y;
    }
    *reinterpret_cast<uint4*>(p) = v;
}
template <>
__device__ __forceinline__ void store_chunk<__nv_bfloat16, 4>(__nv_bfloat16* __restrict__ p,
                                                             float (&x)[4]) {
    uint2 v;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&v);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        h[i] = __floats2bfloat162_rn(x[2 * i], x[2 * i + 1]);
        float2 f = __bfloat1622float2(h[i]);
        x[2 * i] = f.x;
        x[2 * i + 1] = f.y;
    }
    *reinterpret_cast<uint2*>(p) = v;
}

}  // namespace gr
