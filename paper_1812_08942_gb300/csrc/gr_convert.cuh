#pragma once

namespace gr {

// (the host's forms are the test's, which defines GR_CONVERT_FN)
#ifdef __CUDACC__
#define GR_CONVERT_FN __device__ __forceinline__
__device__ __forceinline__ unsigned convert_high(double x) { return (unsigned)__double2hiint(x); }
__device__ __forceinline__ unsigned convert_low(double x) { return (unsigned)__double2loint(x); }
__device__ __forceinline__ unsigned convert_bits(float x) { return (unsigned)__float_as_int(x); }
__device__ __forceinline__ float convert_float(unsigned b) { return __int_as_float((int)b); }
__device__ __forceinline__ double convert_double(unsigned high, unsigned low) { return __hiloint2double((int)high, (int)low); }
#endif

// FP64 <-> FP32 conversions on the integer pipe.  The conversion unit runs at
// the FP64 pipe's rate (measured: 626 G a second against 530 G FP64
// operations and about 20 T integer ones), and a conversion in a branch costs
// its time even where no lane takes the branch, so every range is handled
// with integer operations.  Results are the hardware's, bit for bit (NaN: some NaN).
// To nearest even: the 53-bit significand is cut to FP32's 24 bits (fewer for
// a subnormal result) and the remainder's carry added.
GR_CONVERT_FN float f64_to_f32(double x) {
    const unsigned hi = convert_high(x), lo = convert_low(x);
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
    return convert_float(b | sign);
}
// exact: the exponent rebiased, a subnormal number scaled to a normal one first
GR_CONVERT_FN double f32_to_f64(float x) {
    const unsigned bx = convert_bits(x), ex = (bx >> 23) & 0xffu, sign = bx & 0x80000000u;
    const unsigned b = (ex ? bx : convert_bits(x * 0x1p64f)) & 0x7fffffffu;
    const unsigned bias = ex ? (ex == 0xffu ? 0x70000000u : 0x38000000u) : 0x34000000u;
    return convert_double(sign | (b ? (b >> 3) + bias : 0u), b << 29);
}

}  // namespace gr
