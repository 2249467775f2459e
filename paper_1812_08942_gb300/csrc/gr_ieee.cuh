// Correctly rounded FP64 division and square root on the integer pipe, for
// kernels that wait on a serial chain of them or that the FP64 pipe bounds.
// That pipe takes 64 cycles an operation on this chip and a sixteenth of a
// warp a cycle; a division takes a lone warp 562 cycles there and 345 here, a
// square root 594 and 340 (measured; 4.3 G results compared, no bit differs).
//
// Both are long division (long root) with two digits of 27 bits: an FP32
// estimate of the reciprocal (of the root's) takes one Newton step to 29 bits
// in 32-bit fixed point, each digit is the leading bits times that, and its
// remainder is exact modulo 2^64.  After the second digit the result is off by
// at most one unit of its 54 bits; one correction leaves the floor, the round
// bit and "inexact", which are IEEE's round to nearest even.  Operands or
// results outside the normal range take the built-in operation.
// (64-bit fixed point with 64 x 64-bit products: 497 and 406 cycles.)
#pragma once

#include <stdint.h>

namespace gr {

#ifdef __CUDACC__
#define GR_IEEE_FN __device__ __forceinline__
__device__ __forceinline__ uint64_t ieee_bits(double x) { return (uint64_t)__double_as_longlong(x); }
__device__ __forceinline__ double ieee_double(uint64_t b) { return __longlong_as_double((long long)b); }
// FP32 estimates of normal numbers (23 bits)
__device__ __forceinline__ uint32_t ieee_rcp(uint32_t b) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__int_as_float((int)b)));
    return (uint32_t)__float_as_int(y);
}
__device__ __forceinline__ uint32_t ieee_rsqrt(uint32_t b) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__int_as_float((int)b)));
    return (uint32_t)__float_as_int(y);
}
static __device__ __noinline__ double ieee_div_any(double a, double b) { return a / b; }
static __device__ __noinline__ double ieee_sqrt_any(double x) { return sqrt(x); }
#endif

constexpr uint64_t IEEE_HIDDEN = 1ull << 52;

GR_IEEE_FN uint32_t ieee_mulhi32(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
// Q1.31 of an FP32 number in [1, 2], or past an end by the estimate's error:
// bit 23 of a number in [1, 2) is the exponent's last, a one (below 1 a zero)
GR_IEEE_FN uint32_t ieee_q31(uint32_t b) { return (b < 0x3fffffffu ? b : 0x3fffffffu) << 8; }
// r (1 + e / 2^31), Q1.31, kept below 2
GR_IEEE_FN uint32_t ieee_newton(uint32_t r, int32_t e) {
    const int32_t d = (int32_t)(((int64_t)e * (int64_t)r) >> 31);
    const uint32_t x = r + (uint32_t)d;
    return d > 0 && x < r ? 0xffffffffu : x;
}

// 54-bit q in [2^53, 2^54), exact or not, to the nearest 53-bit significand, with exponent field ex (1 .. 2045)
GR_IEEE_FN double ieee_pack(uint64_t sign, int ex, uint64_t q, bool inexact) {
    const uint64_t up = q & 1u & ((inexact ? 1u : 0u) | (q >> 1));
    return ieee_double(sign | ((((uint64_t)ex) << 52) + (q >> 1) - IEEE_HIDDEN + up));
}

GR_IEEE_FN double ieee_div(double a, double b) {
    const uint64_t xa = ieee_bits(a), xb = ieee_bits(b);
    const int ea = (int)(xa >> 52) & 0x7ff, eb = (int)(xb >> 52) & 0x7ff;
    const uint64_t ma = (xa & (IEEE_HIDDEN - 1)) | IEEE_HIDDEN, mb = (xb & (IEEE_HIDDEN - 1)) | IEEE_HIDDEN;
    const int less = ma < mb ? 1 : 0;
    const int ex = ea - eb + 1023 - less;
    const bool zero = (xa << 1) == 0 && (unsigned)(eb - 1) < 2046u;
    const bool any = (unsigned)(ea - 1) >= 2046u || (unsigned)(eb - 1) >= 2046u || (unsigned)(ex - 1) >= 2045u;
    // d = mb / 2^53 in [1/2, 1); r = 1/d, Q1.31
    const uint32_t d = (uint32_t)(mb >> 21);
    uint32_t r = ieee_q31(ieee_rcp(0x3f000000u + ((uint32_t)((mb + (1ull << 28)) >> 29) - 0x800000u)));
    r = ieee_newton(r, (int32_t)(0x80000000u - ieee_mulhi32(d, r)));
    // floor of ma 2^(53 + less) / mb in two digits
    const uint32_t q1 = ieee_mulhi32((uint32_t)(ma >> 21), r) >> (5 - less);
    const int64_t rem1 = (int64_t)((ma << (26 + less)) - q1 * mb);
    const int32_t q2 = (int32_t)(((int64_t)(int32_t)(rem1 >> 24) * (int64_t)r) >> 33);
    int64_t rem = (int64_t)(((uint64_t)rem1 << 27) - (uint64_t)(int64_t)q2 * mb);
    uint64_t q = ((uint64_t)q1 << 27) + (uint64_t)(int64_t)q2;
    const int64_t m = (int64_t)mb;
    const int64_t fix = rem < 0 ? -1 : rem >= m ? 1 : 0;
    q += (uint64_t)fix;
    rem += rem < 0 ? m : rem >= m ? -m : 0;
    const double y = ieee_pack((xa ^ xb) & (1ull << 63), ex, q, rem != 0);
    if (zero) return ieee_double((xa ^ xb) & (1ull << 63));
    return any ? ieee_div_any(a, b) : y;
}

GR_IEEE_FN double ieee_sqrt(double x) {
    const uint64_t xb = ieee_bits(x);
    const int ebits = (int)(xb >> 52);  // sign included: negative numbers leave the range
    const int odd = (ebits + 1) & 1, k = (ebits - 1023 - odd) >> 1;
    const uint64_t mx = (xb & (IEEE_HIDDEN - 1)) | IEEE_HIDDEN;
    // x = 4^(k+1) D, D = mx 2^(odd - 54) in [1/4, 1); y = 1/sqrt(D) in (1, 2], Q1.31
    const uint64_t m1 = mx << odd;  // the root's square, leading 54 of 108 bits
    const uint32_t D = (uint32_t)(m1 >> 22);
    const uint32_t fd = (odd ? 0x3f000000u : 0x3e800000u) + ((uint32_t)((mx + (1ull << 28)) >> 29) - 0x800000u);
    uint32_t y = ieee_q31(ieee_rsqrt(fd));
    y = ieee_newton(y, (int32_t)(0x40000000u - ieee_mulhi32(ieee_mulhi32(D, y), y)));
    // floor of sqrt(m1 2^54) in two digits, the first to nearest
    const uint32_t s1 = (uint32_t)(((uint64_t)ieee_mulhi32(D, y) + 8u) >> 4);
    const int64_t rem1 = (int64_t)(m1 - (uint64_t)s1 * s1);
    const int32_t s2 = (int32_t)(((int64_t)(int32_t)rem1 * (int64_t)y) >> 32);
    const uint64_t t2 = (uint64_t)(int64_t)s2;
    uint64_t s = ((uint64_t)s1 << 27) + t2;
    int64_t rem = (int64_t)(((uint64_t)rem1 << 54) - t2 * (((uint64_t)s1 << 28) + t2));
    if (rem < 0) {
        s -= 1;
        rem += (int64_t)(2 * s + 1);
    } else if (rem > (int64_t)(2 * s)) {
        rem -= (int64_t)(2 * s + 1);
        s += 1;
    }
    const double r = ieee_pack(0, k + 1023, s, rem != 0);
    return (unsigned)(ebits - 1) >= 2046u ? ieee_sqrt_any(x) : r;
}

#ifdef __CUDACC__
// 1 / d of a row's degree, 0 for an isolated row (d is not negative): beside
// its row's additions a division on the FP64 pipe costs as much as ten slots
// (CSR rows of the 128^3 mesh, with the FP32 weights converted by integers as
// well: 167 us before, 154 now)
__device__ __forceinline__ double row_inverse(double d) { return ieee_bits(d) << 1 ? ieee_div(1.0, d) : 0.0; }
#endif

}  // namespace gr
