"""FP64 <-> FP32 conversions in integer arithmetic (gr_convert.cuh) against the
machine's own, bit for bit (NaN: some NaN): every exponent, ties and their
neighbours, carries into the exponent, overflow, subnormal results, zeros."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DRIVER = r"""
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
namespace gr {
#define GR_CONVERT_FN static inline
static inline uint64_t bits64(double x) { uint64_t b; memcpy(&b, &x, 8); return b; }
static inline unsigned convert_high(double x) { return (unsigned)(bits64(x) >> 32); }
static inline unsigned convert_low(double x) { return (unsigned)bits64(x); }
static inline unsigned convert_bits(float x) { unsigned b; memcpy(&b, &x, 4); return b; }
static inline float convert_float(unsigned b) { float x; memcpy(&x, &b, 4); return x; }
static inline double convert_double(unsigned h, unsigned l) {
    const uint64_t b = (uint64_t)h << 32 | l;
    double x;
    memcpy(&x, &b, 8);
    return x;
}
}
#include "gr_convert.cuh"
using namespace gr;
static long bad = 0;
static void narrow(uint64_t b) {
    for (uint64_t s : {0ull, 1ull << 63}) {
        const double x = convert_double((unsigned)((b | s) >> 32), (unsigned)b);
        const float y = f64_to_f32(x), z = (float)x;
        if (convert_bits(y) != convert_bits(z) && !(y != y && z != z)) ++bad;
    }
}
static void widen(unsigned b) {
    const float x = convert_float(b);
    const double y = f32_to_f64(x), z = (double)x;
    if (bits64(y) != bits64(z) && !(y != y && z != z)) ++bad;
}
int main() {
    std::mt19937_64 R(3);
    typedef unsigned long long u64;
    const u64 M = (1ull << 52) - 1;
    for (uint64_t e = 0; e < 2048; ++e) {
        // significands around every place where the cut may fall: 2^k - 1, 2^k, 2^k + 1, above even and odd bits
        for (int k = 0; k <= 52; ++k)
            for (u64 top : {0ull, 1ull << 29, 3ull << 29, M, (u64)R() & M})
                for (int d = -1; d <= 1; ++d) {
                    const uint64_t low = ((1ull << k) + (uint64_t)(int64_t)d) & M;
                    narrow(e << 52 | ((top & ~((k < 52 ? 1ull << (k + 1) : 0) - 1)) & M) | low);
                    narrow(e << 52 | ((top | low) & M));
                }
        for (int i = 0; i < 2000; ++i) narrow(e << 52 | (R() & M));
    }
    for (unsigned b = 0; b < 1u << 24; ++b) widen(b), widen(b | 1u << 31);
    for (unsigned e = 0; e < 256; ++e)
        for (int i = 0; i < 2000; ++i) widen(e << 23 | (unsigned)(R() & 0x7fffff) | (unsigned)(R() & 1) << 31);
    for (unsigned b : {0x7f7fffffu, 0x7f800000u, 0xff800000u, 0x7f800001u, 0x7fc00000u, 0xffffffffu}) widen(b);
    printf("%ld\n", bad);
    return 0;
}
"""


def test_conversions_are_the_machines(tmp_path):
    src, exe = tmp_path / "convert.cpp", tmp_path / "convert"
    src.write_text(DRIVER)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_1812_08942_gb300", "csrc"), "-o",
                    str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.strip() == "0"
