"""FP64 division and square root in integer arithmetic (gr_ieee.cuh) against the
machine's own, bit for bit: significands of every shape, quotients and roots
that are exact or nearly so, every exponent, and FP32 estimates off by as much
as the device's may be (one unit for a reciprocal, two for a root's)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DRIVER = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
static std::mt19937_64 R(7);
static int jitter = 0;
namespace gr {
#define GR_IEEE_FN static inline
static inline uint64_t ieee_bits(double x) { uint64_t b; memcpy(&b, &x, 8); return b; }
static inline double ieee_double(uint64_t b) { double x; memcpy(&x, &b, 8); return x; }
static inline uint32_t estimate(uint32_t b, bool root) {
    float f;
    memcpy(&f, &b, 4);
    f = (float)(1.0 / (root ? sqrt((double)f) : (double)f));
    memcpy(&b, &f, 4);
    const int w = root ? 2 : 1;
    return jitter ? b + (int)(R() % (2 * w + 1)) - w : b;
}
static inline uint32_t ieee_rcp(uint32_t b) { return estimate(b, false); }
static inline uint32_t ieee_rsqrt(uint32_t b) { return estimate(b, true); }
static inline double ieee_div_any(double a, double b) { return a / b; }
static inline double ieee_sqrt_any(double x) { return sqrt(x); }
}
#include "gr_ieee.cuh"
using namespace gr;
static long bad = 0;
static void same(double x, double y) { if (ieee_bits(x) != ieee_bits(y) && !(x != x && y != y)) ++bad; }
static double draw() {
    uint64_t m = R() & (IEEE_HIDDEN - 1);
    int e = 1023;
    switch (R() % 6) {
        case 0: break;
        case 1: e += (int)(R() % 41) - 20; break;
        case 2: e = (int)(R() % 2048); break;
        case 3: m = R() & 1 ? R() & 255 : IEEE_HIDDEN - 1 - (R() & 255); break;
        case 4: e += (int)(R() % 3) - 1; m &= ~((1ull << (R() % 53)) - 1); break;
        default: e += (int)(R() % 5); m = (1ull << (R() % 53)) - 1;
    }
    return ieee_double((R() & 1) << 63 | (uint64_t)e << 52 | (m & (IEEE_HIDDEN - 1)));
}
int main() {
    for (jitter = 0; jitter < 2; ++jitter)
        for (int i = 0; i < 2000000; ++i) {
            const double a = draw(), b = draw(), z = a * b, s = a * a;
            same(ieee_div(a, b), a / b);
            same(ieee_div(z, b), z / b);
            same(ieee_sqrt(a), sqrt(a));
            same(ieee_sqrt(fabs(b)), sqrt(fabs(b)));
            same(ieee_sqrt(s), sqrt(s));
        }
    for (double x : {0.0, -0.0, 1.0, -1.0, 4.0, (double)INFINITY, -(double)INFINITY, (double)NAN, 5e-324, 1.7976931348623157e308})
        for (double y : {0.0, -0.0, 1.0, -2.0, 3.0, (double)INFINITY, (double)NAN, 5e-324, 1.7976931348623157e308}) {
            same(ieee_div(x, y), x / y);
            same(ieee_sqrt(x), sqrt(x));
        }
    printf("%ld\n", bad);
    return 0;
}
"""


def test_integer_division_and_root_are_correctly_rounded(tmp_path):
    src, exe = tmp_path / "ieee.cpp", tmp_path / "ieee"
    src.write_text(DRIVER)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_1812_08942_gb300", "csrc"), "-o",
                    str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.strip() == "0"
