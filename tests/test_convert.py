"""The integer FP64 <-> FP32 and float-float conversions of the layout kernels (convert.h, host
path) against the casts, bit for bit: random bit patterns over all exponents, values of ordinary
size, rounding ties and their neighbours, the ends of the normal, subnormal and float-float ranges,
zeros, infinities and NaN (as NaN)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <stdio.h>
#include <cmath>
#include <initializer_list>
#include "convert.h"
using namespace ovl;
static uint64_t rng = 88172645463325252ull;
static uint64_t next() { rng ^= rng << 13; rng ^= rng >> 7; rng ^= rng << 17; return rng; }
static double of(uint64_t u) { double x; memcpy(&x, &u, 8); return x; }
static uint64_t bits(double x) { uint64_t u; memcpy(&u, &x, 8); return u; }
static long bad = 0;
static void same_f(float a, float b, double x, const char *w) {
    if (conv_f_bits(a) != conv_f_bits(b) && !(std::isnan(a) && std::isnan(b)) && bad++ < 20) printf("%s %a: %a %a\n", w, x, a, b);
}
static void same_d(double a, double b, double x, const char *w) {
    if (bits(a) != bits(b) && !(std::isnan(a) && std::isnan(b)) && bad++ < 20) printf("%s %a: %a %a\n", w, x, a, b);
}
static void check(double x) {
    volatile double y = x;
    same_f(d2f(x), (float)y, x, "d2f");
    const float f = (float)y;
    same_d(f2d(f), (double)f, x, "f2d");
    float h, l;
    d2ff(x, h, l);
    same_f(h, f, x, "d2ff h");
    const double r = y - (double)f;
    same_f(l, (float)r, x, "d2ff l");
    same_d(ff2d(h, l), (double)h + (double)l, x, "ff2d");
    // low words that d2ff does not make: any size up to an ulp of h, of either sign
    const float any = h * (float)((double)(next() >> 12) / (double)(1ull << 52) * 0x1p-23) * (next() & 1 ? 1.f : -1.f);
    const float small = any * (float)std::ldexp(1.0, -(int)(next() % 40));
    same_d(ff2d(h, any), (double)h + (double)any, x, "ff2d any");
    same_d(ff2d(h, small), (double)h + (double)small, x, "ff2d small");
    if (finite_bits(x) != std::isfinite(x)) bad++;
}
int main() {
    for (int k = 0; k < 3000000; k++) {
        const uint64_t u = next();
        check(of(u));                                                   // any bits
        const uint64_t e = 1023 - 80 + next() % 120;                    // ordinary sizes
        const uint64_t m = (u & 0x800fffffffffffffull) | e << 52;
        check(of(m));
        check(of((m & ~0x1fffffffull) | (0x10000000ull + (int64_t)(next() % 3) - 1)));   // ties and neighbours
        check(of(m & ~0x1fffffffull));                                  // FP32 values
        check(of(m & 0xfff0000000000000ull));                           // powers of two
    }
    const int ends[] = {0, 1, 2, 896 - 30, 896 - 1, 896, 897, 898, 952, 953, 954, 1149, 1150, 1151, 2046, 2047};
    const uint64_t man[] = {0, 1, 0x0fffffffull, 0x10000000ull, 0x10000001ull, 0x1fffffffull, 0x20000000ull,
                            0x3fffffffull, 0xfffffe0000000ull, 0xfffffefffffffull, 0xffffff0000000ull, 0xfffffffffffffull};
    for (int e : ends) for (uint64_t m : man) for (int s = 0; s < 2; s++) check(of((uint64_t)s << 63 | (uint64_t)e << 52 | m));
    check(0.0);
    check(-0.0);
    for (float a : {0.f, -0.f}) for (float b : {0.f, -0.f}) same_d(ff2d(a, b), (double)a + (double)b, a, "ff2d zeros");
    printf("bad %ld\n", bad);
    return bad != 0;
}
"""


def test_conversions_equal_casts(tmp_path):
    src, exe = tmp_path / "convert_test.cpp", tmp_path / "convert_test"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_1410_7170_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
