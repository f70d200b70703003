"""The integer square root and quotient of the Cholesky pivots
(csrc/exact_math.h), compiled for the host: equal to IEEE's correctly rounded
operations bit for bit, with the FP32 approximations at either end of their
error and at operands that round near a tie or a power of two."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2007_15195_gb300", "csrc")

MAIN = r"""
#include "exact_math.h"
#include <cstdio>
#include <random>
using namespace vk::exact;
static std::mt19937_64 r(1);
static double any(int mode) {
    uint64_t m = r() & kMant;
    if (mode % 4 == 1) m &= ~((1ull << 26) - 1);
    if (mode % 4 == 2) m |= (1ull << 40) - 1;
    if (mode % 4 == 3) m = r() % 8;
    const int e = 1023 + (int)(r() % ((mode % 5) ? 60 : 1000)) - ((mode % 5) ? 30 : 500);
    return to_f64(((uint64_t)e << 52) | m);
}
static bool same(double a, double b) { return to_u64(a) == to_u64(b) || (a != a && b != b); }
int main() {
    long bad = 0;
    auto check = [&](double s, double x) {
        const Pivot p = pivot(s);
        bad += !same(p.piv, sqrt(s));
        bad += !same(quotient(x, p), x / p.piv);
        bad += !same(quotient(x, pivot_of(p.piv)), x / p.piv);
    };
    for (long i = 0; i < 1500000; ++i) check(any(i & 63), (r() & 1) ? -any((i >> 3) & 63) : any((i >> 3) & 63));
    for (long i = 0; i < 200000; ++i) {  // squares and products, and their neighbours
        const double t = any(i & 63), x = t * any(i & 31);
        for (int k = -1; k <= 1; ++k) check(to_f64(to_u64(t * t) + k), to_f64(to_u64(x) + k));
    }
    const double sp[] = {0.0, -0.0, 5e-324, 1e-310, 1e-300, 1e300, 1.0, 4.0, 0.25, INFINITY, NAN,
                         to_f64((1023ull << 52) | kMant), to_f64((1022ull << 52) | kMant)};
    for (double s : sp)
        for (double x : sp)
            if (s > 0.0) check(s, x);
    printf("%ld", bad);
}
"""


@pytest.mark.parametrize("scale", ["1.0f", "(1.0f + 0x1p-21f)", "(1.0f - 0x1p-21f)"])
def test_equal_to_ieee(tmp_path, scale):
    src, exe = tmp_path / "m.cpp", tmp_path / "m"
    src.write_text("#define VK_APPROX_TEST(y) ((y) * %s)\n" % scale + MAIN)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout == "0"
