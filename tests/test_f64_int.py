"""The integer-pipe FP64 products of the FP64 stage (csrc/f64_int.cuh), compiled for the host, against the
hardware's products: bit for bit over random significands, rounding ties, powers of two and zeros."""
import os
import subprocess

from conftest import ROOT

HARNESS = r"""
#include "f64_int.cuh"
#include <cmath>
#include <cstdio>
#include <random>
using namespace vk;
static double of(uint64_t u) { double x; memcpy(&x, &u, 8); return x; }
int main()
{
    std::mt19937_64 g(11);
    auto value = [&]() {
        const uint64_t r = g();
        uint64_t m = r & 0xfffffffffffffull;
        switch ((r >> 53) % 8) {
        case 0: m = 0; break;                                     // a power of two
        case 1: m = 0xfffffffffffffull - (r & 7); break;          // just below one
        case 2: m &= 0xffffffc000000ull; break;                   // 26 bits: exact products and ties
        case 3: m = r & 7; break;
        }
        return of((r & 0x8000000000000000ull) | ((uint64_t)(1023 - 450 + g() % 900) << 52) | m);
    };
    long bad = 0;
    for (long t = 0; t < 3000000; ++t) {
        double a = value(), b = value();
        if (t % 100 == 0) a = t % 200 ? 0.0 : -0.0;
        if (t % 100 == 1) b = 0.0;
        const double p = a * b;
        bad += mul_int_zz(a, b) != p || (p != 0.0 && f64_bits(mul_int_zz(a, b)) != f64_bits(p));
        if (b != 0.0) bad += mul_int_z(a, b) != p;
        bad += sq_int(a) != a * a;
        {   // sums of values that are not negative: near, far and equal exponents
            const double u = std::fabs(a), v = t % 3 ? std::fabs(b) : std::ldexp(std::fabs(b) == 0.0 ? 0.0 : 1.0 + std::fabs(std::fmod(b, 1.0)), std::ilogb(u == 0.0 ? 1.0 : u) - (int)(g() % 70));
            bad += add_pos(u, v) != u + v || add_pos(v, u) != u + v;
        }
        bad += mul_small<3>(a) != 3.0 * a || mul_small<5>(a) != 5.0 * a || mul_small<7>(a) != 7.0 * a ||
               mul_small<11>(a) != 11.0 * a;
        bad += scale2<1>(a) != 2.0 * a || scale2<2>(a) != 4.0 * a || scale2<-1>(a) != 0.5 * a ||
               scale2<-2>(a) != 0.25 * a;
        const bool in = a == 0.0 || (std::fabs(a) >= 0x1p-400 && std::fabs(a) < 0x1p100);
        bad += f64_within<400, 100>(a) != in;
    }
    for (double x : {(double)INFINITY, -(double)INFINITY, (double)NAN, 5e-324, 1e300})
        bad += f64_within<400, 100>(x);
    std::printf("%ld\n", bad);
}
"""


def test_integer_products_equal_the_hardware_products(tmp_path):
    src = tmp_path / "f64_int.cpp"
    src.write_text(HARNESS)
    exe = tmp_path / "f64_int"
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_2504_15574_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    assert int(subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout) == 0


CONSTANT_DIVISION = r"""
#include "f64_int.cuh"
#include <cmath>
#include <cstdio>
#include <random>
using namespace vk;
int main()
{
    std::mt19937_64 g(5);
    std::uniform_real_distribution<double> u(1.0, 2.0);
    long bad = 0;
    for (int k = 0; k < 200; ++k) {
        const double fixed[] = {1.0, 0.5, 0.25, 0x1p-6, 0x1p-10, 2.0, 0x1p-99, 0x1p99, 3.0, 6.0, 0.02, 5e-3, 1e-30, 1e30};
        const double d = k < 14 ? fixed[k] : std::ldexp(u(g), (int)(g() % 190) - 95);
        const DivC c = div_const_of(d);
        for (int t = 0; t < 20000; ++t) {
            double x = std::ldexp(u(g), (int)(g() % 500) - 400) * (g() & 1 ? 1.0 : -1.0);
            if (t % 50 == 0) x = 0.0;
            if (t % 50 == 1) x = std::ldexp(1.0, (int)(g() % 500) - 400);
            bad += div_const_int(x, c) != x / d;
        }
    }
    std::printf("%ld\n", bad);
}
"""


def _run(tmp_path, source):
    src = tmp_path / "harness.cpp"
    src.write_text(source)
    exe = tmp_path / "harness"
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_2504_15574_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout


def test_constant_divisions_equal_the_hardware_quotients(tmp_path):
    """x / d as a product and a fused operation, for divisors with an exact reciprocal (tau = 1, 1/2, 1/64, ...)
    and without one, over zero, powers of two and both signs."""
    assert int(_run(tmp_path, CONSTANT_DIVISION)) == 0


DIVISION = r"""
#include "f64_int.cuh"
#include <cmath>
#include <cstdio>
#include <random>
using namespace vk;
static std::mt19937_64 g(7);
static uint64_t inverse(uint64_t d) { uint64_t x = d; for (int k = 0; k < 6; ++k) x *= 2 - d * x; return x; }
// an X in [2^52, 2^53) whose quotient X / D (D odd) lies r / D of the last place from a rounding boundary; 0: none
static uint64_t near_boundary(uint64_t D, int64_t r, int k)
{
    const uint64_t mod = 1ull << k;
    uint64_t N = (0 - (uint64_t)r * inverse(D)) & (mod - 1);
    if (N < (1ull << 53)) N += k == 53 ? mod : 0;
    if (N < (1ull << 53) || !(N & 1)) return 0;
    const __int128 X = ((__int128)N * (int64_t)D + r) >> k;
    if (X < ((__int128)1 << 52) || X >= ((__int128)1 << 53) || (X >= (__int128)D) != (k == 53)) return 0;
    return (uint64_t)X;
}
static long bad = 0, near = 0, missed = 0, random_missed = 0;
static void divide(double a, double b, bool hard)
{
    bool miss = false;
    double q = div_pos(a, b, miss);
    near += hard;
    missed += hard && miss;
    random_missed += !hard && miss;
    if (!miss) bad += q != a / b;
}
int main()
{
    std::uniform_real_distribution<double> u(1.0, 2.0);
    for (int t = 0; t < 3000000; ++t) {
        double b = std::ldexp(u(g), (int)(g() % 900) - 450), a = std::ldexp(u(g), (int)(g() % 900) - 450);
        if (t % 3 == 0) a = t % 2 ? 0.1 : 0.3;
        if (t % 7 == 0) a = b * (double)(1 + g() % 9);   // exact quotients
        if (t % 2) a = -a;
        if (t % 11 == 0) b = std::ldexp(1.0, (int)(g() % 900) - 450);
        divide(a, b, false);
    }
    for (int t = 0; t < 200000; ++t) {
        const uint64_t D = ((1ull << 52) + (g() & ((1ull << 52) - 1))) | 1;
        const uint64_t X = near_boundary(D, (int64_t)(g() % 65) - 32, t & 1 ? 53 : 54);
        if (X) divide(std::ldexp((double)X, (int)(g() % 100)), std::ldexp((double)D, (int)(g() % 100)), true);
    }
    // constants: the x of their hardest quotients
    long inexact = 0, general = 0;
    for (int t = 0; t < 40000; ++t) {
        uint64_t D = (1ull << 52) + (g() & ((1ull << 52) - 1));
        if (t & 1) D &= ~7ull;   // even ones too
        const double d = std::ldexp((double)D, -60);
        const DivC c = div_const_of(d);
        ++general;
        const bool exact = div_const_exact(c);
        inexact += !exact;
        int z = 0;
        for (; !(D & 1); D >>= 1) ++z;
        if (z) continue;
        for (int64_t r = -40; r <= 40; ++r)
            for (int k : {53, 54})
                if (uint64_t X = near_boundary(D, r, k)) {
                    const double x = std::ldexp((double)X, -90);
                    bad += exact && div_const(x, c) != x / d;
                    bad += exact && div_const_int(-x, c) != -x / d;
                }
    }
    for (double d : {3.0, 6.0, 0.02, 5e-3, 2e-3, 1e-3}) bad += !div_const_exact(div_const_of(d));
    std::printf("%ld %ld %ld %ld %ld %ld\n", bad, near, missed, random_missed, inexact, general);
}
"""


def test_divisions_are_the_rounded_quotients(tmp_path):
    """The divisions of the FP64 stage: every quotient is the hardware's, or (div_pos) reported as missed so that
    the caller divides.  Random operands, exact quotients, and operands built to lie next to a rounding
    boundary, where a value good to 2^-88 rounds to the wrong side."""
    bad, near, missed, random_missed, inexact, general = map(int, _run(tmp_path, DIVISION).split())
    assert bad == 0
    assert near > 20000 and missed > near / 4   # about half of the built ones round to the wrong side
    assert random_missed < 3e6 / 2**16          # false alarms of the high words' comparison: 2^-19
    assert inexact < 0.03 * general             # 1.8 % of general divisors miss one or two significands
