"""The integer FP64 division and square root of the device code (f64_soft.cuh),
compiled for the host: every result must have the bits of the host's IEEE
operation, with the FP32 estimates they start from moved by up to 4 units
(the GPU's approximate reciprocal and reciprocal square root are within 2)."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2305_07030_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include "f64_soft.cuh"
using namespace fe2;
static bool same(double x, double y) { return f64_bits(x) == f64_bits(y) || (x != x && y != y); }
static double make(uint64_t s, uint64_t e, uint64_t m) { return f64_from((s << 63) | (e << 52) | (m & kF64Man)); }
int main(int, char **argv) {
    f64_perturb = atoi(argv[1]);
    std::mt19937_64 g(7);
    long bad = 0;
    auto div = [&](double a, double b) { bad += !same(f64_div(a, b), a / b); };
    auto root = [&](double a) { bad += !same(f64_sqrt(a), sqrt(a)); };
    // significands at the edges of their range, exponents over and at theirs
    const uint64_t edge[] = {0, 1, 2, 3, kF64Man, kF64Man - 1, kF64Man - 2, kF64Man >> 1, (kF64Man >> 1) + 1,
                             1ull << 51, 1ull << 22, 1ull << 29, (1ull << 30) - 1};
    for (uint64_t m : edge)
        for (uint64_t n : edge)
            for (uint64_t e : {0ull, 1ull, 2ull, 1022ull, 1023ull, 1024ull, 2045ull, 2046ull, 2047ull})
                for (uint64_t f : {0ull, 1ull, 2ull, 1022ull, 1023ull, 2046ull, 2047ull}) {
                    div(make(m & 1, e, m), make(n & 1, f, n));
                    root(make(0, e, m));
                    root(make(1, f, n));
                    uint32_t v;
                    const double l = f64_sqrt_recip(make(0, f, n), v);
                    bad += !same(f64_div_v<true>(make(m & 1, e, m), l, v), make(m & 1, e, m) / l);
                }
    for (long i = 0; i < 400000; ++i) {
        const uint64_t x = g(), y = g();
        const double a = make(x & 1, 900 + x % 251, x >> 11), b = make(y & 1, 900 + y % 247, y >> 11);
        div(a, b);
        root(fabs(a));
        // quotients and roots next to a representable value or to a midpoint
        div(f64_from(f64_bits(a * b) + x % 5 - 2), b);
        const double s = a * a;
        root(f64_from(f64_bits(s) + y % 5 - 2));
        const double h = make(0, 1000, (x >> 11) & ~0x3ffffffull);  // 26-bit root: its square is exact
        root(h * h);
        // a root as divisor, with the root's own estimate
        uint32_t v;
        const double l = f64_sqrt_recip(f64_from(f64_bits(s) + y % 5 - 2), v);
        bad += !same(f64_div_v<true>(a, l, v), a / l);
        bad += !same(f64_div_v<true>(f64_from(f64_bits(a * l) + x % 5 - 2), l, v), f64_from(f64_bits(a * l) + x % 5 - 2) / l);
        div(a, make(0, 1000, (y >> 11) & (~0ull << (y % 53))));
        div(make(0, 1010, (y >> 11) + x % 7 - 3), make(0, 1003, y >> 11));
    }
    printf("%ld\n", bad);
    return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("f64_soft")
    src = d / "harness.cpp"
    src.write_text(HARNESS)
    exe = d / "harness"
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-x", "c++", str(src), "-o", str(exe)],
                   check=True)
    return str(exe)


@pytest.mark.parametrize("perturb", [-4, -1, 0, 1, 4])
def test_same_bits_as_ieee(harness, perturb):
    out = subprocess.run([harness, str(perturb)], check=True, capture_output=True, text=True).stdout
    assert int(out) == 0
