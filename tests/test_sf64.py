"""sf64.cuh on the CPU: its FP64 quotients and square roots equal the
hardware's bit for bit over the exponent range (edges of it too), for
mantissas of every shape, whatever the last bits of the FP32 estimates."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2504_06067_gb300", "csrc")

PROGRAM = r"""
#include "sf64.cuh"
#include <cstdio>
#include <random>
namespace sf64 { int sf_ulp = 0; }
using sf64::u64;
static std::mt19937_64 g(1);
static double draw(long k)
{
    u64 m = g() & 0xfffffffffffffull;
    switch (k % 6) {
    case 1: m &= ~0ull << (g() % 52); break;             // trailing zeros
    case 2: m |= ~(~0ull << (g() % 52)); break;          // trailing ones
    case 3: m = (m >> 29) << 29; break;                  // an FP32 value
    case 4: m = (g() & 1) ? (g() & 7) : 0xfffffffffffffull - (g() & 7); break;  // next to a power of two
    }
    const u64 e = k % 7 == 0 ? g() % 2048 : (k & 1) ? 983 + g() % 80 : 1 + g() % 2046;
    return sf64::value((e << 52) | (m & 0xfffffffffffffull) | ((g() & 1) << 63));
}
static long bad = 0;
static void same(double x, double y, const char* what, double a, double b)
{
    if (sf64::bits(x) == sf64::bits(y) || (x != x && y != y)) return;
    if (bad++ < 10) printf("%s(%a, %a) = %a, not %a\n", what, a, b, x, y);
}
int main()
{
    for (int u = -3; u <= 3; ++u) {
        sf64::sf_ulp = u;
        for (long i = 0; i < 600000; ++i) {
            const double a = draw(i), b = draw(i / 6);
            same(sf64::div(a, b), a / b, "div", a, b);
            same(sf64::div(a * b, b), (a * b) / b, "div", a * b, b);
            same(sf64::sqrt_rn(a), sqrt(a), "sqrt", a, a);
            const double s = (double)((g() >> 12) + 1);
            same(sf64::sqrt_rn(s * s), sqrt(s * s), "sqrt", s * s, 0);
        }
    }
    printf("%ld\n", bad);
    return bad ? 1 : 0;
}
"""


def test_quotients_and_roots_equal_the_hardware(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
