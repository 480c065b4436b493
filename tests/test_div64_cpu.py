"""The integer division of a double by a float and the widening of a float
(csrc/div64.cuh), compiled for the host, against the processor's own: every
result has the same bits, for reciprocals anywhere within the stated bound."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2109_05410_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cmath>
#include <initializer_list>
#include <limits>
#include "div64.cuh"
using namespace ooc;
static uint64_t s = 88172645463325252ull;
static uint64_t rnd() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; }
static long bad = 0;
template <typename U, typename T> void same(T a, T b)
{
    if (!(a != a && b != b) && bits_as<U>(a) != bits_as<U>(b) && bad++ < 5)
        printf("%a %a\n", (double)a, (double)b);
}
static void one(double g, float k)
{
    const double r0 = 1.0 / (double)significand(k);
    for (double d : {-2.38418579e-7, 0.0, 2.38418579e-7})  // 2^-22
        same<uint64_t>(div_f64_f32(g, k, (float)(r0 * (1.0 + d))), g / (double)k);
}
int main()
{
    const double gs[] = {0.0, -0.0, 1.0, -3.0, 5e-324, 2.2250738585072014e-308, 1.7976931348623157e308, INFINITY, NAN,
                         std::nextafter(2.0, 0.0), std::nextafter(1.0, 2.0), 1e-300, -1e300};
    const float ks[] = {0.0f, -0.0f, 1.0f, -3.0f, 1e-45f, 1.17549435e-38f, 3.40282347e38f, INFINITY, NAN,
                        std::nextafter(2.0f, 0.0f), std::nextafter(1.0f, 2.0f)};
    for (double g : gs)
        for (float k : ks)
            one(g, k);
    for (float k : ks)
        same<uint64_t>(widen(k), (double)k);
    for (int i = 0; i < 3000000; ++i) {
        const uint64_t a = rnd(), b = rnd();
        const float any = bits_as<float>((uint32_t)b), k = bits_as<float>((uint32_t)(b & 0x807fffff) | 0x3d800000u);
        one(bits_as<double>(a), any);                                            // all patterns
        one(bits_as<double>((a & 0x800fffffffffffffull) | 0x3f50000000000000ull), k);  // usual exponents
        // quotients next to a float of 24 bits and to a midpoint of two doubles
        const double q = (double)bits_as<float>((uint32_t)(a & 0x007fffff) | 0x3f800000u) + (a >> 62) * 0x1p-52;
        one(q * (double)k, k);
        one((double)bits_as<float>((uint32_t)(a & 0x007fffff) | 0x3f800000u) * 0x1p-30, k);
        same<uint64_t>(widen(any), (double)any);
    }
    return bad != 0;
}
"""


def test_division_and_widening_have_the_processors_bits(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(MAIN)
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
