"""The integer conversions between binary64 and float pairs
(paper_2411_18511_gb300/csrc/hr_cvt.cuh) compiled as plain C++ on the host: where
they report success, the bits are those of the native conversions; they report it
for the numbers that fields hold."""

import os
import platform
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_18511_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "hr_cvt.cuh"
using namespace hr;
static long bad = 0, refused = 0, tried = 0;
static void both(double x, bool must) {
    volatile float h = (float)x;
    volatile float l = (float)(x - (double)h);
    float a, b;
    double y, w;
    ++tried;
    if (cvt_split(x, a, b)) {
        if (fx_bits(a) != fx_bits(h) || fx_bits(b) != fx_bits(l)) ++bad;
    } else if (must) ++refused;
    volatile double s = (double)h + (double)l;
    if (cvt_join(h, l, y) && fx_dbits(y) != fx_dbits(s)) ++bad;
    volatile double v = (double)h;
    if (cvt_widen(h, w) && fx_dbits(w) != fx_dbits(v)) ++bad;
}
static long joined = 0, joins = 0;
static void pair(float h, float l) {
    double y;
    volatile double s = (double)h + (double)l;
    ++joins;
    if (cvt_join(h, l, y)) {
        ++joined;
        if (fx_dbits(y) != fx_dbits(s)) ++bad;
    }
}
int main() {
    std::mt19937_64 g(5);
    std::normal_distribution<double> nd;
    for (int k = 0; k < 2000000; ++k) both(nd(g), true);
    // every exponent, every pattern of low bits: ties, carries, short and long numbers
    for (int k = 0; k < 4000000; ++k) {
        const int e = (int)(g() % 240) - 120;
        double m = 1.0 + (double)(g() >> 12) * 0x1p-52;
        if (k % 4 == 1) m = 1.0 + std::ldexp((double)(g() >> 40), -24) + std::ldexp((double)(g() % 5), -27 + (int)(g() % 3));
        if (k % 4 == 2) m = 2.0 - std::ldexp((double)(g() % 9), -52 + (int)(g() % 30));
        if (k % 4 == 3) m = 1.0 + std::ldexp((double)(g() % 9), -52 + (int)(g() % 30));
        both(std::ldexp(g() & 1 ? m : -m, e), e >= -63 && e < 119 && m < 2.0);
    }
    for (double x : {0.0, -0.0, 1.0, -1.0, 0x1p-63, 0x1p-64, 0x1p120, 0x1.8p119, 1e300, -1e-300, 5e-324, (double)INFINITY,
                     -(double)INFINITY, 0x1p-126, 0x1p-149})
        both(x, false);
    {
        float a, b;
        if (cvt_split(NAN, a, b) || cvt_split(INFINITY, a, b) || cvt_split(1e39, a, b)) ++bad;
        double y;
        if (cvt_join(NAN, 0.f, y) || cvt_join(INFINITY, 1.f, y) || cvt_join(1.f, NAN, y) || cvt_join(1.f, INFINITY, y)) ++bad;
        if (cvt_widen(NAN, y) || cvt_widen(INFINITY, y) || cvt_widen(1e-42f, y)) ++bad;
    }
    // pairs as arithmetic leaves them: l anywhere below half a unit of h, of any length
    std::uniform_real_distribution<double> un(-1, 1);
    for (int k = 0; k < 4000000; ++k) {
        const float h = std::ldexp((float)nd(g), (int)(g() % 60) - 30);
        if (h == 0.f) continue;
        float l = std::ldexp((float)un(g), std::ilogb(h) - 24 - (k % 8 == 0 ? (int)(g() % 40) : 0));
        if (k % 16 == 1) l = std::ldexp(g() & 1 ? 1.f : -1.f, std::ilogb(h) - 24);
        if (k % 16 == 2) l = 0.f;
        pair(h, l);
    }
    for (float h : {0.f, -0.f, 1.f, -1.f, 2.f, 1e-40f, 0x1p-126f})
        for (float l : {0.f, -0.f, 0x1p-25f, -0x1p-25f, 0x1p-24f, -0x1p-30f, 1e-42f, 1.f, -1.f}) pair(h, l);
    std::printf("%ld %ld %ld %.4f\n", bad, refused, tried, (double)joined / joins);
    return 0;
}
"""


def test_conversions_have_the_native_bits(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src = tmp_path / "cvt.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "cvt"
    flags = ["-O2", "-std=c++17", "-ffp-contract=off"]
    if platform.machine() == "x86_64":
        flags.append("-mfma")
    subprocess.run([gxx, *flags, "-I", CSRC, str(src), "-o", str(exe)], check=True)
    bad, refused, tried, joined = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert int(bad) == 0
    assert int(refused) == 0 and int(tried) > 5_000_000
    assert float(joined) > 0.9
