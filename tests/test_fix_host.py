"""The two-digit fixed-point arithmetic (paper_2411_18511_gb300/csrc/hr_fix.cuh)
compiled as plain C++ on the host: digits of doubles and of float pairs, sums of
products, shifted blocks and quaternion products against long double, with an
error no larger than binary64 arithmetic makes on the same inputs."""

import os
import platform
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_18511_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <random>
#include "hr_fix.cuh"
using namespace hr;
using L = long double;
static L val(fx v) { return v.h * 0x1p-28L + v.l * 0x1p-56L; }
int main() {
    std::mt19937_64 g(11);
    std::normal_distribution<double> nd;
    std::uniform_real_distribution<double> un(-1, 1);
    // digits of doubles: truncated at 2^-56, every magnitude below 4
    L conv = 0;
    for (int k = 0; k < 200000; ++k) {
        const double x = std::ldexp(un(g), (int)(g() % 70) - 67);
        const L d = fabsl(val(fx_from_double(x)) - (L)x);
        if (d > conv) conv = d;
    }
    for (double x : {0.0, -0.0, 1.0, -1.0, 3.999, 5e-324, -1e-300, 0x1p-56, -0x1p-57})
        conv = fmaxl(conv, fabsl(val(fx_from_double(x)) - (L)x));
    // digits of normalised float pairs over the whole exponent range
    L pair = 0;
    long bad = 0;
    for (int k = 0; k < 400000; ++k) {
        const int E = 21 + (int)(g() % 234);
        const float hi = std::ldexp((float)un(g), E - 126 - (k % 3 ? 0 : (int)(g() % 60)));
        const float lo = std::ldexp((float)un(g), std::ilogb(hi == 0 ? 1e-30f : hi) - 24);
        if (hi == 0 || std::fabs(hi) >= std::ldexp(1.0L, E - 126) || (float)(hi + lo) != hi) continue;
        const fx v = fx_from_pair(hi, lo, fx_pair_scale(E));
        const L d = fabsl(val(v) * powl(2.0L, E - kFxPairBias) - ((L)hi + lo)) / powl(2.0L, E - kFxPairBias);
        if (d > pair) pair = d;
        if (v.l > (1 << 27) + (1 << 17) || v.l < -(1 << 27) - (1 << 17)) ++bad;
    }
    // quaternion products of unit quaternions, three in a chain
    L eq = 0, ed = 0, nq = 0;
    for (int k = 0; k < 20000; ++k) {
        double a[3][4];
        for (auto &q : a) {
            double n = 0;
            for (double &c : q) { c = nd(g); n += c * c; }
            for (double &c : q) c /= std::sqrt(n);
        }
        auto mul = [](auto *r, const auto *x, const auto *y) {
            r[0] = x[0] * y[0] - x[1] * y[1] - x[2] * y[2] - x[3] * y[3];
            r[1] = x[0] * y[1] + x[1] * y[0] - x[2] * y[3] + x[3] * y[2];
            r[2] = x[0] * y[2] + x[2] * y[0] - x[3] * y[1] + x[1] * y[3];
            r[3] = x[0] * y[3] + x[3] * y[0] - x[1] * y[2] + x[2] * y[1];
        };
        L l[3][4], lt[4], lr[4];
        double dt[4], dr[4];
        fxq f[3];
        for (int q = 0; q < 3; ++q)
            for (int c = 0; c < 4; ++c) { l[q][c] = a[q][c]; f[q].c[c] = fx_from_double(a[q][c]); }
        mul(lt, l[0], l[1]); mul(lr, lt, l[2]);
        mul(dt, a[0], a[1]); mul(dr, dt, a[2]);
        const fxq fr = fxq_mul(fxq_mul(f[0], f[1]), f[2]);
        for (int c = 0; c < 4; ++c) {
            eq += (val(fr.c[c]) - lr[c]) * (val(fr.c[c]) - lr[c]);
            ed += (dr[c] - lr[c]) * (dr[c] - lr[c]);
            nq += lr[c] * lr[c];
        }
    }
    // blocks of sums at every magnitude, brought to a common shift
    L shifted = 0;
    for (int k = 0; k < 200000; ++k) {
        const int down = (int)(g() % 61), downb = (int)(g() % 61);
        fxa s[2];
        unsigned long long used = 0;
        for (auto &v : s) {
            v.a = (long long)(un(g) * 0x1p60) >> down;
            v.b = (long long)(un(g) * 0x1p61) >> downb;
            used |= fx_used(v);
        }
        const int sh = fx_block_shift(used);
        for (auto &v : s) {
            const long long t = fx_shifted(v, sh);
            const L want = (v.a + v.b * 0x1p-28L) * powl(2.0L, sh);
            if (fabsl((L)t) >= 0x1p58L) ++bad;
            shifted = fmaxl(shifted, fabsl((L)t - want));
        }
    }
    std::printf("%Lg %Lg %Lg %Lg %Lg %ld\n", conv, pair, sqrtl(eq / nq), sqrtl(ed / nq), shifted, bad);
}
"""


def test_fixed_point_matches_long_double(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    if platform.machine() not in ("x86_64", "aarch64"):
        pytest.skip("needs a long double wider than binary64")
    src, exe = tmp_path / "fix.cpp", tmp_path / "fix"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    conv, pair, eq, ed, shifted, bad = map(float, subprocess.run([str(exe)], check=True, capture_output=True,
                                                                 text=True).stdout.split())
    assert conv < 2.0 ** -56           # truncation
    assert pair <= 2.0 ** -56          # one rounding at 2^-57 and the residuals' FP32 sum
    assert eq < ed                     # a chain of products: no further off than binary64
    assert shifted <= 1.0 + 2.0 ** -10 # truncated units (the 80-bit reference rounds too)
    assert bad == 0
