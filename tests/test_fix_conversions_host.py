"""The fixed-point conversions that the link kernels use (hr_fix.cuh: fx_from_unit,
fx_from_double in units of a block, fx_to_pair, fx_to_double), compiled as plain
C++ on the host, and quaternion chains from cut digits against binary64."""

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
    std::mt19937_64 g(12);
    std::normal_distribution<double> nd;
    std::uniform_real_distribution<double> un(-1, 1);
    long bad = 0;
    L unit = 0, block = 0, pair = 0, dbl = 0;
    auto cut = [&](double x) {
        const fx v = fx_from_unit(x);
        unit = fmaxl(unit, fabsl(val(v) - (L)x));
        if (v.l <= -(1 << 28) || v.l >= 1 << 28 || (v.l && (v.l < 0) != (x < 0)) || fabsl(val(v)) > fabsl((L)x)) ++bad;
    };
    for (int k = 0; k < 200000; ++k) cut(std::ldexp(un(g), (int)(g() % 70) - 68));
    for (double x : {0.0, -0.0, 1.0, -1.0, 1.999, 5e-324, -1e-300, 0x1p-56, -0x1p-57, -0x1p-28}) cut(x);
    for (int k = 0; k < 200000; ++k) {
        const int E = 60 + (int)(g() % 1900);
        const double x = std::ldexp(un(g), E - 1022 - (k & 1 ? 0 : (int)(g() % 64)));
        const L got = val(fx_from_double(x, E));
        block = fmaxl(block, fabsl(got - ldexpl((L)x, 1022 - E)));
    }
    for (int k = 0; k < 400000; ++k) {
        const long long t = (long long)(g() >> 5) >> (g() % 59) << (g() % 3 ? 0 : 2), u = g() & 1 ? -t : t;
        if (u == 0 || u >= 1LL << 59 || u <= -(1LL << 59)) continue;
        float hi, lo;
        fx_to_pair(u, hi, lo);
        const L want = u * 0x1p-56L;
        pair = fmaxl(pair, fabsl(((L)hi + lo - want) / want));
        if ((float)(hi + lo) != hi) ++bad;
        const int s = (int)(g() % 901);
        dbl = fmaxl(dbl, fabsl((fx_to_double(u, s) - ldexpl(want, -s)) / ldexpl(want, -s)));
    }
    if (fx_to_double(0, 900) != 0.0) ++bad;
    // |q|^2 and chains of three products from cut digits
    L eq = 0, ed = 0, worst = 0, mean = 0;
    const int n = 20000;
    for (int k = 0; k < n; ++k) {
        double a[3][4];
        for (auto &q : a) {
            double s = 0;
            for (double &c : q) { c = nd(g); s += c * c; }
            for (double &c : q) c /= std::sqrt(s);
        }
        auto mul = [](auto *r, const auto *x, const auto *y) {
            r[0] = x[0] * y[0] - x[1] * y[1] - x[2] * y[2] - x[3] * y[3];
            r[1] = x[0] * y[1] + x[1] * y[0] - x[2] * y[3] + x[3] * y[2];
            r[2] = x[0] * y[2] + x[2] * y[0] - x[3] * y[1] + x[1] * y[3];
            r[3] = x[0] * y[3] + x[3] * y[0] - x[1] * y[2] + x[2] * y[1];
        };
        L l[3][4], lt[4], lr[4], norm = 0;
        double dt[4], dr[4];
        fxq f[3];
        fxa s = {0, 0};
        for (int q = 0; q < 3; ++q)
            for (int c = 0; c < 4; ++c) { l[q][c] = a[q][c]; f[q].c[c] = fx_from_unit(a[q][c]); }
        for (int c = 0; c < 4; ++c) { fx_mac(s, f[0].c[c], f[0].c[c]); norm += l[0][c] * l[0][c]; }
        const L off = fx_round(s) * 0x1p-56L - norm;
        worst = fmaxl(worst, fabsl(off));
        mean += off / n;
        mul(lt, l[0], l[1]); mul(lr, lt, l[2]);
        mul(dt, a[0], a[1]); mul(dr, dt, a[2]);
        const fxq fr = fxq_mul(fxq_mul(f[0], f[1]), f[2]);
        for (int c = 0; c < 4; ++c) {
            eq += (val(fr.c[c]) - lr[c]) * (val(fr.c[c]) - lr[c]);
            ed += (dr[c] - lr[c]) * (dr[c] - lr[c]);
        }
    }
    std::printf("%Lg %Lg %Lg %Lg %Lg %Lg %Lg %Lg %ld\n", unit, block, pair, dbl, sqrtl(eq), sqrtl(ed), worst, fabsl(mean), bad);
}
"""


def test_conversions_match_long_double(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    if platform.machine() not in ("x86_64", "aarch64"):
        pytest.skip("needs a long double wider than binary64")
    src, exe = tmp_path / "fix.cpp", tmp_path / "fix"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    unit, block, pair, dbl, eq, ed, worst, mean, bad = map(
        float, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    ulp = 2.0 ** -56
    assert unit < ulp and block < ulp      # truncation
    assert pair <= 2.0 ** -49 * 1.001      # of the value, as two floats split from a double
    assert dbl <= 2.0 ** -53
    assert eq < ed                         # a chain of products: no further off than binary64
    # |q|^2: four dropped products of cut digits and four cut numbers
    assert worst <= 5 * ulp and mean <= 2 * ulp
    assert bad == 0
