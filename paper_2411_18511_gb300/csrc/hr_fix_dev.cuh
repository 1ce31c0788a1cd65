// hr_fix_dev.cuh -- lexicographic site steps and canonical links as digits, shared
// by the fixed-point kernels (gauge force, clover build, clover force).
#pragma once

#include "hr_fix.cuh"
#include "hr_internal.cuh"

namespace hr {

// a site by its lexicographic index, with 32-bit steps to its neighbours
struct LexSite {
    int t, x0, x1, x2, x3;
};
__device__ __forceinline__ LexSite lex_site(const Geom &g, int t)
{
    LexSite s;
    const int row = fdiv(t >> 1, g.div_h3), r1 = fdiv(row, g.div_d2);
    s.t = t;
    s.x3 = t - row * g.d[3];
    s.x2 = row - r1 * g.d[2];
    s.x0 = fdiv(r1, g.div_d1);
    s.x1 = r1 - s.x0 * g.d[1];
    return s;
}
// index steps from the site to x + mu and x - mu (periodic)
__device__ __forceinline__ void lex_steps(const Geom &g, const LexSite &s, int mu, int &up, int &down)
{
    const int x = mu == 0 ? s.x0 : mu == 1 ? s.x1 : mu == 2 ? s.x2 : s.x3;
    const int d = mu == 0 ? g.d[0] : mu == 1 ? g.d[1] : mu == 2 ? g.d[2] : g.d[3];
    const int st = mu == 3 ? 1 : mu == 2 ? g.d[3] : mu == 1 ? g.d[3] * g.d[2] : g.d[3] * g.d[2] * g.d[1];
    up = x == d - 1 ? -(d - 1) * st : st;
    down = x == 0 ? (d - 1) * st : -st;
}
// a canonical link as digits (low ones up to 2^28); ok stays true only for links of unit length to 1 %
// (VEC: the field is 16-byte aligned)
template <bool VEC> __device__ __forceinline__ void load_link4(const double *q, size_t link, double (&c)[4])
{
    if constexpr (VEC) {
        const double2 *p = (const double2 *)q + 2 * link;
        const double2 a = p[0], b = p[1];
        c[0] = a.x; c[1] = a.y; c[2] = b.x; c[3] = b.y;
    } else {
        const double *p = q + 4 * link;
#pragma unroll
        for (int k = 0; k < 4; ++k) c[k] = p[k];
    }
}
// (top: raised to the high word of the largest vector component)
template <bool VEC> __device__ __forceinline__ fxq load_fxq(const double *q, size_t link, bool &ok, unsigned &top)
{
    double c[4];
    load_link4<VEC>(q, link, c);
    const unsigned v = max(max(fx_abs_high(c[1]), fx_abs_high(c[2])), fx_abs_high(c[3])), m = max(v, fx_abs_high(c[0]));
    const fxq r = {{fx_from_unit(c[0]), fx_from_unit(c[1]), fx_from_unit(c[2]), fx_from_unit(c[3])}};
    ok = ok && m < kFxHigh2 && fxq_near_unit(r);
    top = max(top, v);
    return r;
}
template <bool VEC> __device__ __forceinline__ fxq load_fxq(const double *q, size_t link, bool &ok)
{
    unsigned top = 0;
    return load_fxq<VEC>(q, link, ok, top);
}

// the 16 reals of a packed FP64 spinor as digits, [2 (2 spin + colour) + (0 re, 1 im)],
// in units of 2^(E - kFxPairBias); E = biased exponent of the largest |hi|.  false: out
// of range (a nonzero spinor below 2^-105, Inf or NaN)
__device__ __forceinline__ bool load_fx(const void *base, int j, fx (&v)[16], int &E)
{
    const float4 *p = (const float4 *)base;
    float4 w[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) w[k] = __ldg(p + vec_index(j, k, 8));
    unsigned m = 0;
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const float4 h = w[2 * s];
        m = max(max(m, max(__float_as_uint(h.x) & 0x7fffffffu, __float_as_uint(h.y) & 0x7fffffffu)),
                max(__float_as_uint(h.z) & 0x7fffffffu, __float_as_uint(h.w) & 0x7fffffffu));
    }
    E = (int)(m >> 23);
    const bool ok = m == 0 || (E >= kFxMinExp && E < 255);
    E = ok ? max(E, kFxMinExp) : 127;
    const float sc = fx_pair_scale(E);
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        const float4 h = w[2 * s], l = w[2 * s + 1];
        v[4 * s + 0] = fx_from_pair(h.x, l.x, sc);
        v[4 * s + 1] = fx_from_pair(h.z, l.z, sc);
        v[4 * s + 2] = fx_from_pair(h.y, l.y, sc);
        v[4 * s + 3] = fx_from_pair(h.w, l.w, sc);
    }
    return ok;
}

} // namespace hr
