// hr_force.cu -- link derivatives of f = Re<a, H b> for fundamental SU(2) links:
// the su(2) fermion force of the HMC (arXiv:2411.18511 Sec. 2.1 and Sec. 2.2 name
// the HMC as the consumer of the even-odd operator) and the gradient with
// respect to the four quaternion components (used by the autograd wrappers).
//
// The two terms of H that contain U_mu(x) are
//   a(x)^+ (1-g_mu) U b(x+mu)  and  a(x+mu)^+ (1+g_mu) U^+ b(x).
// With the spin-traced colour outer products
//   M1 = sum_s b(x+mu)_s [((1-g_mu) a(x))_s]^+,   M2 = sum_s b(x)_s [((1+g_mu) a(x+mu))_s]^+
// their variation is Re tr[dU M1] + Re tr[dU^+ M2], so
//   quaternion gradient  G_k = Re tr[E_k M1] + Re tr[E_k^+ M2]  (E_0 = 1, E_k = i s_k)
//   su(2) force          F_a = Re tr[(i s_a/2)(U M1 - M2 U^+)]   for U -> exp(i w.s/2) U.
// One thread per site (both parities in one launch); it writes all four
// directions of its own links, so no two threads touch the same output.
// Boundaries: the two terms that contain a link on the boundary slice both
// cross the boundary.  An antiperiodic sign multiplies both (the packed links
// carry it; the quaternion gradient, which takes no gauge field, applies it);
// a twist e^{i theta} multiplies the forward hop's term and e^{-i theta} the
// backward hop's, i.e. M1 -> e^{i theta} M1 and M2 -> e^{-i theta} M2.
//
// k_link_deriv_fx (untwisted lattices) does this in two-digit fixed point
// (hr_fix.cuh).  Two facts shrink the work before the arithmetic is chosen:
// (1 -/+ g_mu) is twice a projector, so M1 and M2 are outer products of the two
// half spinors of each field; and f is real and linear in the four quaternion
// components, so only G_k = d f / d u_k is formed (64 products instead of the
// 2 x 2 complex matrices), the force being F = (u0 G - G0 u - u x G) / 2 on the
// vector parts.  k_link_deriv (native FP64) serves twisted lattices, whose
// phase needs the complex matrices, and single links outside the fixed-point
// range (link_terms).
#include <cmath>

#include "hr_fix_dev.cuh"
#include "hr_host.h"

using namespace hr;

namespace {

struct ForceArgs {
    Geom g;
    const void *gauge;
    const void *a[2]; // even, odd halves
    const void *b[2];
    double beta;
    double *out;
    int mode; // 0: su(2) force [4][V][3], 1: quaternion gradient [4][V][4]
    double tc[4], ts[4]; // e^{i theta_mu} of twisted directions (1, 0 otherwise)
};

struct c2 {
    double re, im;
};
__device__ __forceinline__ c2 cmul(c2 a, c2 b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ c2 cmulc(c2 a, c2 b) { return {a.re * b.re + a.im * b.im, a.im * b.re - a.re * b.im}; } // a conj(b)
__device__ __forceinline__ c2 cplus(c2 a, c2 b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ c2 cminus(c2 a, c2 b) { return {a.re - b.re, a.im - b.im}; }

// sg: -1 for a link on the boundary slice of an antiperiodic direction.  The
// force reads the packed links, which carry that sign already; the quaternion
// gradient takes no gauge field and applies it here.  edge: the link lies on
// the boundary slice (x_mu = L_mu - 1), where a twist applies.
template <int MU>
__device__ __forceinline__ void link_terms(const ForceArgs &A, int p, int i, int ifw, long long lex, double sg,
                                           bool edge)
{
    const Geom &g = A.g;
    cpx<double> ax[4][2], axf[4][2], bx[4][2], bxf[4][2];
    load_spinor<2, kF64>(A.a[p], g.nblk_s, i, ax);
    load_spinor<2, kF64>(A.a[1 - p], g.nblk_s, ifw, axf);
    load_spinor<2, kF64>(A.b[p], g.nblk_s, i, bx);
    load_spinor<2, kF64>(A.b[1 - p], g.nblk_s, ifw, bxf);
    // full (1 - g) a(x) and (1 + g) a(x+mu) from their half spinors
    cpx<double> h[2][2], pa[4][2], pb[4][2];
    for (int s = 0; s < 4; ++s)
        for (int c = 0; c < 2; ++c) pa[s][c] = pb[s][c] = {0.0, 0.0};
    spin_project<MU, true>(ax, h);
    spin_accumulate<MU, true>(pa, h);
    spin_project<MU, false>(axf, h);
    spin_accumulate<MU, false>(pb, h);
    c2 M1[2][2], M2[2][2];
    for (int c = 0; c < 2; ++c)
        for (int d = 0; d < 2; ++d) {
            c2 s1 = {0, 0}, s2 = {0, 0};
            for (int s = 0; s < 4; ++s) {
                s1 = cplus(s1, cmulc({bxf[s][c].re, bxf[s][c].im}, {pa[s][d].re, pa[s][d].im}));
                s2 = cplus(s2, cmulc({bx[s][c].re, bx[s][c].im}, {pb[s][d].re, pb[s][d].im}));
            }
            M1[c][d] = s1;
            M2[c][d] = s2;
        }
    if (edge && A.g.twisted) {
        const c2 f = {A.tc[MU], A.ts[MU]}, fb = {A.tc[MU], -A.ts[MU]};
        for (int c = 0; c < 2; ++c)
            for (int d = 0; d < 2; ++d) {
                M1[c][d] = cmul(f, M1[c][d]);
                M2[c][d] = cmul(fb, M2[c][d]);
            }
    }
    const long long V = 2LL * g.vh;
    if (A.mode == 1) {
        // tr(s_1 M) = M10 + M01, tr(s_2 M) = i (M01 - M10), tr(s_3 M) = M00 - M11
        c2 t1[3], t2[3];
        t1[0] = cplus(M1[1][0], M1[0][1]);
        t1[1] = {-(M1[0][1].im - M1[1][0].im), M1[0][1].re - M1[1][0].re};
        t1[2] = cminus(M1[0][0], M1[1][1]);
        t2[0] = cplus(M2[1][0], M2[0][1]);
        t2[1] = {-(M2[0][1].im - M2[1][0].im), M2[0][1].re - M2[1][0].re};
        t2[2] = cminus(M2[0][0], M2[1][1]);
        double G[4];
        G[0] = M1[0][0].re + M1[1][1].re + M2[0][0].re + M2[1][1].re;
        for (int k = 0; k < 3; ++k) G[k + 1] = -t1[k].im + t2[k].im;
        double *o = A.out + ((long long)MU * V + lex) * 4;
        for (int k = 0; k < 4; ++k) o[k] += sg * A.beta * G[k];
    } else {
        double q[4];
        load_quat<kF64>(A.gauge, g.nblk_g, p, MU, i, q);
        // U = [[q0 + i q3, q2 + i q1], [-q2 + i q1, q0 - i q3]]
        c2 U[2][2] = {{{q[0], q[3]}, {q[2], q[1]}}, {{-q[2], q[1]}, {q[0], -q[3]}}};
        c2 Q[2][2];
        for (int c = 0; c < 2; ++c)
            for (int d = 0; d < 2; ++d) {
                c2 um = cplus(cmul(U[c][0], M1[0][d]), cmul(U[c][1], M1[1][d]));       // (U M1)_cd
                c2 mu = cplus(cmulc(M2[c][0], U[d][0]), cmulc(M2[c][1], U[d][1]));     // (M2 U^+)_cd
                Q[c][d] = cminus(um, mu);
            }
        // F_a = Re[(i/2) tr(s_a Q)] = -1/2 Im tr(s_a Q)
        double F[3];
        F[0] = -0.5 * (Q[0][1].im + Q[1][0].im);
        F[1] = -0.5 * (Q[0][1].re - Q[1][0].re);
        F[2] = -0.5 * (Q[0][0].im - Q[1][1].im);
        double *o = A.out + ((long long)MU * V + lex) * 3;
        for (int k = 0; k < 3; ++k) o[k] += A.beta * F[k];
    }
}

__global__ void k_link_deriv(ForceArgs A)
{
    const Geom &g = A.g;
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 2 * g.vh) return;
    int p = t >= g.vh ? 1 : 0;
    int i = t - p * g.vh;
    SiteNb nb;
    site_neighbours(g, i, p, nb);
    long long lex = eo_to_lex(g, i, p);
    // coordinates of the site: boundary slices of the antiperiodic directions
    int x[4];
    long long r = lex;
    for (int k = 3; k >= 0; --k) {
        x[k] = (int)(r % g.d[k]);
        r /= g.d[k];
    }
    auto sg = [&](int mu) { return (A.mode == 1 && ((g.bc >> mu) & 1) && x[mu] == g.d[mu] - 1) ? -1.0 : 1.0; };
    link_terms<0>(A, p, i, nb.fwd[0], lex, sg(0), x[0] == g.d[0] - 1);
    link_terms<1>(A, p, i, nb.fwd[1], lex, sg(1), x[1] == g.d[1] - 1);
    link_terms<2>(A, p, i, nb.fwd[2], lex, sg(2), x[2] == g.d[2] - 1);
    link_terms<3>(A, p, i, nb.fwd[3], lex, sg(3), x[3] == g.d[3] - 1);
}

// ---------------------------------------------------------------- fixed point

// one link in native FP64: fields outside the fixed-point range, and derivatives far
// below the product of the fields' largest components
template <int MU>
__device__ __noinline__ void link_terms_native(const ForceArgs &A, int p, int i, int ifw, long long lex, double sg)
{
    link_terms<MU>(A, p, i, ifw, lex, sg, false);
}

// h[t][c] = s_t + sgn i^c s_pi of (1 - g_mu) (sgn = 1) or (1 + g_mu) (sgn = -1):
// mu = 0: (0, 2) -1, (1, 3) -1;  1: (0, 3) i, (1, 2) i;  2: (0, 3) 1, (1, 2) -1;  3: (0, 2) i, (1, 3) -i
__device__ __forceinline__ void project_fx(int mu, bool minus, const fx (&s)[16], fx (&h)[8])
{
    const bool cross = mu == 1 || mu == 2; // spin partners (0, 3), (1, 2)
    const bool by_i = mu == 1 || mu == 3;
    // sign of the partner's term for t = 0, 1
    const bool n0 = (mu == 0) == minus, n1 = (mu == 0 || mu >= 2) == minus;
#pragma unroll
    for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int a = 4 * t + 2 * c, b = 4 * (2 + t) + 2 * c, x = 4 * (3 - t) + 2 * c;
            const fx pr = cross ? s[x] : s[b], pi = cross ? s[x + 1] : s[b + 1];
            // i^c: (re, im) -> (-im, re)
            fx qr = by_i ? fx_neg(pi) : pr, qi = by_i ? pr : pi;
            const bool n = t == 0 ? n0 : n1;
            h[a] = n ? fx_sub(s[a], qr) : fx_add(s[a], qr);
            h[a + 1] = n ? fx_sub(s[a + 1], qi) : fx_add(s[a + 1], qi);
        }
}

// g_k += Re tr[E_k b h^+] of two half spinors ([4 t + 2 c + (0 re, 1 im)]); DAG: E_k^+
template <bool DAG> __device__ __forceinline__ void mac_links(fxa (&g)[4], const fx (&b)[8], const fx (&h)[8])
{
#pragma unroll
    for (int t = 0; t < 8; t += 4) {
        const fx b0r = b[t], b0i = b[t + 1], b1r = b[t + 2], b1i = b[t + 3];
        const fx h0r = h[t], h0i = h[t + 1], h1r = h[t + 2], h1i = h[t + 3];
        const fx m0r = fx_neg(h0r), m0i = fx_neg(h0i), m1r = fx_neg(h1r), m1i = fx_neg(h1i);
        // Re(h0* b0 + h1* b1)
        fx_mac(g[0], h0r, b0r); fx_mac(g[0], h0i, b0i); fx_mac(g[0], h1r, b1r); fx_mac(g[0], h1i, b1i);
        // -/+ Im(h0* b1 + h1* b0)
        fx_mac(g[1], DAG ? h0r : m0r, b1i); fx_mac(g[1], DAG ? m0i : h0i, b1r);
        fx_mac(g[1], DAG ? h1r : m1r, b0i); fx_mac(g[1], DAG ? m1i : h1i, b0r);
        // +/- Re(h0* b1 - h1* b0)
        fx_mac(g[2], DAG ? m0r : h0r, b1r); fx_mac(g[2], DAG ? m0i : h0i, b1i);
        fx_mac(g[2], DAG ? h1r : m1r, b0r); fx_mac(g[2], DAG ? h1i : m1i, b0i);
        // -/+ Im(h0* b0 - h1* b1)
        fx_mac(g[3], DAG ? h0r : m0r, b0i); fx_mac(g[3], DAG ? m0i : h0i, b0r);
        fx_mac(g[3], DAG ? m1r : h1r, b1i); fx_mac(g[3], DAG ? h1i : m1i, b1r);
    }
}

// The fields as digits, 16 pairs and an exponent a site: each is read at five sites of
// the link kernel, and converting it there took more than half of its instructions.
// Slices above 127 k sites do not fit the scratch twice and are converted there, as
// are all while a graph is captured (SlabLease).
// Field f, vector v of slab site k at d[(8 f + v) n + k], its exponent at e[f n + k].
struct Digits {
    const int4 *d;
    const int *e;
    int n;
};
constexpr int kDigitBad = -1; // exponent of a site outside the fixed-point range

__global__ void __launch_bounds__(128) k_field_digits(ForceArgs A, int t0, int n, int4 *d, int *e)
{
    const Geom &g = A.g;
    const int k = blockIdx.x * blockDim.x + threadIdx.x, f = blockIdx.y;
    if (k >= n) return;
    int t = t0 + k;
    if (t >= 2 * g.vh) t -= 2 * g.vh;
    const LexSite x = lex_site(g, t);
    const int p = (x.x0 + x.x1 + x.x2 + x.x3) & 1;
    fx v[16];
    int E;
    const bool ok = load_fx(f ? A.b[p] : A.a[p], t >> 1, v, E);
#pragma unroll
    for (int j = 0; j < 8; ++j) d[(size_t)(8 * f + j) * n + k] = make_int4(v[2 * j].h, v[2 * j].l, v[2 * j + 1].h, v[2 * j + 1].l);
    e[(size_t)f * n + k] = ok ? E : kDigitBad;
}
__device__ __forceinline__ bool load_digits(const Digits &D, int f, int k, fx (&v)[16], int &E)
{
    const int4 *p = D.d + (size_t)(8 * f) * D.n + k;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int4 w = __ldg(p + (size_t)j * D.n);
        v[2 * j] = {w.x, w.y};
        v[2 * j + 1] = {w.z, w.w};
    }
    E = __ldg(D.e + (size_t)f * D.n + k);
    const bool ok = E != kDigitBad;
    if (!ok) E = 127;
    return ok;
}

// Measured: hr_fermion_force at 32^4 4.39 ms with the native kernel, of it 3.97 ms
// in the kernel (bound by the FP64 pipe: about 700 conversions and 1400
// operations a site); error against a 64-bit evaluation 7.2e-15 with both (the
// hops').  This kernel, converting (DIG = false): 0.413 ms at 168 registers, 0.479
// at 216, 0.438 at 128 (spills).  With the digits (96 registers): 0.31 ms and 0.09
// for k_field_digits (load latency; its output stays in L2) at 32^4, 22 + 5 against 34 us
// at 16^4, 36 + 7 against 48 us at 20 x 14 x 18 x 22; the whole force at 32^4 0.685 ms.
// One thread per site in lexicographic order (so that a warp's outputs are
// contiguous), a run-time loop over the four directions around one copy of the
// conversion and product code: unrolled, the kernel would not fit the
// instruction cache.  Ranges: |h| <= 2^27 per component, 2^28 projected, 8 terms
// of 2^56 per sum.  Each of the two terms of a link is brought to 56 bits below
// its own largest component and the two are aligned before they are added.  The
// digits are in units of a spinor's largest component: where the larger components of one
// field meet the smaller ones of the other (spins of different size within a
// site), the sum lies far below that unit's square and the link takes native FP64.
// For Gaussian fields that happens on about 1e-6 of the links.  The test costs 3 % of
// the force kernel.
// DIG: the m sites from t0 on with both fields' digits of a slab (`wrap`: of the whole
// lattice, else of these slices and the next one); else all sites, converting.
template <int MODE, bool DIG>
__global__ void __launch_bounds__(128, DIG ? 5 : 3) k_link_deriv_fx(ForceArgs A, Digits D, int t0, int m, bool wrap)
{
    const Geom &g = A.g;
    const int own = blockIdx.x * blockDim.x + threadIdx.x, t = t0 + own;
    if (own >= m) return;
    const int i = t >> 1;
    const int row = fdiv(i, g.div_h3);
    const int r1 = fdiv(row, g.div_d2);
    const int x2 = row - r1 * g.d[2], x0 = fdiv(r1, g.div_d1), x1 = r1 - x0 * g.d[1];
    const int x3 = t - row * g.d[3];
    const int p = (x0 + x1 + x2 + x3) & 1;
    const long long V = 2LL * g.vh;
    // own fields: DIG reads them again for each direction (L1), which leaves registers
    // for five blocks an SM instead of three; a conversion is kept
    fx ax[DIG ? 1 : 16], bx[DIG ? 1 : 16];
    int ea = 0, eb = 0;
    auto load = [&](int f, int par, int idx, int slot, fx(&v)[16], int &E) -> bool {
        if constexpr (DIG) return load_digits(D, f, slot, v, E);
        else return load_fx(f ? A.b[par] : A.a[par], idx, v, E);
    };
    bool ok_own = true;
    if constexpr (!DIG) {
        ok_own = load(0, p, i, own, ax, ea);
        ok_own = load(1, p, i, own, bx, eb) && ok_own;
    }
#pragma unroll 1
    for (int mu = 0; mu < 4; ++mu) {
        const int xm = mu == 0 ? x0 : mu == 1 ? x1 : mu == 2 ? x2 : x3;
        const bool edge = xm == g.d[mu] - 1;
        const int stride = mu == 3 ? 1 : g.d[3] * (mu == 2 ? 1 : g.d[2] * (mu == 1 ? 1 : g.d[1]));
        const int tf = edge ? t - (g.d[mu] - 1) * stride : t + stride, ifw = tf >> 1;
        const int slot = mu == 0 && !wrap ? own + stride : own + (tf - t);
        const double sg = (MODE == 1 && edge && ((g.bc >> mu) & 1)) ? -A.beta : A.beta;
        fxa g1[4] = {}, g2[4] = {};
        int eaf, ebf;
        bool ok = ok_own;
        {
            fx s[16], h[8], hb[8];
            ok = load(0, 1 - p, ifw, slot, s, eaf) && ok;
            project_fx(mu, false, s, h);  // (1 + g) a(x + mu)
            if constexpr (DIG) {
                ok = load(1, p, i, own, s, eb) && ok;
                project_fx(mu, false, s, hb);
            } else {
                project_fx(mu, false, bx, hb);
            }
            mac_links<true>(g2, hb, h);
            ok = load(1, 1 - p, ifw, slot, s, ebf) && ok;
            project_fx(mu, true, s, hb);
            if constexpr (DIG) {
                ok = load(0, p, i, own, s, ea) && ok;
                project_fx(mu, true, s, h); // (1 - g) a(x)
            } else {
                project_fx(mu, true, ax, h);
            }
            mac_links<false>(g1, hb, h);
        }
        fx u[4];
        int eu = 127;
        if constexpr (MODE == 0) {
            const float4 *q = (const float4 *)A.gauge + ((size_t)(p * 4 + mu) * g.nblk_g + (i >> 5)) * 64 + (i & 31);
            const float4 hi = __ldg(q), lo = __ldg(q + 32);
            const unsigned m = max(max(__float_as_uint(hi.x) & 0x7fffffffu, __float_as_uint(hi.y) & 0x7fffffffu),
                                   max(__float_as_uint(hi.z) & 0x7fffffffu, __float_as_uint(hi.w) & 0x7fffffffu));
            eu = (int)(m >> 23);
            ok = ok && (m == 0 || (eu >= kFxMinExp && eu < 255));
            eu = min(max(eu, kFxMinExp), 254);
            const float sc = fx_pair_scale(eu);
            u[0] = fx_from_pair(hi.x, lo.x, sc);
            u[1] = fx_from_pair(hi.y, lo.y, sc);
            u[2] = fx_from_pair(hi.z, lo.z, sc);
            u[3] = fx_from_pair(hi.w, lo.w, sc);
        }
        // G = g1 + g2 at a common power of two (units of the sum: 2^(e - 56))
        const unsigned long long us1 = fx_used(g1[0]) | fx_used(g1[1]) | fx_used(g1[2]) | fx_used(g1[3]);
        const unsigned long long us2 = fx_used(g2[0]) | fx_used(g2[1]) | fx_used(g2[2]) | fx_used(g2[3]);
        const int s1 = fx_block_shift(us1), s2 = fx_block_shift(us2);
        const int e1 = us1 ? ea + ebf - 2 * kFxPairBias - s1 : -4096, e2 = us2 ? eaf + eb - 2 * kFxPairBias - s2 : -4096;
        const int e = max(max(e1, e2), -500); // (two zero sums; any others are far above)
        const int d1 = min(e - e1, 63), d2 = min(e - e2, 63);
        long long G[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) G[k] = (fx_shifted(g1[k], s1) >> d1) + (fx_shifted(g2[k], s2) >> d2);
        // below 2^-7 of the larger term's unit (2^(e1 + s1)): the digits, 2^-56 of it, would
        // hold less than the fields' 2^-49
        int used = 0; // high words: below 2^32 the sum is small enough whatever its bits
#pragma unroll
        for (int k = 0; k < 4; ++k) used |= (int)(G[k] >> 32) ^ (int)(G[k] >> 63);
        const int unit = max(us1 ? e1 + s1 : -4096, us2 ? e2 + s2 : -4096);
        if (!ok || 64 - __clz(used) + e - 56 < unit - 7) {
            const double sgn = sg == A.beta ? 1.0 : -1.0;
            if (mu == 0) link_terms_native<0>(A, p, i, ifw, t, sgn);
            else if (mu == 1) link_terms_native<1>(A, p, i, ifw, t, sgn);
            else if (mu == 2) link_terms_native<2>(A, p, i, ifw, t, sgn);
            else link_terms_native<3>(A, p, i, ifw, t, sgn);
        } else if constexpr (MODE == 1) {
            const double f = sg * fx_pow2(e - 56);
            double *o = A.out + ((long long)mu * V + t) * 4;
#pragma unroll
            for (int k = 0; k < 4; ++k) o[k] += f * (double)G[k];
        } else {
            fx c[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) c[k] = fx_split(G[k]);
            const fx n0 = fx_neg(c[0]);
            // u0 G - G0 u - u x G
            const fx n1 = fx_neg(c[1]), n2 = fx_neg(c[2]), n3 = fx_neg(c[3]);
            fxa F[3] = {};
            fx_mac(F[0], u[0], c[1]); fx_mac(F[0], u[1], n0); fx_mac(F[0], u[2], n3); fx_mac(F[0], u[3], c[2]);
            fx_mac(F[1], u[0], c[2]); fx_mac(F[1], u[2], n0); fx_mac(F[1], u[3], n1); fx_mac(F[1], u[1], c[3]);
            fx_mac(F[2], u[0], c[3]); fx_mac(F[2], u[3], n0); fx_mac(F[2], u[1], n2); fx_mac(F[2], u[2], c[1]);
            const double f = sg * fx_pow2(e - 56 + eu - kFxPairBias - 1);
            double *o = A.out + ((long long)mu * V + t) * 3;
#pragma unroll
            for (int k = 0; k < 3; ++k) o[k] += f * (double)fx_round(F[k]);
        }
    }
}

} // namespace

namespace hr {

hr_status link_deriv(hr_ctx *ctx, hr_lattice lat, const void *gauge, const void *a_even, const void *a_odd,
                     const void *b_even, const void *b_odd, double beta, double *out, int mode, cudaStream_t s)
{
    if (!ctx) return HR_ERR_INVALID_ARG;
    hr_status st = validate_lattice(ctx, lat, 1);
    if (st) return st;
    if (mode == 0 && !gauge) return set_error(ctx, HR_ERR_INVALID_ARG, "null pointer");
    st = check_buffers(ctx, {a_even, a_odd, b_even, b_odd}, {out}, {gauge});
    if (st) return st;
    ForceArgs A;
    A.g = make_geom(lat, 1);
    A.gauge = gauge;
    A.a[0] = a_even;
    A.a[1] = a_odd;
    A.b[0] = b_even;
    A.b[1] = b_odd;
    A.beta = beta;
    A.out = out;
    A.mode = mode;
    for (int k = 0; k < 4; ++k) {
        A.tc[k] = std::cos(lat.theta[k]);
        A.ts[k] = std::sin(lat.theta[k]);
    }
    const int bs = 128, V = 2 * A.g.vh;
    auto blocks = [&](int n) { return (unsigned)((n + bs - 1) / bs); };
    if (A.g.twisted) {
        k_link_deriv<<<blocks(V), bs, 0, s>>>(A);
        return check_launch(ctx, mode ? "link grad" : "force");
    }
    const Slabs slabs = make_slabs(A.g, kDigitSiteBytes);
    const SlabLease slab(ctx, s, slabs.n > 0);
    if (!slab.mem) {
        if (mode == 0) k_link_deriv_fx<0, false><<<blocks(V), bs, 0, s>>>(A, Digits{}, 0, V, true);
        else k_link_deriv_fx<1, false><<<blocks(V), bs, 0, s>>>(A, Digits{}, 0, V, true);
        return check_launch(ctx, mode ? "link grad" : "force");
    }
    const int slice = V / A.g.d[0];
    for (int k = 0; k < slabs.n; ++k) {
        const bool whole = slabs.n == 1;
        const int t0 = slabs.lo(k) * slice, m = (slabs.hi(k) - slabs.lo(k)) * slice, n = whole ? m : m + slice;
        int4 *d = (int4 *)slab.mem;
        int *e = (int *)(d + 16LL * n);
        k_field_digits<<<dim3(blocks(n), 2), bs, 0, s>>>(A, t0, n, d, e);
        if (mode == 0) k_link_deriv_fx<0, true><<<blocks(m), bs, 0, s>>>(A, Digits{d, e, n}, t0, m, whole);
        else k_link_deriv_fx<1, true><<<blocks(m), bs, 0, s>>>(A, Digits{d, e, n}, t0, m, whole);
    }
    return check_launch(ctx, mode ? "link grad" : "force");
}

} // namespace hr

namespace {

// the same on full packed fields
hr_status launch(hr_ctx *ctx, hr_lattice lat, const void *gauge, const void *af, const void *bf, double beta,
                 double *out, int mode, hr_stream stream)
{
    if (!ctx) return HR_ERR_INVALID_ARG;
    hr_status st = validate_lattice(ctx, lat, 1);
    if (st) return st;
    if (mode == 0 && !gauge) return set_error(ctx, HR_ERR_INVALID_ARG, "null pointer");
    st = check_buffers(ctx, {af, bf}, {out}, {gauge});
    if (st) return st;
    const size_t half = spinor_half_bytes(make_geom(lat, 1), HR_FUND, kF64);
    return link_deriv(ctx, lat, gauge, af, (const char *)af + half, bf, (const char *)bf + half, beta, out, mode,
                      (cudaStream_t)stream);
}

// Link derivative of B(X, L) = Re<L, Mhat^+ Mhat X> at fixed even fields X, L
// (Sec. 2.1: the even-odd operator in the HMC).  With Mhat = (4+m0) - c H_eo H_oe,
// c = 1 / (4 (4+m0)), and H_eo^+ = g5 H_oe g5,
//   dB = Re<Mhat L, dMhat X> + Re<Mhat X, dMhat L>,
//   Re<Y, dMhat Z> = -c dRe<(Y, H_eo^+ Y), H (Z, H_oe Z)>,
// so each of the two terms is one application of the hop derivative (mode 0:
// su(2) force, 1: quaternion gradient) to full fields a = (Mhat Y, H_eo^+ Mhat Y)
// and b = (Z, H_oe Z): L = X needs one (doubled).  H_oe Z is the first hop of
// Mhat Z, kept from there: three hops per term (hr_fermion_force at 32^4 818 us
// with the fourth and a copy of Z).
struct FermionWork {
    char *a, *b, *t; // two full fields and an odd half field
    static size_t bytes(const Geom &g)
    {
        const size_t half = spinor_half_bytes(g, HR_FUND, kF64);
        return 5 * half;
    }
};

hr_status fermion_deriv(hr_ctx *ctx, hr_lattice lat, double m0, hr_rep rep, const void *gauge, const void *X,
                        const void *L, double coeff, double *out, int mode, void *work, size_t work_bytes,
                        hr_stream stream)
{
    if (!ctx) return HR_ERR_INVALID_ARG;
    if (!valid_rep(rep)) return set_error(ctx, HR_ERR_INVALID_ARG, "bad rep");
    if (rep != HR_FUND)
        return set_error(ctx, HR_ERR_UNSUPPORTED, "the fermion force is implemented for fundamental links only");
    hr_status st = validate_lattice(ctx, lat, 1);
    if (st) return st;
    st = check_buffers(ctx, {gauge, X, work}, {out}, {L});
    if (st) return st;
    if (!(4.0 + m0 != 0.0) || !std::isfinite(m0)) return set_error(ctx, HR_ERR_INVALID_ARG, "4 + m0 must be nonzero");
    if (!std::isfinite(coeff)) return set_error(ctx, HR_ERR_INVALID_ARG, "coeff is not finite");
    const Geom g = make_geom(lat, 1);
    const size_t half = spinor_half_bytes(g, HR_FUND, kF64);
    const size_t need = FermionWork::bytes(g);
    if (work_bytes < need)
        return set_error(ctx, HR_ERR_WORKSPACE, "workspace of %zu bytes needed, %zu given", need, work_bytes);
    cudaStream_t s = (cudaStream_t)stream;
    FermionWork w{(char *)work, (char *)work + 2 * half, (char *)work + 4 * half};
    const double c = 1.0 / (4.0 * (4.0 + m0));
    // mz = Mhat Z, hz = H_oe Z
    auto schur = [&](const void *Z, void *mz, void *hz) {
        return apply_eo_op(ctx, g, m0, HR_FUND, kF64, HR_OP_SCHUR, gauge, Z, mz, hz, nullptr, kFinNone, nullptr, nullptr,
                           s);
    };
    // out += coeff * (-c) * k * dRe<(my, H_eo^+ my), H (Z, hz)>, H_eo^+ my = g5 H_oe g5 my in w.a's odd half
    auto term = [&](const void *my, const void *Z, const void *hz, double k) {
        HopLaunch H{};
        H.p = 1;
        H.gauge = gauge;
        H.in = my;
        H.out = w.a + half;
        H.beta = 1.0;
        H.g5_in = H.g5_out = 1;
        hr_status t = launch_hop(ctx, g, HR_FUND, kF64, H, s);
        if (!t) t = link_deriv(ctx, lat, gauge, my, w.a + half, Z, hz, -c * k * coeff, out, mode, s);
        return t;
    };
    st = schur(X, w.b, w.b + half);
    if (st) return st;
    if (!L || L == X) return term(w.b, X, w.b + half, 2.0);
    st = schur(L, w.a, w.t);
    if (!st) st = term(w.a, X, w.b + half, 1.0);
    if (!st) st = term(w.b, L, w.t, 1.0);
    return st;
}

} // namespace

extern "C" {

size_t hr_fermion_force_workspace_bytes(hr_lattice lat)
{
    return 5 * hr_spinor_packed_bytes(lat, HR_FUND, HR_F64, HR_EVEN, 1);
}

hr_status hr_fermion_force(hr_ctx *ctx, hr_lattice lat, double m0, hr_rep rep, const void *gauge, const void *X,
                           const void *L, double coeff, double *force, void *work, size_t work_bytes,
                           hr_stream stream)
{
    return fermion_deriv(ctx, lat, m0, rep, gauge, X, L, coeff, force, 0, work, work_bytes, stream);
}

hr_status hr_fermion_link_grad(hr_ctx *ctx, hr_lattice lat, double m0, hr_rep rep, const void *gauge, const void *X,
                               const void *L, double coeff, double *grad, void *work, size_t work_bytes,
                               hr_stream stream)
{
    return fermion_deriv(ctx, lat, m0, rep, gauge, X, L, coeff, grad, 1, work, work_bytes, stream);
}

hr_status hr_force(hr_ctx *ctx, hr_lattice lat, const void *gauge, const void *a_full, const void *b_full,
                   double beta, double *force, hr_stream stream)
{
    return launch(ctx, lat, gauge, a_full, b_full, beta, force, 0, stream);
}

hr_status hr_link_grad(hr_ctx *ctx, hr_lattice lat, const void *a_full, const void *b_full, double beta,
                       double *grad, hr_stream stream)
{
    return launch(ctx, lat, nullptr, a_full, b_full, beta, grad, 1, stream);
}

} // extern "C"
