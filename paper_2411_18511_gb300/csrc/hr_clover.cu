// hr_clover.cu -- the clover and exponential-clover site terms
// (arXiv:2411.18511 Sec. 2.2): building the packed field once per gauge field
// (A and A^-1, or (4+m0) exp(+-c_sw C/(4+m0)), on both parities), converting it
// to FP32 for the mixed-precision operators, applying it on one parity, and
// the full and even-odd operators with the site term.  The products inside the
// hop (A_ee on the aux term, A_oo^-1 on the result) run in the hop epilogue
// (hr_hop_dev.cuh), so every hop kernel variant carries them.
//
// Build (fundamental: fixed point, k_clover_build_fx; else native FP64).  Per site x:
//   Q_mn   the four leaves of the (mu, nu) plane from x, mu-first,
//   F_mn = (Q_mn - Q_mn^+) / 8, B_l = e_jkl F_jk / 2 (B_1 = F_23, B_2 = F_31, B_3 = F_12),
//   in the chiral basis s_0k = diag(-s_k, s_k) and s_jk = -e_jkl diag(s_l, s_l), so
//   C = (i/4) sum s_mn F_mn = diag(C+, C-),
//   C+ = sum_l s_l (x) (-(i/2)(F_0l + B_l)),   C- = sum_l s_l (x) ((i/2)(F_0l - B_l)),
//   clover:      A = (4+m0) + c_sw C,            A^-1 by Gauss-Jordan elimination,
//   exponential: A = (4+m0) exp(c_sw C/(4+m0)),  A^-1 = exp(-c_sw C/(4+m0)) / (4+m0),
// the exponential by scaling and squaring of a degree-16 Taylor polynomial
// (the argument is scaled below 1/2 in the 1-norm: truncation < 1e-19).
// Storing the explicit inverse instead of LDL factors: the same n^2 reals, and
// a matrix-vector product has no sequential dependency chain.
#include <algorithm>
#include <cmath>

#include "hr_clover.cuh"
#include "hr_clover_leaf.cuh"
#include "hr_eigh.cuh"
#include "hr_fix_dev.cuh"
#include "hr_host.h"
#include "hr_plaq.cuh"

using namespace hr;

namespace {

struct zc {
    double re, im;
};
__device__ __forceinline__ zc zadd(zc a, zc b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ zc zsub(zc a, zc b) { return {a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ zc zmul(zc a, zc b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ zc zconj(zc a) { return {a.re, -a.im}; }
__device__ __forceinline__ zc zscale(double s, zc a) { return {s * a.re, s * a.im}; }

template <int NC> struct CM {
    zc m[NC][NC];
};

// U_mu(x) as a colour matrix from the canonical quaternion (fundamental
// 2x2, or the real adjoint R_ab = 1/2 tr(s_a U s_b U^+))
template <int NC> __device__ CM<NC> link_mat(const double *can, long long V, int mu, long long x)
{
    const double *q = can + ((long long)mu * V + x) * 4;
    const double a0 = q[0], a1 = q[1], a2 = q[2], a3 = q[3];
    CM<NC> U;
    if constexpr (NC == 2) {
        U.m[0][0] = {a0, a3};
        U.m[0][1] = {a2, a1};
        U.m[1][0] = {-a2, a1};
        U.m[1][1] = {a0, -a3};
    } else {
        const double w = a0 * a0 - (a1 * a1 + a2 * a2 + a3 * a3);
        const double a[3] = {a1, a2, a3};
        for (int r = 0; r < 3; ++r)
            for (int c = 0; c < 3; ++c) U.m[r][c] = {2.0 * a[r] * a[c] + (r == c ? w : 0.0), 0.0};
        U.m[0][1].re += 2.0 * a0 * a3;
        U.m[0][2].re -= 2.0 * a0 * a2;
        U.m[1][0].re -= 2.0 * a0 * a3;
        U.m[1][2].re += 2.0 * a0 * a1;
        U.m[2][0].re += 2.0 * a0 * a2;
        U.m[2][1].re -= 2.0 * a0 * a1;
    }
    return U;
}

// A B, with either factor optionally daggered
template <int NC> __device__ CM<NC> cmul(const CM<NC> &A, bool da, const CM<NC> &B, bool db)
{
    CM<NC> C;
    for (int r = 0; r < NC; ++r)
        for (int c = 0; c < NC; ++c) {
            zc s = {0.0, 0.0};
            for (int k = 0; k < NC; ++k) {
                const zc a = da ? zconj(A.m[k][r]) : A.m[r][k];
                const zc b = db ? zconj(B.m[c][k]) : B.m[k][c];
                s = zadd(s, zmul(a, b));
            }
            C.m[r][c] = s;
        }
    return C;
}

__device__ long long lex_of(const Geom &g, const int (&x)[4])
{
    return (((long long)x[0] * g.d[1] + x[1]) * g.d[2] + x[2]) * g.d[3] + x[3];
}
// the site x + s1 m1 + s2 m2 (periodic; s = 0 leaves a direction alone)
__device__ long long nb(const Geom &g, const int (&x)[4], int m1, int s1, int m2 = 0, int s2 = 0)
{
    int y[4] = {x[0], x[1], x[2], x[3]};
    y[m1] = (y[m1] + s1 + g.d[m1]) % g.d[m1];
    y[m2] = (y[m2] + s2 + g.d[m2]) % g.d[m2];
    return lex_of(g, y);
}

// F_mn(x) = (Q_mn - Q_mn^+)/8 from the four leaves that start at x
template <int NC> __device__ CM<NC> field_strength(const Geom &g, const double *can, const int (&x)[4], int mu, int nu)
{
    const long long V = 2LL * g.vh;
    const long long x0 = lex_of(g, x);
    const long long xpm = nb(g, x, mu, 1), xpn = nb(g, x, nu, 1), xmm = nb(g, x, mu, -1), xmn = nb(g, x, nu, -1);
    const long long xmm_pn = nb(g, x, mu, -1, nu, 1), xmm_mn = nb(g, x, mu, -1, nu, -1), xmn_pm = nb(g, x, nu, -1, mu, 1);
    auto U = [&](int d, long long s) { return link_mat<NC>(can, V, d, s); };
    // U_mu(x) U_nu(x+mu) U_mu(x+nu)^+ U_nu(x)^+
    CM<NC> Q = cmul(cmul(U(mu, x0), false, U(nu, xpm), false), false, cmul(U(nu, x0), false, U(mu, xpn), false), true);
    // U_nu(x) U_mu(x-mu+nu)^+ U_nu(x-mu)^+ U_mu(x-mu)
    CM<NC> t = cmul(cmul(U(nu, x0), false, U(mu, xmm_pn), true), false, cmul(U(nu, xmm), true, U(mu, xmm), false), false);
    for (int r = 0; r < NC; ++r)
        for (int c = 0; c < NC; ++c) Q.m[r][c] = zadd(Q.m[r][c], t.m[r][c]);
    // U_mu(x-mu)^+ U_nu(x-mu-nu)^+ U_mu(x-mu-nu) U_nu(x-nu)
    t = cmul(cmul(U(nu, xmm_mn), false, U(mu, xmm), false), true, cmul(U(mu, xmm_mn), false, U(nu, xmn), false), false);
    for (int r = 0; r < NC; ++r)
        for (int c = 0; c < NC; ++c) Q.m[r][c] = zadd(Q.m[r][c], t.m[r][c]);
    // U_nu(x-nu)^+ U_mu(x-nu) U_nu(x-nu+mu) U_mu(x)^+
    t = cmul(cmul(U(nu, xmn), true, U(mu, xmn), false), false, cmul(U(mu, x0), false, U(nu, xmn_pm), true), true);
    for (int r = 0; r < NC; ++r)
        for (int c = 0; c < NC; ++c) Q.m[r][c] = zadd(Q.m[r][c], t.m[r][c]);
    CM<NC> F;
    for (int r = 0; r < NC; ++r)
        for (int c = 0; c < NC; ++c) F.m[r][c] = zscale(0.125, zsub(Q.m[r][c], zconj(Q.m[c][r])));
    return F;
}

template <int N> struct ZM {
    zc m[N][N];
};

template <int N> __device__ ZM<N> zmm(const ZM<N> &A, const ZM<N> &B)
{
    ZM<N> C;
#pragma unroll 1
    for (int r = 0; r < N; ++r)
        for (int c = 0; c < N; ++c) {
            zc s = {0.0, 0.0};
            for (int k = 0; k < N; ++k) s = zadd(s, zmul(A.m[r][k], B.m[k][c]));
            C.m[r][c] = s;
        }
    return C;
}

// exp(X) by scaling and squaring of the degree-16 Taylor polynomial
template <int N> __device__ ZM<N> expm(ZM<N> X)
{
    double nrm = 0.0;
    for (int c = 0; c < N; ++c) {
        double s = 0.0;
        for (int r = 0; r < N; ++r) s += hypot(X.m[r][c].re, X.m[r][c].im);
        nrm = fmax(nrm, s);
    }
    int sq = 0;
    while (nrm > 0.5 && sq < 60) {
        nrm *= 0.5;
        ++sq;
    }
    const double sc = ldexp(1.0, -sq);
    for (int r = 0; r < N; ++r)
        for (int c = 0; c < N; ++c) X.m[r][c] = zscale(sc, X.m[r][c]);
    // Horner: E = 1 + X (1 + X/2 (1 + X/3 (... (1 + X/16))))
    ZM<N> E;
    for (int r = 0; r < N; ++r)
        for (int c = 0; c < N; ++c) E.m[r][c] = {r == c ? 1.0 : 0.0, 0.0};
#pragma unroll 1
    for (int k = 16; k >= 1; --k) {
        ZM<N> T = zmm(X, E);
        for (int r = 0; r < N; ++r)
            for (int c = 0; c < N; ++c) E.m[r][c] = zadd(zscale(1.0 / k, T.m[r][c]), {r == c ? 1.0 : 0.0, 0.0});
    }
#pragma unroll 1
    for (int k = 0; k < sq; ++k) E = zmm(E, E);
    return E;
}

// A^-1 by Gauss-Jordan elimination with partial pivoting (false if singular)
template <int N> __device__ bool inverse(ZM<N> A, ZM<N> &I)
{
    for (int r = 0; r < N; ++r)
        for (int c = 0; c < N; ++c) I.m[r][c] = {r == c ? 1.0 : 0.0, 0.0};
#pragma unroll 1
    for (int k = 0; k < N; ++k) {
        int piv = k;
        double best = -1.0;
        for (int r = k; r < N; ++r) {
            const double m = A.m[r][k].re * A.m[r][k].re + A.m[r][k].im * A.m[r][k].im;
            if (m > best) {
                best = m;
                piv = r;
            }
        }
        if (!(best > 0.0)) return false;
        if (piv != k)
            for (int c = 0; c < N; ++c) {
                zc t = A.m[k][c];
                A.m[k][c] = A.m[piv][c];
                A.m[piv][c] = t;
                t = I.m[k][c];
                I.m[k][c] = I.m[piv][c];
                I.m[piv][c] = t;
            }
        const zc p = A.m[k][k];
        const double pn = p.re * p.re + p.im * p.im;
        const zc pinv = {p.re / pn, -p.im / pn};
        for (int c = 0; c < N; ++c) {
            A.m[k][c] = zmul(A.m[k][c], pinv);
            I.m[k][c] = zmul(I.m[k][c], pinv);
        }
        for (int r = 0; r < N; ++r) {
            if (r == k) continue;
            const zc f = A.m[r][k];
            for (int c = 0; c < N; ++c) {
                A.m[r][c] = zsub(A.m[r][c], zmul(f, A.m[k][c]));
                I.m[r][c] = zsub(I.m[r][c], zmul(f, I.m[k][c]));
            }
        }
    }
    return true;
}

// the n^2 reals of a Hermitian block (diagonal, then the upper triangle as re, im)
template <int N> __device__ void block_reals(const ZM<N> &M, double *out)
{
    int r = 0;
    for (int k = 0; k < N; ++k) out[r++] = M.m[k][k].re;
    for (int p = 0; p < N; ++p)
        for (int q = p + 1; q < N; ++q) {
            out[r++] = M.m[p][q].re;
            out[r++] = M.m[p][q].im;
        }
}

template <int NC, int CP> __device__ void store_site(void *half, int i, const double *reals)
{
    using L = CloverLayout<NC, CP>;
    float4 *base = (float4 *)half;
#pragma unroll 1
    for (int v = 0; v < L::NVEC; ++v) {
        float4 w;
        if constexpr (CP == kF64) {
            const double a = reals[2 * v], b = reals[2 * v + 1];
            const float ah = (float)a, bh = (float)b;
            w = make_float4(ah, (float)(a - (double)ah), bh, (float)(b - (double)bh));
        } else {
            w = make_float4((float)reals[4 * v], (float)reals[4 * v + 1], (float)reals[4 * v + 2],
                            (float)reals[4 * v + 3]);
        }
        base[((size_t)(i >> 5) * L::NVEC + v) * 32 + (i & 31)] = w;
    }
}

struct BuildArgs {
    Geom g;
    const double *can;
    double m0, csw;
    int kind;
    void *half[4]; // A even, A odd, A^-1 even, A^-1 odd
    unsigned *bad; // kBuildSingular, kBuildOutside
};
// an A is singular; a site lies outside the fixed-point range (the whole field is then built in native FP64)
constexpr unsigned kBuildSingular = 1u, kBuildOutside = 2u;

// one lexicographic site in native FP64
template <int NC, int CP> __device__ void build_site(const BuildArgs &B, long long t)
{
    constexpr int N = 2 * NC;
    const Geom &g = B.g;
    int x[4];
    long long r = t;
    for (int k = 3; k >= 0; --k) {
        x[k] = (int)(r % g.d[k]);
        r /= g.d[k];
    }
    const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
    const int i = (int)(t >> 1);
    // F_mn for the six planes
    CM<NC> F01 = field_strength<NC>(g, B.can, x, 0, 1), F02 = field_strength<NC>(g, B.can, x, 0, 2),
           F03 = field_strength<NC>(g, B.can, x, 0, 3), F12 = field_strength<NC>(g, B.can, x, 1, 2),
           F13 = field_strength<NC>(g, B.can, x, 1, 3), F23 = field_strength<NC>(g, B.can, x, 2, 3);
    const CM<NC> *E[3] = {&F01, &F02, &F03};
    const double a = 4.0 + B.m0;
    double reals[2][2 * N * N]; // [forward / inverse][both blocks]
#pragma unroll 1
    for (int b = 0; b < 2; ++b) {
        // G_l = -(i/2)(F_0l + B_l) (upper block) or (i/2)(F_0l - B_l) (lower)
        ZM<N> C;
        for (int rr = 0; rr < N; ++rr)
            for (int cc = 0; cc < N; ++cc) C.m[rr][cc] = {0.0, 0.0};
        for (int l = 0; l < 3; ++l) {
            const CM<NC> &Bm = l == 0 ? F23 : l == 1 ? F13 : F12;
            const double sB = l == 1 ? -1.0 : 1.0; // B_2 = F_31 = -F_13
            for (int c = 0; c < NC; ++c)
                for (int d = 0; d < NC; ++d) {
                    const zc f = E[l]->m[c][d], bb = zscale(sB, Bm.m[c][d]);
                    const zc s = b == 0 ? zadd(f, bb) : zsub(f, bb);
                    // times -(i/2) or +(i/2)
                    const double h = b == 0 ? -0.5 : 0.5;
                    const zc G = {-h * s.im, h * s.re};
                    // s_l (x) G: s_1 = [[0,1],[1,0]], s_2 = [[0,-i],[i,0]], s_3 = diag(1,-1)
                    if (l == 0) {
                        C.m[c][NC + d] = zadd(C.m[c][NC + d], G);
                        C.m[NC + c][d] = zadd(C.m[NC + c][d], G);
                    } else if (l == 1) {
                        C.m[c][NC + d] = zadd(C.m[c][NC + d], {G.im, -G.re});  // -i G
                        C.m[NC + c][d] = zadd(C.m[NC + c][d], {-G.im, G.re});  // +i G
                    } else {
                        C.m[c][d] = zadd(C.m[c][d], G);
                        C.m[NC + c][NC + d] = zsub(C.m[NC + c][NC + d], G);
                    }
                }
        }
        ZM<N> A, Ai;
        if (B.kind == HR_CLOVER_EXP) {
            ZM<N> X = C, Y = C;
            for (int rr = 0; rr < N; ++rr)
                for (int cc = 0; cc < N; ++cc) {
                    X.m[rr][cc] = zscale(B.csw / a, C.m[rr][cc]);
                    Y.m[rr][cc] = zscale(-B.csw / a, C.m[rr][cc]);
                }
            A = expm(X);
            Ai = expm(Y);
            for (int rr = 0; rr < N; ++rr)
                for (int cc = 0; cc < N; ++cc) {
                    A.m[rr][cc] = zscale(a, A.m[rr][cc]);
                    Ai.m[rr][cc] = zscale(1.0 / a, Ai.m[rr][cc]);
                }
        } else {
            for (int rr = 0; rr < N; ++rr)
                for (int cc = 0; cc < N; ++cc)
                    A.m[rr][cc] = zadd(zscale(B.csw, C.m[rr][cc]), {rr == cc ? a : 0.0, 0.0});
            if (!inverse(A, Ai)) atomicOr(B.bad, kBuildSingular);
        }
        block_reals(A, &reals[0][b * N * N]);
        block_reals(Ai, &reals[1][b * N * N]);
    }
    store_site<NC, CP>(B.half[p], i, reals[0]);
    store_site<NC, CP>(B.half[2 + p], i, reals[1]);
}

// native FP64, one thread per lexicographic site: the adjoint field, and a
// fundamental one outside the fixed-point range
template <int NC, int CP> __global__ void __launch_bounds__(64) k_clover_build(BuildArgs B)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < 2LL * B.g.vh) build_site<NC, CP>(B, t);
}

// ---------------------------------------------------------------- fundamental build in fixed point
//
// For SU(2) fundamental links F_mn = (i/4) f_mn.s with f_mn the vector part of
// the sum of the four leaves (quaternions), so each chiral block is
//   C_b = sum_lk M_lk s_l (x) s_k,  M_lk = (f_0l + b_l)_k / 8 (upper), -(f_0l - b_l)_k / 8 (lower),
// real coefficients, and the whole site term lives in the four-dimensional
// algebra of 1, X, X^2, X^3, X = sum N_lk s_l (x) s_k, N = c_sw M / a, a = 4 + m0:
//   X^2 = t - 2 K,  X^3 = 3 t X - 6 d - 2 L,  X^4 = 2 t X^2 - 8 d X - q,
//   t = |N|^2, d = det N, K = cof N, L = N N^T N, q = t^2 - 4 |K|^2
// (matrices K, L read as K_lk s_l (x) s_k).  Clover: A = a (1 + X) and
//   A^-1 = [(1 - t - 2 d) - ((1 + t) N + 2 K - 2 L)] / (a D),  D = det(1 + X) = 1 - 2 t - 8 d + q;
// exponential: the Taylor series of exp(+-X) to degree 18 (|X| <= 1: remainder
// 8e-18) by Horner's rule on the four coefficients, three products a step
// where a 4 x 4 complex matrix product has 256.  All of it in two-digit fixed
// point (hr_fix.cuh).
// N is held as N' = 2^k N.  k = 0 on rough fields with c_sw / a of 1/16 or more.  Where
// every plaquette of a site comes from links near the identity (doubles,
// hr_plaq.cuh), a second pass takes them in units of the largest; a small c_sw / a
// adds its power of two.  A's numbers off the diagonal are then as accurate as they
// are small, and t, K, L, d, q, of second order and higher in N, are shifted back.
// A site with links off unit length, |N| too large, k above 40, numbers of very
// different size (a row of N below 2^-8 of the others: a pair holds 2^-49), D near
// 0 or a factor out of range sets kBuildOutside, and the call, which reads its
// status word in any case, builds the field again in native FP64 (a call to
// the native code inside this kernel would hold it at 255 registers).
// Measured: the clover solve of 24^4 (build, FP32-inner CG to 1e-10, links and
// source in, solution out) 9.75 ms with the native build, 3.36 ms of it the
// build, 7.03 ms with this one and 0.61 ms of it the build; leaves from the
// plaquettes' vectors took another 0.33 ms off that build (5.80 -> 5.47 ms for
// the solve by then); solution error against 64 bits unchanged.  The build alone at
// 32^4: 10.1 ms native; 0.915 (exponential 1.29) on rough links, of it 0.04 for N's
// own scale; 1.41 to 1.84 on links near the identity.

struct FxMat {
    fx m[3][3];
};

// vector part of the sum of the four leaves of the (mu, nu) plane at x, in units of 2^-56
// (top: raised to the largest vector component of the links)
template <bool VEC>
__device__ __forceinline__ void leaf_sum(const Geom &g, const double *can, const LexSite &x, int mu, int nu,
                                         long long (&f)[3], bool &ok, unsigned &top)
{
    int um, dm, un, dn;
    lex_steps(g, x, mu, um, dm);
    lex_steps(g, x, nu, un, dn);
    const size_t V = 2 * (size_t)g.vh, bm = (size_t)mu * V + x.t, bn = (size_t)nu * V + x.t;
    auto U = [&](size_t at) { return load_fxq<VEC>(can, at, ok, top); };
    fxa s[3] = {};
    const fxq a = U(bm), b = U(bn);
    // U_mu(x) U_nu(x+mu) [U_nu(x) U_mu(x+nu)]^+
    fxq l = fxq_mul(a, U(bn + um)), r = fxq_mul(b, U(bm + un));
    fxq_mac_vec(s, l, fxq_conj(r));
    // U_nu(x) U_mu(x-mu+nu)^+ U_nu(x-mu)^+ U_mu(x-mu)
    const fxq am = U(bm + dm);
    l = fxq_mul(b, fxq_conj(U(bm + dm + un)));
    r = fxq_mul(fxq_conj(U(bn + dm)), am);
    fxq_mac_vec(s, l, r);
    // [U_nu(x-mu-nu) U_mu(x-mu)]^+ U_mu(x-mu-nu) U_nu(x-nu)
    const fxq bd = U(bn + dn);
    l = fxq_conj(fxq_mul(U(bn + dm + dn), am));
    r = fxq_mul(U(bm + dm + dn), bd);
    fxq_mac_vec(s, l, r);
    // U_nu(x-nu)^+ U_mu(x-nu) [U_mu(x) U_nu(x-nu+mu)^+]^+
    l = fxq_mul(fxq_conj(bd), U(bm + dn));
    r = fxq_conj(fxq_mul(a, fxq_conj(U(bn + dn + um))));
    fxq_mac_vec(s, l, r);
#pragma unroll
    for (int k = 0; k < 3; ++k) f[k] = fx_round(s[k]);
}

// the 16 reals of a block u + 2^-k sum P_lk s_l (x) s_k (units of 2^-56), each times
// the digits `sc` and the power of two ksc, as pairs; k <= 100
__device__ __forceinline__ void block_pairs(long long u, const FxMat &P, int k, fx sc, float ksc, float2 (&out)[16])
{
    const float koff = ksc * fx_float((unsigned)(127 - k) << 23);
    auto pair_by = [&](long long t, float by) {
        fxa s = {0, 0};
        fx_mac(s, fx_split(t), sc);
        float2 v;
        fx_to_pair(fx_round(s), v.x, v.y);
        return make_float2(v.x * by, v.y * by);
    };
    auto pair = [&](long long t) { return pair_by(t, koff); };
    auto T = [](fx v) { return fx_units64(v); };
    auto neg = [](float2 v) { return make_float2(-v.x, -v.y); };
    const long long d = T(P.m[2][2]) >> min(k, 63);
    const float2 dp = pair_by(u + d, ksc), dm = pair_by(u - d, ksc);
    out[0] = dp; out[1] = dm; out[2] = dm; out[3] = dp;
    const float2 p31 = pair(T(P.m[2][0])), p32 = pair(T(P.m[2][1])), p13 = pair(T(P.m[0][2])), p23 = pair(T(P.m[1][2]));
    out[4] = p31; out[5] = neg(p32);                 // (0, 1)
    out[6] = p13; out[7] = neg(p23);                 // (0, 2)
    out[8] = pair(T(P.m[0][0]) - T(P.m[1][1]));      // (0, 3)
    out[9] = neg(pair(T(P.m[1][0]) + T(P.m[0][1])));
    out[10] = pair(T(P.m[0][0]) + T(P.m[1][1]));     // (1, 2)
    out[11] = pair(T(P.m[0][1]) - T(P.m[1][0]));
    out[12] = neg(p13); out[13] = p23;               // (1, 3)
    out[14] = neg(p31); out[15] = p32;               // (2, 3)
}
template <int CP> __device__ __forceinline__ void store_block(void *half, int i, int b, const float2 (&r)[16])
{
    using L = CloverLayout<2, CP>;
    float4 *base = (float4 *)half + (size_t)(i >> 5) * L::NVEC * 32 + (i & 31);
    if constexpr (CP == kF64) {
#pragma unroll
        for (int v = 0; v < 8; ++v) base[(8 * b + v) * 32] = make_float4(r[2 * v].x, r[2 * v].y, r[2 * v + 1].x, r[2 * v + 1].y);
    } else {
#pragma unroll
        for (int v = 0; v < 4; ++v)
            base[(4 * b + v) * 32] = make_float4(r[4 * v].x, r[4 * v + 1].x, r[4 * v + 2].x, r[4 * v + 3].x);
    }
}

// The same from the plaquettes' vectors of a slab that starts at slice `first`: the
// leaf at x of the plaquette below in mu is its vector transported by U_mu(x - mu),
// below in nu by U_nu(x - nu), and below in both by the one and then the other,
//   sum = P(x) + T_mu P(x - mu) + T_nu [P(x - nu) + T_mu P(x - mu - nu)].
// low: the transports by the four links below x.  One conversion and three
// transports of 15 products where the leaves take 16 conversions and 11
// quaternion products.
struct LowLinks {
    int4 (*w)[64]; // [4 mu + k][thread]
    __device__ void put(int mu, const Transport &T)
    {
        w[4 * mu + 0][threadIdx.x] = make_int4(T.u[0].h, T.u[0].l, T.u[1].h, T.u[1].l);
        w[4 * mu + 1][threadIdx.x] = make_int4(T.u[2].h, T.u[2].l, T.w[0].h, T.w[0].l);
        w[4 * mu + 2][threadIdx.x] = make_int4(T.w[1].h, T.w[1].l, T.w[2].h, T.w[2].l);
        w[4 * mu + 3][threadIdx.x] = make_int4(T.w[3].h, T.w[3].l, 0, 0);
    }
    __device__ Transport get(int mu) const
    {
        const int4 a = w[4 * mu][threadIdx.x], b = w[4 * mu + 1][threadIdx.x], c = w[4 * mu + 2][threadIdx.x],
                   e = w[4 * mu + 3][threadIdx.x];
        return {{{a.x, a.y}, {a.z, a.w}, {b.x, b.y}}, {{b.z, b.w}, {c.x, c.y}, {c.z, c.w}, {e.x, e.y}}};
    }
};
template <bool VEC>
__device__ __forceinline__ void leaf_sum_slab(const Geom &g, const double *can, const LexSite &x, const PlaqVecs &P,
                                              int first, const LowLinks &low, int mu, int nu, int E, long long (&f)[3],
                                              PlaqKinds &kinds, bool &ok)
{
    const int slice = g.d[1] * g.d[2] * g.d[3], own = x.t - first * slice, plane = plane_of(mu, nu);
    int unused, dm, dn;
    lex_steps(g, x, mu, unused, dm);
    lex_steps(g, x, nu, unused, dn);
    // (the slab's first slice is the one before its first site's, unless it is the whole lattice; nu > 0)
    const int sm = mu == 0 && x.x0 > first ? -slice : dm;
    fx v[3];
    load_plaq(P, plane, own, E, v, kinds);
#pragma unroll
    for (int k = 0; k < 3; ++k) f[k] = fx_units64(v[k]);
    load_plaq(P, plane, own + sm, E, v, kinds);
    const Transport Tm = low.get(mu);
    transport_add(Tm, v, f);
    long long h[3];
    load_plaq(P, plane, own + dn, E, v, kinds);
#pragma unroll
    for (int k = 0; k < 3; ++k) h[k] = fx_units64(v[k]);
    load_plaq(P, plane, own + sm + dn, E, v, kinds);
    const Transport Tw = make_transport(load_fxq<VEC>(can, (size_t)mu * 2 * g.vh + (x.t + dm + dn), ok), ok);
    transport_add(Tw, v, h);
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = fx_split(h[k]);
    const Transport Tn = low.get(nu);
    transport_add(Tn, v, f);
}

struct BuildFx {
    fx kappa;    // 2^kk c_sw / a
    int kk;
    fx am;       // a = am 2^ka, am in [1, 2)
    float ka;    // 2^ka
    double inva; // 1 / a
};

// The m sites from t0 on; SLAB: with the plaquettes' vectors of the slab from slice
// `first` on, else (slices too large for the scratch) from the 16 links of each plane.
template <int CP, bool EXP, bool VEC, bool SLAB>
__global__ void __launch_bounds__(64, 6) k_clover_build_fx(BuildArgs B, BuildFx X, PlaqVecs P, int t0, int m, int first)
{
    const Geom &g = B.g;
    __shared__ int4 low_words[SLAB ? 16 : 1][64]; // this thread's slots: no other thread reads them
    const int t = t0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= t0 + m) return;
    const unsigned bad = *(volatile const unsigned *)B.bad; // looked at once the first links are on their way
    const LexSite x = lex_site(g, t);
    const int p = (x.x0 + x.x1 + x.x2 + x.x3) & 1, i = t >> 1;
    bool ok = true;
    LowLinks low = {low_words};
    if constexpr (SLAB) {
#pragma unroll 1
        for (int mu = 0; mu < 4; ++mu) {
            int unused, dm;
            lex_steps(g, x, mu, unused, dm);
            low.put(mu, make_transport(load_fxq<VEC>(B.can, (size_t)mu * 2 * g.vh + (t + dm), ok), ok));
        }
    }
    if (bad & kBuildOutside) return; // the field will be built in native FP64
    FxMat N[2];
    int E = 1022; // vectors in units of 2^(E - 1022)
#pragma unroll 1
    for (;;) {
        bool rough = false;
        unsigned top = 0, least = 0xffffffffu; // over the rows from links near the identity
#pragma unroll 1
        for (int l = 0; l < 3; ++l) {
            long long e[3], f[3] = {0, 0, 0};
            PlaqKinds row;
            // B_1 = F_23, B_2 = F_31 = -F_13, B_3 = F_12
            const int mu = l == 0 ? 2 : 1, nu = l == 2 ? 2 : 3;
            if constexpr (SLAB) {
                // (one copy of the code for both: 32^4 945 -> 913 us, exponential 1440 -> 1293)
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) e[k] = f[k];
                    leaf_sum_slab<VEC>(g, B.can, x, P, first, low, h ? mu : 0, h ? nu : l + 1, E, f, row, ok);
                }
            } else {
                leaf_sum<VEC>(g, B.can, x, 0, l + 1, e, ok, row.top);
                leaf_sum<VEC>(g, B.can, x, mu, nu, f, ok, row.top);
            }
            ok = ok && !row.bad;
            rough = rough || row.rough;
            if (!row.rough) {
                top = max(top, row.top);
                if (row.top) least = min(least, row.top);
            }
            fx r[2][3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const long long bk = l == 1 ? -f[k] : f[k];
                fxa u = {0, 0}, d = {0, 0};
                fx_mac(u, fx_split((e[k] + bk) >> 3), X.kappa);
                fx_mac(d, fx_split((bk - e[k]) >> 3), X.kappa);
                r[0][k] = fx_of(u);
                r[1][k] = fx_of(d);
            }
#pragma unroll
            for (int b = 0; b < 2; ++b)
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    if (l == 0) N[b].m[0][k] = r[b][k];
                    else if (l == 1) N[b].m[1][k] = r[b][k];
                    else N[b].m[2][k] = r[b][k];
                }
        }
        const bool units = !SLAB || rough; // digits in units of 1 are what there is
        if (least != 0xffffffffu && least + (8u << 20) < (units ? kFxHigh1 : top)) ok = false;
        if (!ok || units || top == 0 || E < 1022) break;
        E = (int)(top >> 20) + 2; // below 1/4: a site sums eight of them
        if (E >= 1022) {
            E = 1022;
            break;
        }
        if (E < 1022 - 40) {
            ok = false;
            break;
        }
    }
    const int ks = 1022 - E + X.kk, k1 = min(ks, 63), k2 = min(2 * ks, 63), k3 = min(3 * ks, 63), k4 = min(4 * ks, 63);
    const long long one = 1LL << 56;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        const FxMat &n = N[b];
        fxa ta = {0, 0}, da = {0, 0}, ka = {0, 0};
        FxMat K, L;
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                fx_mac(ta, n.m[r][c], n.m[r][c]);
                const int r1 = (r + 1) % 3, r2 = (r + 2) % 3, c1 = (c + 1) % 3, c2 = (c + 2) % 3;
                fxa s = {0, 0};
                fx_mac(s, n.m[r1][c1], n.m[r2][c2]);
                fx_mac(s, fx_neg(n.m[r1][c2]), n.m[r2][c1]);
                K.m[r][c] = fx_of(s);
            }
        const long long ts = fx_round(ta), tt = ts >> k2;
        if (ts > one || (EXP && tt > one / 3)) ok = false;
        fx S[3][3]; // N N^T (symmetric)
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int c = r; c < 3; ++c) {
                fxa s = {0, 0};
#pragma unroll
                for (int k = 0; k < 3; ++k) fx_mac(s, n.m[r][k], n.m[c][k]);
                S[r][c] = S[c][r] = fx_of(s);
            }
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                fxa s = {0, 0};
#pragma unroll
                for (int k = 0; k < 3; ++k) fx_mac(s, S[r][k], n.m[k][c]);
                L.m[r][c] = fx_of(s);
                fx_mac(ka, K.m[r][c], K.m[r][c]);
            }
#pragma unroll
        for (int c = 0; c < 3; ++c) fx_mac(da, n.m[0][c], K.m[0][c]);
        const fx td = fx_split(tt);
        const long long dt = fx_round(da) >> k3;
        fxa qa = {-((4 * fx_round(ka)) >> k4), 0};
        fx_mac(qa, td, td);
        const long long qt = fx_round(qa);
        if (ks) { // K and L in N's units
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    K.m[r][c] = fx_split(fx_units64(K.m[r][c]) >> k1);
                    L.m[r][c] = fx_split(fx_units64(L.m[r][c]) >> k2);
                }
        }
        // coefficients of 1, X, X^2, X^3 of A / a and A^-1 a (clover: times D)
        FxMat P, Q;
        long long u, v;
        fx sc_inv;
        float ks_inv = 1.f;
        if constexpr (EXP) {
            const fx q = fx_split(-qt), d8 = fx_split(-8 * dt), t2 = fx_split(2 * tt);
#pragma unroll
            for (int inv = 0; inv < 2; ++inv) {
                // 1/k! 2^56 for k = 18 .. 0
                constexpr double rf[19] = {1.0 / 6402373705728000.0, 1.0 / 355687428096000.0, 1.0 / 20922789888000.0,
                                           1.0 / 1307674368000.0, 1.0 / 87178291200.0, 1.0 / 6227020800.0,
                                           1.0 / 479001600.0, 1.0 / 39916800.0, 1.0 / 3628800.0, 1.0 / 362880.0,
                                           1.0 / 40320.0, 1.0 / 5040.0, 1.0 / 720.0, 1.0 / 120.0, 1.0 / 24.0,
                                           1.0 / 6.0, 0.5, 1.0, 1.0};
                fx c0 = fx_split((long long)(rf[0] * 0x1p56)), c1 = {0, 0}, c2 = {0, 0}, c3 = {0, 0};
#pragma unroll 1
                for (int k = 1; k < 19; ++k) {
                    const long long f = (long long)(rf[k] * 0x1p56);
                    fxa s0 = {inv && (k & 1) ? -f : f, 0}, s1 = {fx_units64(c0), 0}, s2 = {fx_units64(c1), 0};
                    fx_mac(s0, q, c3);
                    fx_mac(s1, d8, c3);
                    fx_mac(s2, t2, c3);
                    c3 = c2;
                    c0 = fx_of(s0);
                    c1 = fx_of(s1);
                    c2 = fx_of(s2);
                }
                // c0 + c2 t - 6 d c3,  c1 + 3 t c3,  -2 c2,  -2 c3
                fxa w = {fx_units64(c0), 0}, e1 = {fx_units64(c1), 0};
                fx_mac(w, c2, td);
                fx_mac(w, c3, fx_split(-6 * dt));
                fx_mac(e1, c3, fx_split(3 * tt));
                const fx k1 = fx_of(e1), k2 = {-2 * c2.h, -2 * c2.l}, k3 = {-2 * c3.h, -2 * c3.l};
                FxMat &O = inv ? Q : P;
#pragma unroll
                for (int r = 0; r < 3; ++r)
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        fxa s = {0, 0};
                        fx_mac(s, k1, n.m[r][c]);
                        fx_mac(s, k2, K.m[r][c]);
                        fx_mac(s, k3, L.m[r][c]);
                        O.m[r][c] = fx_of(s);
                    }
                if (inv) v = fx_round(w);
                else u = fx_round(w);
            }
        } else {
            u = one;
            P = n;
            v = one - tt - 2 * dt;
            const fx t1 = fx_split(-one - tt);
#pragma unroll
            for (int r = 0; r < 3; ++r)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    fxa s = {2 * (fx_units64(L.m[r][c]) - fx_units64(K.m[r][c])), 0};
                    fx_mac(s, t1, n.m[r][c]);
                    Q.m[r][c] = fx_of(s);
                }
        }
        double inv = X.inva;
        if constexpr (!EXP) {
            const long long D = one - 2 * tt - 8 * dt + qt;
            if (D < one / 16) ok = false;
            inv = inv / fx_to_double(D);
        }
        {
            // 1 / a (clover: 1 / (a D)) = m 2^k, m in [1, 2)
            const unsigned long long ib = fx_dbits(inv);
            const int k = (int)(ib >> 52) - 1023;
            if (k < -60 || k > 60) ok = false;
            sc_inv = fx_from_double(fx_double((ib & 0xfffffffffffffULL) | 0x3ff0000000000000ULL));
            ks_inv = fx_float((unsigned)(127 + min(max(k, -60), 60)) << 23);
        }
        float2 out[16];
        block_pairs(u, P, ks, X.am, X.ka, out);
        store_block<CP>(B.half[p], i, b, out);
        block_pairs(v, Q, ks, sc_inv, ks_inv, out);
        store_block<CP>(B.half[2 + p], i, b, out);
    }
    if (!ok) atomicOr(B.bad, kBuildOutside);
}

template <int CP, bool EXP, bool VEC>
void launch_build_slabs(const BuildArgs &B, const BuildFx &X, const Slabs &slabs, void *scratch, cudaStream_t s)
{
    const Geom &g = B.g;
    const int slice = g.d[1] * g.d[2] * g.d[3];
    for (int k = 0; k < slabs.n; ++k) {
        const int a = slabs.lo(k), b = slabs.hi(k), first = slabs.n == 1 ? 0 : a - 1; // with the slice before it
        const int n = (b - first) * slice, m = (b - a) * slice;
        int4 *pa = (int4 *)scratch;
        int2 *pb = (int2 *)(pa + 6LL * n);
        launch_plaq_vec<VEC>(g, B.can, first, n, pa, pb, s);
        k_clover_build_fx<CP, EXP, VEC, true>
            <<<(unsigned)((m + 63) / 64), 64, 0, s>>>(B, X, PlaqVecs{pa, pb, n}, a * slice, m, first);
    }
}
template <int CP>
void launch_build_fx(hr_ctx *ctx, const BuildArgs &B, double a, cudaStream_t s)
{
    BuildFx X;
    int k;
    const double am = 2.0 * std::frexp(a, &k); // [1, 2)
    int e;
    std::frexp(B.csw / a, &e);
    X.kk = std::max(0, -3 - e); // from 1/16 on as it is, smaller ones between 1/16 and 1/8
    X.kappa = fx_from_double(std::ldexp(B.csw / a, X.kk));
    X.am = fx_from_double(am);
    X.ka = std::ldexp(1.f, k - 1);
    X.inva = 1.0 / a;
    const bool vec = ((uintptr_t)B.can & 15u) == 0, ex = B.kind == HR_CLOVER_EXP;
    const Slabs slabs = make_slabs(B.g, kPlaqSiteBytes);
    const SlabLease slab(ctx, s, slabs.n > 0);
    if (!slab.mem) {
        const int V = 2 * B.g.vh;
        (ex ? k_clover_build_fx<CP, true, false, false> : k_clover_build_fx<CP, false, false, false>)
            <<<(unsigned)((V + 63) / 64), 64, 0, s>>>(B, X, PlaqVecs{}, 0, V, 0);
    } else if (ex && vec) {
        launch_build_slabs<CP, true, true>(B, X, slabs, slab.mem, s);
    } else if (ex) {
        launch_build_slabs<CP, true, false>(B, X, slabs, slab.mem, s);
    } else if (vec) {
        launch_build_slabs<CP, false, true>(B, X, slabs, slab.mem, s);
    } else {
        launch_build_slabs<CP, false, false>(B, X, slabs, slab.mem, s);
    }
}

// FP64 -> FP32 field, one thread per FP32 vector
template <int NC> __global__ void k_clover_to_f32(int nvec_total, const float4 *src, float4 *dst)
{
    using L64 = CloverLayout<NC, kF64>;
    using L32 = CloverLayout<NC, kF32>;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nvec_total) return;
    const int lane = t & 31, v = (t >> 5) % L32::NVEC, blk = (t >> 5) / L32::NVEC;
    const float4 a = src[((size_t)blk * L64::NVEC + 2 * v) * 32 + lane];
    const float4 b = src[((size_t)blk * L64::NVEC + 2 * v + 1) * 32 + lane];
    dst[((size_t)blk * L32::NVEC + v) * 32 + lane] = make_float4(a.x + a.y, a.z + a.w, b.x + b.y, b.z + b.w);
}

// out = A in (or A^-1 in) on the sites of one parity (every right-hand side)
template <int NC, int PREC> __global__ void k_clover_apply(Geom g, const void *half, const void *in, void *out)
{
    using T = typename PrecTraits<PREC>::T;
    const int nv = g.vh << g.lrhs;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < nv; j += gridDim.x * blockDim.x) {
        cpx<T> v[4][NC];
        load_spinor<NC, PREC>(in, g.nblk_s, j, v);
        clover_apply<clover_prec(PREC)>(half, j >> g.lrhs, v);
        store_spinor<NC, PREC>(out, g.nblk_s, j, v);
    }
}

bool valid_clover_prec(int prec) { return prec == kF64 || prec == kF32; }

} // namespace

namespace hr {

size_t clover_half_bytes(const Geom &g, int rep, int cp)
{
    if (rep_nc(rep) == 2) return cp == kF64 ? CloverLayout<2, kF64>::half_bytes(g.nblk_g) : CloverLayout<2, kF32>::half_bytes(g.nblk_g);
    return cp == kF64 ? CloverLayout<3, kF64>::half_bytes(g.nblk_g) : CloverLayout<3, kF32>::half_bytes(g.nblk_g);
}

const void *clover_half(const void *base, const Geom &g, int rep, int cp, bool inverse, int parity)
{
    if (!base) return nullptr;
    return (const char *)base + (size_t)((inverse ? 2 : 0) + parity) * clover_half_bytes(g, rep, cp);
}

hr_status clover_convert_f32(hr_ctx *ctx, const Geom &g, int rep, const void *src, void *dst, cudaStream_t s)
{
    const int nc = rep_nc(rep);
    const size_t h64 = clover_half_bytes(g, rep, kF64), h32 = clover_half_bytes(g, rep, kF32);
    const int nvec = g.nblk_g * 32 * (nc == 2 ? CloverLayout<2, kF32>::NVEC : CloverLayout<3, kF32>::NVEC);
    const int bs = 256, grid = (nvec + bs - 1) / bs;
    for (int h = 0; h < 4; ++h) {
        const float4 *a = (const float4 *)((const char *)src + h * h64);
        float4 *b = (float4 *)((char *)dst + h * h32);
        if (nc == 2) k_clover_to_f32<2><<<grid, bs, 0, s>>>(nvec, a, b);
        else k_clover_to_f32<3><<<grid, bs, 0, s>>>(nvec, a, b);
    }
    return check_launch(ctx, "clover convert");
}

hr_status clover_apply_half(hr_ctx *ctx, const Geom &g, int rep, int prec, const void *half, const void *in,
                            void *out, cudaStream_t s)
{
    const long long nv = (long long)g.vh << g.lrhs;
    const int bs = 128, grid = grid_for(nv, bs, 1 << 30);
    const bool three = rep_nc(rep) == 3;
    switch (prec) {
    case kF64:
        if (three) k_clover_apply<3, kF64><<<grid, bs, 0, s>>>(g, half, in, out);
        else k_clover_apply<2, kF64><<<grid, bs, 0, s>>>(g, half, in, out);
        break;
    case kF32:
        if (three) k_clover_apply<3, kF32><<<grid, bs, 0, s>>>(g, half, in, out);
        else k_clover_apply<2, kF32><<<grid, bs, 0, s>>>(g, half, in, out);
        break;
    default:
        if (three) k_clover_apply<3, kF16><<<grid, bs, 0, s>>>(g, half, in, out);
        else k_clover_apply<2, kF16><<<grid, bs, 0, s>>>(g, half, in, out);
        break;
    }
    return check_launch(ctx, "clover apply");
}

} // namespace hr

extern "C" {

size_t hr_clover_packed_bytes(hr_lattice lat, hr_rep rep, hr_prec prec)
{
    if (!valid_rep(rep) || !valid_clover_prec(prec) || hr_gauge_packed_bytes(lat, rep, prec) == 0) return 0;
    return 4 * clover_half_bytes(make_geom(lat, 1), rep, prec);
}

hr_status hr_clover_build(hr_ctx *ctx, hr_lattice lat, hr_rep rep, hr_prec prec, hr_clover_kind kind, double m0,
                          double c_sw, const double *canonical, void *clover, hr_stream stream)
{
    if (!ctx) return HR_ERR_INVALID_ARG;
    if (!valid_rep(rep)) return set_error(ctx, HR_ERR_INVALID_ARG, "bad rep");
    if (!valid_clover_prec(prec)) return set_error(ctx, HR_ERR_UNSUPPORTED, "clover fields are FP64 or FP32");
    if (kind != HR_CLOVER_SW && kind != HR_CLOVER_EXP) return set_error(ctx, HR_ERR_INVALID_ARG, "bad clover kind");
    hr_status st = validate_lattice(ctx, lat, 1);
    if (st) return st;
    st = check_buffers(ctx, {clover}, {canonical});
    if (st) return st;
    if (!(4.0 + m0 != 0.0) || !std::isfinite(m0) || !std::isfinite(c_sw))
        return set_error(ctx, HR_ERR_INVALID_ARG, "4 + m0 must be nonzero and finite, c_sw finite");
    const Geom g = make_geom(lat, 1);
    cudaStream_t s = (cudaStream_t)stream;
    BuildArgs B;
    B.g = g;
    B.can = canonical;
    B.m0 = m0;
    B.csw = c_sw;
    B.kind = kind;
    for (int h = 0; h < 4; ++h) B.half[h] = (void *)clover_half(clover, g, rep, prec, h >= 2, h & 1);
    B.bad = ctx->d_counters + C_STATUS;
    const long long V = 2LL * g.vh;
    const int bs = 64, grid = (int)((V + bs - 1) / bs);
    const bool three = rep_nc(rep) == 3;
    // fixed point: fundamental links, 0 < a and |c_sw / a| within the digits' range
    const double a = 4.0 + m0;
    bool fixed = !three && a > 0x1p-20 && a < 0x1p20 && std::fabs(c_sw) < 2.0 * a &&
                 (c_sw == 0.0 || std::fabs(c_sw) > 0x1p-40 * a);
    unsigned bad = 0;
    for (;;) {
        cudaError_t e = cudaMemsetAsync(B.bad, 0, sizeof(unsigned), s);
        if (e != cudaSuccess) return set_error(ctx, HR_ERR_CUDA, "status reset: %s", cudaGetErrorString(e));
        if (prec == kF64) {
            if (fixed) launch_build_fx<kF64>(ctx, B, a, s);
            else if (three) k_clover_build<3, kF64><<<grid, bs, 0, s>>>(B);
            else k_clover_build<2, kF64><<<grid, bs, 0, s>>>(B);
        } else {
            if (fixed) launch_build_fx<kF32>(ctx, B, a, s);
            else if (three) k_clover_build<3, kF32><<<grid, bs, 0, s>>>(B);
            else k_clover_build<2, kF32><<<grid, bs, 0, s>>>(B);
        }
        st = check_launch(ctx, "clover build");
        if (st) return st;
        e = cudaMemcpyAsync(&bad, B.bad, sizeof bad, cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return set_error(ctx, HR_ERR_CUDA, "clover build status: %s", cudaGetErrorString(e));
        if (!(bad & kBuildOutside)) break;
        fixed = false;
    }
    if (bad & kBuildSingular) return set_error(ctx, HR_ERR_NUMERIC, "a clover site block is singular (no inverse)");
    return HR_OK;
}

hr_status hr_clover_apply(hr_ctx *ctx, hr_lattice lat, hr_rep rep, hr_prec prec, hr_parity parity, int inverse,
                          int n_rhs, const void *clover, const void *in, void *out, hr_stream stream)
{
    if (!ctx) return HR_ERR_INVALID_ARG;
    if (!valid_rep(rep) || !valid_prec(prec)) return set_error(ctx, HR_ERR_INVALID_ARG, "bad rep/prec");
    if (parity != HR_EVEN && parity != HR_ODD) return set_error(ctx, HR_ERR_INVALID_ARG, "parity HR_EVEN or HR_ODD");
    hr_status st = validate_lattice(ctx, lat, n_rhs);
    if (st) return st;
    st = check_buffers(ctx, {clover, in, out});
    if (st) return st;
    const Geom g = make_geom(lat, n_rhs);
    const Geom g1 = make_geom(lat, 1);
    const void *half = clover_half(clover, g1, rep, clover_prec(prec), inverse != 0, parity);
    return clover_apply_half(ctx, g, rep, prec, half, in, out, (cudaStream_t)stream);
}

hr_status hr_dirac_apply_clover(hr_ctx *ctx, hr_lattice lat, hr_rep rep, hr_prec prec, const void *gauge,
                                const void *clover, const void *in, void *out, hr_stream stream)
{
    if (!ctx) return HR_ERR_INVALID_ARG;
    if (!valid_rep(rep) || !valid_prec(prec)) return set_error(ctx, HR_ERR_INVALID_ARG, "bad rep/prec");
    hr_status st = validate_lattice(ctx, lat, 1);
    if (st) return st;
    st = check_buffers(ctx, {gauge, clover, in, out});
    if (st) return st;
    if (in == out) return set_error(ctx, HR_ERR_INVALID_ARG, "in and out must not alias");
    const Geom g = make_geom(lat, 1);
    const size_t half = spinor_half_bytes(g, rep, prec);
    cudaStream_t s = (cudaStream_t)stream;
    // out_p = A_pp in_p - 1/2 H_{p,1-p} in_{1-p}: one hop per parity, A on the aux term
    for (int p = 0; p < 2; ++p) {
        HopLaunch L{};
        L.p = p;
        L.gauge = gauge;
        L.in = (const char *)in + (1 - p) * half;
        L.aux = (const char *)in + p * half;
        L.out = (char *)out + p * half;
        L.alpha = 1.0;
        L.beta = -0.5;
        L.clov = clover_half(clover, g, rep, clover_prec(prec), false, p);
        L.clov_mode = kClovAux;
        st = launch_hop(ctx, g, rep, prec, L, s);
        if (st) return st;
    }
    return HR_OK;
}

hr_status hr_dirac_eo_clover(hr_ctx *ctx, hr_lattice lat, hr_rep rep, hr_prec prec, hr_parity out_parity, hr_op op,
                             int n_rhs, const void *gauge, const void *clover, const void *in, void *out, void *work,
                             size_t work_bytes, hr_stream stream)
{
    if (!ctx) return HR_ERR_INVALID_ARG;
    if (!clover) return set_error(ctx, HR_ERR_INVALID_ARG, "null clover field");
    if (op == HR_OP_HOP) return hr_dirac_eo(ctx, lat, 0.0, rep, prec, out_parity, op, n_rhs, gauge, in, out, work,
                                             work_bytes, stream);
    if (!valid_rep(rep) || !valid_prec(prec)) return set_error(ctx, HR_ERR_INVALID_ARG, "bad rep/prec");
    hr_status st = validate_lattice(ctx, lat, n_rhs);
    if (st) return st;
    st = check_buffers(ctx, {gauge, clover, in, out}, {}, {work});
    if (st) return st;
    if (in == out) return set_error(ctx, HR_ERR_INVALID_ARG, "in and out must not alias");
    if (op != HR_OP_SCHUR && op != HR_OP_SCHUR_DAG && op != HR_OP_NORMAL)
        return set_error(ctx, HR_ERR_INVALID_ARG, "bad op %d", (int)op);
    if (out_parity != HR_EVEN) return set_error(ctx, HR_ERR_INVALID_ARG, "Schur operators act on even sites");
    const size_t need = hr_dirac_workspace_bytes(lat, rep, prec, op, n_rhs);
    if (!work || work_bytes < need)
        return set_error(ctx, HR_ERR_WORKSPACE, "workspace of %zu bytes needed, %zu given", need, work_bytes);
    const Geom g = make_geom(lat, n_rhs);
    const size_t half = spinor_half_bytes(g, rep, prec);
    void *wo = work;
    void *we = (op == HR_OP_NORMAL) ? (char *)work + half : nullptr;
    return apply_eo_op(ctx, g, 0.0, rep, prec, op, gauge, in, out, wo, we, kFinNone, nullptr, nullptr,
                       (cudaStream_t)stream, nullptr, clover);
}

} // extern "C"

// ---------------------------------------------------------------- HMC force of the clover term
//
// Fundamental links, SW form.  For a spin-colour insertion Lam(y),
//   f = Re sum_y tr[C(y) Lam(y)] = Re sum_y (i/2) sum_{mu<nu} tr_c[F_mn(y) K_mn(y)],
// and in the chiral blocks (C+ on spins 0, 1, C- on 2, 3, as in the build), with
// P_l^b = sum_{s,t} (s_l)_st Lam[(2b+t, .), (2b+s, .)] (colour 2x2),
//   K_0l = P_l^1 - P_l^0,  K_23 = -(P_1^0 + P_1^1),  K_13 = P_2^0 + P_2^1,  K_12 = -(P_3^0 + P_3^1).
// Only kappa_k = Re tr(s_k K) of a plane enters f (F_mn is (i/4) f.s with real f),
// so the field kept is double [6][3][V] (planes 01 02 03 12 13 23, lexicographic site).
// The link derivative of f: each link lies on two plaquettes of each of the
// three planes that contain its direction, and each plaquette enters the
// leaves of its four corners; hr_clover_leaf.cuh sums the four corner
// insertions around one staple per plaquette.
//
// Two flavours of clover fermions through the even-odd pseudofermion (Mhat =
// A_ee - H_eo A_oo^-1 H_oe / 4): with X = (Mhat^+ Mhat)^-1 eta, Y = Mhat X,
// Z = A_oo^-1 H_oe X, W = A_oo^-1 H_eo^+ Y,
//   dS_pf = 1/2 dRe<a, H b> (a = (Y, W), b = (X, Z)) + c_sw df[Lam],
//   Lam = -2 X Y^+ (even), -1/2 Z W^+ (odd),
// and S_det = -2 sum_{odd} log det A adds Lam_det = -2 A^-1 (odd).

namespace {

// (s_l)_st, l = 0, 1, 2 for s_1, s_2, s_3
__device__ __forceinline__ zc pauli(int l, int s, int t)
{
    if (l == 0) return {s != t ? 1.0 : 0.0, 0.0};
    if (l == 1) return s == t ? zc{0.0, 0.0} : (s == 0 ? zc{0.0, -1.0} : zc{0.0, 1.0});
    return {s != t ? 0.0 : (s == 0 ? 1.0 : -1.0), 0.0};
}

// P[b][l][d][c] += coef * lam((2b+t, d), (2b+s, c)) summed with (s_l)_st
template <class Lam> __device__ void add_blocks(zc (&P)[2][3][2][2], double coef, Lam lam)
{
    for (int b = 0; b < 2; ++b)
        for (int l = 0; l < 3; ++l)
            for (int d = 0; d < 2; ++d)
                for (int c = 0; c < 2; ++c) {
                    zc acc = {0.0, 0.0};
                    for (int s = 0; s < 2; ++s)
                        for (int t = 0; t < 2; ++t) {
                            const zc sg = pauli(l, s, t);
                            if (sg.re == 0.0 && sg.im == 0.0) continue;
                            acc = zadd(acc, zmul(sg, lam(2 * b + t, d, 2 * b + s, c)));
                        }
                    P[b][l][d][c] = zadd(P[b][l][d][c], zscale(coef, acc));
                }
}

// kappa_k = Re tr(s_k K) of the six planes, double [6][3][V]; with Pi^b_lk =
// Re tr_c(s_k P_l^b): kappa_0l = Pi^1_l - Pi^0_l, kappa_23 = -(Pi^0_1 + Pi^1_1),
// kappa_13 = Pi^0_2 + Pi^1_2, kappa_12 = -(Pi^0_3 + Pi^1_3)
__device__ __forceinline__ void store_kappa(double *K, long long V, long long x, int l, int k, double lower, double upper)
{
    K[((long long)l * 3 + k) * V + x] = upper - lower;
    const int pl = l == 0 ? 5 : l == 1 ? 4 : 3;
    K[((long long)pl * 3 + k) * V + x] = l == 1 ? lower + upper : -(lower + upper);
}
__device__ void store_k(double *K, long long V, long long x, const zc (&P)[2][3][2][2])
{
    for (int l = 0; l < 3; ++l) {
        double pi[2][3];
        for (int b = 0; b < 2; ++b) {
            pi[b][0] = P[b][l][0][1].re + P[b][l][1][0].re;
            pi[b][1] = P[b][l][1][0].im - P[b][l][0][1].im;
            pi[b][2] = P[b][l][0][0].re - P[b][l][1][1].re;
        }
        for (int k = 0; k < 3; ++k) store_kappa(K, V, x, l, k, pi[0][k], pi[1][k]);
    }
}

// kappa from a canonical insertion Lam: complex [V][8][8], index spin * 2 + colour
__global__ void k_clover_k_from_lam(long long V, const double *lam, double *K)
{
    const long long x = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= V) return;
    const double *L = lam + x * 128;
    zc P[2][3][2][2] = {};
    add_blocks(P, 1.0, [&](int t, int d, int s, int c) {
        const int r = t * 2 + d, q = s * 2 + c;
        return zc{L[(r * 8 + q) * 2], L[(r * 8 + q) * 2 + 1]};
    });
    store_k(K, V, x, P);
}

struct KFieldArgs {
    Geom g;
    const void *X, *Y; // even halves (packed FP64)
    const void *Z, *W; // odd halves
    const void *ainv;  // A^-1 odd half-field (packed FP64 clover), or nullptr: no det term
    const void *afwd[2]; // exponential form: A on even / odd sites
    int exp_kind;        // 1: A = a exp(c_sw C / a), the insertion goes through exp_insertion
    double a;            // 4 + m0
    double *K;
};

// Exponential form: Lam' = int_0^1 exp((1-s) X) Lam exp(s X) ds per chiral block,
// from the eigen-decomposition of the block of A = a exp(X) (eigenvalues mu =
// a e^l): (V^+ Lam' V)_ij = (V^+ Lam V)_ij (e^l_i - e^l_j) / (l_i - l_j).
__device__ void exp_insertion_block(const zd (&Ab)[4][4], double a, zd (&L)[4][4])
{
    zd M[4][4], V[4][4];
    double mu[4], l[4];
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) M[i][j] = Ab[i][j];
    jacobi_eigh<4>(M, V, mu);
    for (int i = 0; i < 4; ++i) l[i] = log(mu[i] / a);
    zd T[4][4], R[4][4];
    for (int i = 0; i < 4; ++i) // T = V^+ L V
        for (int j = 0; j < 4; ++j) {
            zc acc = {0.0, 0.0};
            for (int k = 0; k < 4; ++k)
                for (int m = 0; m < 4; ++m)
                    acc = zadd(acc, zmul(zmul(zconj(zc{V[k][i].re, V[k][i].im}), zc{L[k][m].re, L[k][m].im}),
                                         zc{V[m][j].re, V[m][j].im}));
            const double d = l[i] - l[j];
            const double phi = fabs(d) > 1e-8 ? (exp(l[i]) - exp(l[j])) / d : exp(0.5 * (l[i] + l[j]));
            T[i][j] = {phi * acc.re, phi * acc.im};
        }
    for (int i = 0; i < 4; ++i) // R = V T V^+
        for (int j = 0; j < 4; ++j) {
            zc acc = {0.0, 0.0};
            for (int k = 0; k < 4; ++k)
                for (int m = 0; m < 4; ++m)
                    acc = zadd(acc, zmul(zmul(zc{V[i][k].re, V[i][k].im}, zc{T[k][m].re, T[k][m].im}),
                                         zconj(zc{V[j][m].re, V[j][m].im})));
            R[i][j] = {acc.re, acc.im};
        }
    for (int i = 0; i < 4; ++i)
        for (int j = 0; j < 4; ++j) L[i][j] = R[i][j];
}

// the two 4 x 4 blocks of a packed FP64 clover half-field at site i
__device__ void read_blocks(const void *half, int i, zd (&M)[2][4][4])
{
    CloverReader<2, kF64, dd> rd(half, i); // double-float reals, converted exactly
    int q = 0;
    for (int b = 0; b < 2; ++b) {
        for (int k = 0; k < 4; ++k) M[b][k][k] = {dd_to_double(rd.get(q++)), 0.0};
        for (int r = 0; r < 4; ++r)
            for (int c = r + 1; c < 4; ++c) {
                const double re = dd_to_double(rd.get(q++)), im = dd_to_double(rd.get(q++));
                M[b][r][c] = {re, im};
                M[b][c][r] = {re, -im};
            }
    }
}

// kappa of the two-flavour clover pseudofermion (and det A_oo) insertion at one site, native FP64
__device__ void kappa_site(const KFieldArgs &A, long long x, int p)
{
    const Geom &g = A.g;
    const long long V = 2LL * g.vh;
    const int i = (int)(x >> 1);
    zc P[2][3][2][2] = {};
    cpx<double> u[4][2], v[4][2];
    load_spinor<2, kF64>(p == 0 ? A.X : A.Z, g.nblk_s, i, u);
    load_spinor<2, kF64>(p == 0 ? A.Y : A.W, g.nblk_s, i, v);
    // Lam = coef u v^+ : Lam[(t, d), (s, c)] = coef u[t][d] conj(v[s][c])
    const double coef = p == 0 ? -2.0 : -0.5;
    if (A.exp_kind) {
        zd Ab[2][4][4], Lb[2][4][4];
        read_blocks(A.afwd[p], i, Ab);
        for (int b = 0; b < 2; ++b) {
            for (int k = 0; k < 4; ++k)
                for (int m = 0; m < 4; ++m) {
                    const zc z = zmul(zc{u[2 * b + k / 2][k % 2].re, u[2 * b + k / 2][k % 2].im},
                                      zconj(zc{v[2 * b + m / 2][m % 2].re, v[2 * b + m / 2][m % 2].im}));
                    Lb[b][k][m] = {coef * z.re, coef * z.im};
                }
            exp_insertion_block(Ab[b], A.a, Lb[b]);
        }
        add_blocks(P, 1.0, [&](int t, int d, int s, int c) {
            const zd z = Lb[t >> 1][(t & 1) * 2 + d][(s & 1) * 2 + c];
            return zc{z.re, z.im};
        });
        store_k(A.K, V, x, P);
        return;
    }
    add_blocks(P, coef, [&](int t, int d, int s, int c) {
        return zmul(zc{u[t][d].re, u[t][d].im}, zconj(zc{v[s][c].re, v[s][c].im}));
    });
    if (p == 1 && A.ainv) {
        // Lam_det = -2 A^-1: block b (spins 2b, 2b+1) as n = 4 reals per diagonal, then the upper triangle
        // (double-float reals, converted exactly)
        CloverReader<2, kF64, dd> rd(A.ainv, i);
        zc M[2][4][4];
        int q = 0;
        for (int b = 0; b < 2; ++b) {
            for (int k = 0; k < 4; ++k) M[b][k][k] = {dd_to_double(rd.get(q++)), 0.0};
            for (int a = 0; a < 4; ++a)
                for (int c = a + 1; c < 4; ++c) {
                    const double re = dd_to_double(rd.get(q++)), im = dd_to_double(rd.get(q++));
                    M[b][a][c] = {re, im};
                    M[b][c][a] = {re, -im};
                }
        }
        add_blocks(P, -2.0, [&](int t, int d, int s, int c) {
            const int b = t >> 1; // same block as s (diagonal blocks only are read)
            return M[b][(t & 1) * 2 + d][(s & 1) * 2 + c];
        });
    }
    store_k(A.K, V, x, P);
}
__device__ __forceinline__ int site_parity(const LexSite &x) { return (x.x0 + x.x1 + x.x2 + x.x3) & 1; }

// the exponential form: the insertion goes through the eigenbasis of A
__global__ void k_clover_kappa_exp(KFieldArgs A)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < 2 * A.g.vh) kappa_site(A, t, site_parity(lex_site(A.g, t)));
}

__device__ __noinline__ void kappa_site_native(const KFieldArgs &A, long long x, int p) { kappa_site(A, x, p); }

// Re v^+ (s_l (x) s_k) u of one chiral block, u and v [4 spin + 2 colour + (re, im)]
__device__ __forceinline__ long long sigma_sigma(const fx *u, const fx *v, int l, int k)
{
    fxa s = {0, 0};
#pragma unroll
    for (int sp = 0; sp < 2; ++sp)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            // row (sp, c) of s_l (x) s_k has one entry, i^n at column (sc, cc)
            const int sc = l < 2 ? 1 - sp : sp, cc = k < 2 ? 1 - c : c;
            const int n = ((l == 1 ? (sp ? 1 : 3) : l == 2 && sp ? 2 : 0) + (k == 1 ? (c ? 1 : 3) : k == 2 && c ? 2 : 0)) & 3;
            const fx vr = v[4 * sp + 2 * c], vi = v[4 * sp + 2 * c + 1];
            const fx ur = u[4 * sc + 2 * cc], ui = u[4 * sc + 2 * cc + 1];
            // Re(conj(v) i^n u)
            if (n == 0) { fx_mac(s, vr, ur); fx_mac(s, vi, ui); }
            else if (n == 1) { fx_mac(s, fx_neg(vr), ui); fx_mac(s, vi, ur); }
            else if (n == 2) { fx_mac(s, fx_neg(vr), ur); fx_mac(s, fx_neg(vi), ui); }
            else { fx_mac(s, vr, ui); fx_mac(s, fx_neg(vi), ur); }
        }
    return fx_round(s);
}

// Clover form, one thread per lexicographic site, in fixed point (hr_fix.cuh):
// Pi^b_lk = coef Re v^+ (s_l (x) s_k) u needs the real parts of 9 x 8 products
// a block instead of the complex outer product u v^+; on odd sites the
// determinant adds -8 (A^-1)_lk, the coefficient of s_l (x) s_k in A^-1.
// One unit for a site's spinors is enough: a link's force sums the planes of four
// corners of both parities and the hops' term of the same fields, whose native sums
// round at the largest of them too, and the fields and A^-1 are pairs of 2^-49.
__global__ void __launch_bounds__(128, 3) k_clover_kappa(KFieldArgs A)
{
    const Geom &g = A.g;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 2 * g.vh) return;
    const long long V = 2LL * g.vh;
    const int p = site_parity(lex_site(g, t)), i = t >> 1;
    fx u[16], v[16];
    int eu, ev;
    bool ok = load_fx(p == 0 ? A.X : A.Z, i, u, eu);
    ok = load_fx(p == 0 ? A.Y : A.W, i, v, ev) && ok;
    if (!ok) {
        kappa_site_native(A, t, p);
        return;
    }
    const double f = (p == 0 ? -2.0 : -0.5) * fx_pow2(eu + ev - 2 * kFxPairBias - 56);
    const bool det = p == 1 && A.ainv;
    double pi[2][9];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
#pragma unroll
        for (int e = 0; e < 9; ++e) pi[b][e] = f * (double)sigma_sigma(u + 8 * b, v + 8 * b, e / 3, e % 3);
        if (det) {
            // block reals 0-3: diagonal; 4-15: (0,1) (0,2) (0,3) (1,2) (1,3) (2,3) as (re, im)
            const float4 *q = (const float4 *)A.ainv + ((size_t)(i >> 5) * 16 + 8 * b) * 32 + (i & 31);
            float4 w[8];
            unsigned m = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                w[k] = __ldg(q + k * 32);
                m = max(m, max(__float_as_uint(w[k].x) & 0x7fffffffu, __float_as_uint(w[k].z) & 0x7fffffffu));
            }
            const int E = min(max((int)(m >> 23), kFxMinExp), 254);
            const float sc = fx_pair_scale(E);
            long long R[16];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                R[2 * k] = fx_units64(fx_from_pair(w[k].x, w[k].y, sc));
                R[2 * k + 1] = fx_units64(fx_from_pair(w[k].z, w[k].w, sc));
            }
            // 4 N_lk
            const long long n[9] = {2 * (R[10] + R[8]), 2 * (R[11] - R[9]), 2 * (R[6] - R[12]),
                                    -2 * (R[9] + R[11]), 2 * (R[10] - R[8]), 2 * (R[13] - R[7]),
                                    2 * (R[4] - R[14]), 2 * (R[15] - R[5]), (R[0] - R[1]) - (R[2] - R[3])};
            const double h = -2.0 * fx_pow2(E - kFxPairBias - 56);
#pragma unroll
            for (int e = 0; e < 9; ++e) pi[b][e] += h * (double)n[e];
        }
    }
#pragma unroll
    for (int e = 0; e < 9; ++e) store_kappa(A.K, V, t, e / 3, e % 3, pi[0][e], pi[1][e]);
}

// one link in native FP64: links off unit length, NaN or Inf
__device__ __noinline__ void leaf_force_native(const Geom &g, const double *can, const double *K, double scale, int rho,
                                               int t, double *o)
{
    LeafLattice L;
    for (int k = 0; k < 4; ++k) L.d[k] = g.d[k];
    const LexSite s = lex_site(g, t);
    const int x[4] = {s.x0, s.x1, s.x2, s.x3};
    double out[3];
    leaf_force_link(L, can, KappaField{K, 2LL * g.vh}, rho, x, out);
    for (int a = 0; a < 3; ++a) o[a] += scale * out[a];
}

// F[rho][z][a] += scale * d/dw_a Re sum_y tr[C Lam], one thread per link (rho =
// blockIdx.y, z): the two plaquettes of each of the three planes that hold rho,
// each as the loop V e1 e2 e3 from z (V = U_rho(z)) with the four corner
// vectors k0 .. k3 (pure quaternions) inserted around one staple S = e1 e2 e3,
//   F = -/+ vec(V B) / 16,  B = k1 S + e1 (k2 e2 + e2 k3) e3 + S k0
// (- where the loop runs mu-first in the plane's orientation), V taken out of
// the sum of the six B.  Fixed point (hr_fix.cuh): about 110 products a
// plaquette, where the 2 x 2 complex matrices of hr_clover_leaf.cuh take 700.
// The kappa of a plaquette are read in units of their largest component, and
// the running sum of the B follows the largest unit met so far (native FP64 rounds
// at that size as well: B is the sum of the rotated kappa).  20 x 14 x 18 x 22:
// 4.99 ms in native FP64, 0.252 ms here (0.286 with conversions of 20 instead of 13
// instructions a number; 128 registers: 0.298); the whole clover force (hops, link
// derivatives, kappa, this) 5.77 -> 0.42 ms, error against 64 bits unchanged
// (7.8e-15, the hops').
template <bool VEC>
__global__ void __launch_bounds__(128, 3) k_clover_leaf_force(Geom g, const double *__restrict__ can,
                                                              const double *__restrict__ K, double scale,
                                                              double *__restrict__ F)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x, rho = blockIdx.y;
    const int V = 2 * g.vh;
    if (t >= V) return;
    const LexSite x = lex_site(g, t);
    int ur, unused;
    lex_steps(g, x, rho, ur, unused);
    bool ok = true;
    const size_t br = (size_t)rho * V + t;
    long long B[4] = {0, 0, 0, 0};
    int eB = -4096; // B in units of 2^(eB - 56)
#pragma unroll 1
    for (int k = 2; k < 8; ++k) {
        const int sig = (rho + (k >> 1)) & 3;
        const bool down = k & 1;
        int us, ds;
        lex_steps(g, x, sig, us, ds);
        const int off = down ? ds : us, s0 = down ? ds : 0;
        const size_t bs = (size_t)sig * V + t;
        fxq e1 = load_fxq<VEC>(can, bs + ur + s0, ok), e3 = load_fxq<VEC>(can, bs + s0, ok);
        const fxq e2 = fxq_conj(load_fxq<VEC>(can, br + off, ok));
        if (down) e1 = fxq_conj(e1);
        else e3 = fxq_conj(e3);
        const int lo = min(rho, sig), hi = max(rho, sig);
        const int pl = lo == 0 ? hi - 1 : lo == 1 ? hi + 1 : 5; // 01 02 03 12 13 23
        const double *kp = K + (size_t)pl * 3 * V + t;
        double kd[4][3];
        unsigned m = 0;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double *q = kp + (size_t)a * V;
            kd[0][a] = __ldg(q);
            kd[1][a] = __ldg(q + ur);
            kd[2][a] = __ldg(q + ur + off);
            kd[3][a] = __ldg(q + off);
#pragma unroll
            for (int c = 0; c < 4; ++c) m = max(m, fx_abs_high(kd[c][a]));
        }
        const int E = (int)(m >> 20);
        ok = ok && E < 2047;
        fx kq[4][3];
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int a = 0; a < 3; ++a) kq[c][a] = fx_from_double(kd[c][a], E);
        const fxq S = fxq_mul(e1, fxq_mul(e2, e3));
        fxa ya[4] = {}, ta[4] = {};
        fxq_mac_pure_l(ya, kq[2], e2);
        fxq_mac_pure_r(ya, e2, kq[3]);
        fxq_mac(ta, fxq_mul(e1, fxq_of(ya)), e3);
        fxq_mac_pure_l(ta, kq[1], S);
        fxq_mac_pure_r(ta, S, kq[0]);
        if (E == 0) continue; // all zero (or subnormal)
        const int e = E - 1022, dn = min(max(eB - e, 0), 63), db = min(max(e - eB, 0), 63);
        const bool minus = (rho < sig) != down;
        eB = max(eB, e);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const long long v = fx_round(ta[c]) >> dn;
            B[c] = (B[c] >> db) + (minus ? -v : v);
        }
    }
    const fxq U = load_fxq<VEC>(can, br, ok);
    double *o = F + br * 3;
    if (!ok) {
        leaf_force_native(g, can, K, scale, rho, t, o);
        return;
    }
    if (eB == -4096) return;
    // |B| < 42 units: down to digits below 2^30
    unsigned long long used = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) used |= (unsigned long long)(B[c] ^ (B[c] >> 63));
    const int r = max(0, 6 - fx_clz(used | 1u));
    fxq Bq;
#pragma unroll
    for (int c = 0; c < 4; ++c) Bq.c[c] = fx_split(B[c] >> r);
    fxa w[3] = {};
    fxq_mac_vec(w, U, Bq);
    const int ex = eB + r - 60; // 2^-56 and the 1/16
    if (ex > -1000 && ex < 900) {
        const double f = scale * fx_pow2(ex);
#pragma unroll
        for (int a = 0; a < 3; ++a) o[a] += f * (double)fx_round(w[a]);
    } else {
        leaf_force_native(g, can, K, scale, rho, t, o);
    }
}

// block sums of sum_{odd sites} log det A (both blocks, Cholesky), one partial per block
template <int NC> __global__ void __launch_bounds__(128) k_clover_logdet(Geom g, const void *half, double *partial,
                                                                         unsigned *bad)
{
    constexpr int N = 2 * NC;
    double acc = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.vh; i += gridDim.x * blockDim.x) {
        CloverReader<NC, kF64, dd> rd(half, i); // double-float reals, converted exactly
        int q = 0;
        for (int b = 0; b < 2; ++b) {
            zc M[N][N];
            for (int k = 0; k < N; ++k) M[k][k] = {dd_to_double(rd.get(q++)), 0.0};
            for (int a = 0; a < N; ++a)
                for (int c = a + 1; c < N; ++c) {
                    const double re = dd_to_double(rd.get(q++)), im = dd_to_double(rd.get(q++));
                    M[a][c] = {re, im};
                    M[c][a] = {re, -im};
                }
            // Cholesky M = L L^+ in place (lower triangle); log det = 2 sum log L_kk
            for (int k = 0; k < N; ++k) {
                double dkk = M[k][k].re;
                for (int j = 0; j < k; ++j) dkk -= M[k][j].re * M[k][j].re + M[k][j].im * M[k][j].im;
                if (!(dkk > 0.0)) {
                    atomicExch(bad, 1u);
                    dkk = 1.0;
                }
                const double lkk = sqrt(dkk);
                acc += 2.0 * log(lkk);
                for (int a = k + 1; a < N; ++a) {
                    zc s = M[a][k];
                    for (int j = 0; j < k; ++j) s = zsub(s, zmul(M[a][j], zconj(M[k][j])));
                    M[a][k] = zscale(1.0 / lkk, s);
                }
            }
        }
    }
    __shared__ double red[128];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}

constexpr int kLogdetBlocks = 256;

// the insertion field's share of a caller's workspace: 48 doubles a site as the
// entry points have always asked for, of which the field fills 18
size_t k_field_bytes(const Geom &g) { return ((size_t)2 * g.vh * 48 * sizeof(double) + 255) & ~(size_t)255; }

hr_status leaf_force(hr_ctx *ctx, const Geom &g, const double *can, const double *K, double scale, double *F,
                     cudaStream_t s)
{
    const dim3 grid((unsigned)((2LL * g.vh + 127) / 128), 4);
    if (((uintptr_t)can & 15u) == 0) k_clover_leaf_force<true><<<grid, 128, 0, s>>>(g, can, K, scale, F);
    else k_clover_leaf_force<false><<<grid, 128, 0, s>>>(g, can, K, scale, F);
    return check_launch(ctx, "clover force");
}

} // namespace

extern "C" {

size_t hr_clover_force_workspace_bytes(hr_lattice lat)
{
    if (hr_gauge_packed_bytes(lat, HR_FUND, HR_F64) == 0) return 0;
    const Geom g = make_geom(lat, 1);
    const size_t half = spinor_half_bytes(g, HR_FUND, kF64);
    return k_field_bytes(g) + 5 * half;
}

hr_status hr_clover_insertion_force(hr_ctx *ctx, hr_lattice lat, double c_sw, const double *gauge, const double *lam,
                                    double coeff, double *force, void *work, size_t work_bytes, hr_stream stream)
{
    if (!ctx) return HR_ERR_INVALID_ARG;
    hr_status st = validate_lattice(ctx, lat, 1);
    if (st) return st;
    st = check_buffers(ctx, {work}, {gauge, lam, force});
    if (st) return st;
    if (!std::isfinite(c_sw) || !std::isfinite(coeff)) return set_error(ctx, HR_ERR_INVALID_ARG, "c_sw, coeff finite");
    const Geom g = make_geom(lat, 1);
    if (work_bytes < k_field_bytes(g))
        return set_error(ctx, HR_ERR_WORKSPACE, "workspace of %zu bytes needed, %zu given", k_field_bytes(g), work_bytes);
    cudaStream_t s = (cudaStream_t)stream;
    const long long V = 2LL * g.vh;
    k_clover_k_from_lam<<<(unsigned)((V + 127) / 128), 128, 0, s>>>(V, lam, (double *)work);
    st = check_launch(ctx, "clover insertion");
    if (!st) st = leaf_force(ctx, g, gauge, (const double *)work, coeff * c_sw, force, s);
    return st;
}

hr_status hr_clover_fermion_force(hr_ctx *ctx, hr_lattice lat, hr_clover_kind kind, double m0, double c_sw,
                                  const double *gauge, const void *gauge_packed, const void *clover, const void *X,
                                  const void *Y, int with_det, double coeff, double *force, void *work,
                                  size_t work_bytes, hr_stream stream)
{
    if (ctx && kind != HR_CLOVER_SW && kind != HR_CLOVER_EXP)
        return set_error(ctx, HR_ERR_INVALID_ARG, "bad clover kind");
    if (!ctx) return HR_ERR_INVALID_ARG;
    hr_status st = validate_lattice(ctx, lat, 1);
    if (st) return st;
    st = check_buffers(ctx, {gauge_packed, clover, X, work}, {gauge, force}, {Y});
    if (st) return st;
    if (!(4.0 + m0 != 0.0) || !std::isfinite(c_sw) || !std::isfinite(coeff))
        return set_error(ctx, HR_ERR_INVALID_ARG, "4 + m0 nonzero, c_sw and coeff finite");
    const size_t need = hr_clover_force_workspace_bytes(lat);
    if (work_bytes < need) return set_error(ctx, HR_ERR_WORKSPACE, "workspace of %zu bytes needed, %zu given", need, work_bytes);
    const Geom g = make_geom(lat, 1);
    cudaStream_t s = (cudaStream_t)stream;
    const size_t half = spinor_half_bytes(g, HR_FUND, kF64);
    char *w = (char *)work;
    double *K = (double *)w;
    char *a = w + k_field_bytes(g); // full field (Y | W)
    char *z = a + 2 * half;         // odd half field Z
    const void *ainv_odd = clover_half(clover, g, HR_FUND, kF64, true, 1);
    // dst = A_oo^-1 [g5] H_oe [g5] src (A commutes with g5)
    auto hop_oe = [&](const void *src, void *dst, int g5) {
        HopLaunch L{};
        L.p = 1;
        L.gauge = gauge_packed;
        L.in = src;
        L.out = dst;
        L.beta = 1.0;
        L.g5_in = L.g5_out = g5;
        L.clov = ainv_odd;
        L.clov_mode = kClovOut;
        return launch_hop(ctx, g, HR_FUND, kF64, L, s);
    };
    // Z = A_oo^-1 H_oe X, and Y = Mhat X, whose first hop is Z, unless Y is given
    const void *y = Y ? Y : a;
    st = Y ? hop_oe(X, z, 0)
           : apply_eo_op(ctx, g, m0, HR_FUND, kF64, HR_OP_SCHUR, gauge_packed, X, a, z, nullptr, kFinNone, nullptr,
                         nullptr, s, nullptr, clover);
    // W = A_oo^-1 g5 H_oe g5 Y
    if (!st) st = hop_oe(y, a + half, 1);
    // the hops: 1/2 dRe<(Y, W), H (X, Z)>
    if (!st) st = link_deriv(ctx, lat, gauge_packed, y, a + half, X, z, 0.5 * coeff, force, 0, s);
    if (st) return st;
    // the site term: c_sw df[Lam]
    KFieldArgs A;
    A.g = g;
    A.X = X;
    A.Y = y;
    A.Z = z;
    A.W = a + half;
    // the exponential form's det A_oo is a constant (C is traceless): no det force
    A.ainv = (with_det && kind == HR_CLOVER_SW) ? ainv_odd : nullptr;
    A.afwd[0] = clover_half(clover, g, HR_FUND, kF64, false, 0);
    A.afwd[1] = clover_half(clover, g, HR_FUND, kF64, false, 1);
    A.exp_kind = kind == HR_CLOVER_EXP;
    A.a = 4.0 + m0;
    A.K = K;
    const long long V = 2LL * g.vh;
    const unsigned kgrid = (unsigned)((V + 127) / 128);
    if (A.exp_kind) k_clover_kappa_exp<<<kgrid, 128, 0, s>>>(A);
    else k_clover_kappa<<<kgrid, 128, 0, s>>>(A);
    st = check_launch(ctx, "clover insertion");
    if (!st) st = leaf_force(ctx, g, gauge, K, coeff * c_sw, force, s);
    return st;
}

hr_status hr_clover_logdet(hr_ctx *ctx, hr_lattice lat, hr_rep rep, const void *clover, hr_parity parity,
                           double *logdet, hr_stream stream)
{
    if (!ctx) return HR_ERR_INVALID_ARG;
    if (!logdet) return set_error(ctx, HR_ERR_INVALID_ARG, "null result pointer");
    if (rep != HR_FUND && rep != HR_ADJ) return set_error(ctx, HR_ERR_INVALID_ARG, "HR_FUND or HR_ADJ");
    if (parity != HR_EVEN && parity != HR_ODD) return set_error(ctx, HR_ERR_INVALID_ARG, "bad parity");
    hr_status st = validate_lattice(ctx, lat, 1);
    if (st) return st;
    st = check_buffers(ctx, {clover});
    if (st) return st;
    const Geom g = make_geom(lat, 1);
    cudaStream_t s = (cudaStream_t)stream;
    const void *half = clover_half(clover, g, rep, kF64, false, parity);
    unsigned *bad = ctx->d_counters + C_STATUS;
    cudaError_t e = cudaMemsetAsync(bad, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return set_error(ctx, HR_ERR_CUDA, "status reset: %s", cudaGetErrorString(e));
    if (rep == HR_FUND) k_clover_logdet<2><<<kLogdetBlocks, 128, 0, s>>>(g, half, ctx->d_partials, bad);
    else k_clover_logdet<3><<<kLogdetBlocks, 128, 0, s>>>(g, half, ctx->d_partials, bad);
    st = check_launch(ctx, "clover log det");
    if (st) return st;
    double h[kLogdetBlocks];
    unsigned hb = 0;
    e = cudaMemcpyAsync(h, ctx->d_partials, sizeof h, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hb, bad, sizeof hb, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return set_error(ctx, HR_ERR_CUDA, "log det readback: %s", cudaGetErrorString(e));
    if (hb) return set_error(ctx, HR_ERR_NUMERIC, "a clover block is not positive definite");
    double acc = 0.0;
    for (int k = 0; k < kLogdetBlocks; ++k) acc += h[k];
    *logdet = acc;
    return HR_OK;
}

} // extern "C"
