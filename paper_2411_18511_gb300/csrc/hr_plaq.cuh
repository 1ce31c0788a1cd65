// hr_plaq.cuh -- the vector parts of the plaquettes, vec P_mn(x) with
// P_mn(x) = U_m(x) U_n(x+m) U_m(x+n)^+ U_n(x)^+, in two-digit fixed point (hr_fix.cuh),
// and their transport by one link: shared by the gauge force (hr_hmc.cu) and the
// clover build (hr_clover.cu), which need each at several sites.
#pragma once

#include "hr_fix_dev.cuh"
#include "hr_host.h"

namespace hr {

static_assert(kPlaqSiteBytes == 6 * (sizeof(int4) + sizeof(int2)), "six vectors a site");

// A vector in the scratch is three digit pairs (int4, int2) in units of 1.  Digits hold
// an absolute 2^-56 and the products some 2^-56 more (1.3e-17 in root mean square),
// native FP64 rounds at 2^-53 of the links' vector parts (1.3e-16 of them): the
// same where the largest component of the four links is 1/8.  Links below that (near the
// identity: cold starts, smooth fields) give the plaquette in native FP64, and the
// scratch holds its three doubles, marked: the top two bits of a leading digit are equal
// (|h| < 2^30), those of a double's high word are made to differ (it is below 2, so
// the second is free).
constexpr unsigned kPlaqWeak = (1023u - 3u) << 20; // high word of 1/8
constexpr int kPlaqBad = 0x7fffffff;               // links outside the fixed-point range (marked too)
__device__ __forceinline__ bool plaq_marked(int first) { return (first ^ (first << 1)) < 0; }

struct PlaqVec {
    double v[3];
};
__device__ __forceinline__ void store_marked(const PlaqVec &P, int4 &a, int2 &b)
{
    const int h = __double2hiint(P.v[0]);
    a = make_int4((h & (int)0xbfffffff) | (int)(~(unsigned)h >> 1 & 0x40000000u), __double2loint(P.v[0]),
                  __double2hiint(P.v[1]), __double2loint(P.v[1]));
    b = make_int2(__double2hiint(P.v[2]), __double2loint(P.v[2]));
}
// the vector of either kind as doubles (kPlaqBad excepted)
__device__ __forceinline__ PlaqVec plaq_doubles(int4 a, int2 b)
{
    if (plaq_marked(a.x))
        return {{__hiloint2double(a.x & (int)0xbfffffff, a.y), __hiloint2double(a.z, a.w), __hiloint2double(b.x, b.y)}};
    return {{fx_to_double(fx_units64({a.x, a.y})), fx_to_double(fx_units64({a.z, a.w})), fx_to_double(fx_units64({b.x, b.y}))}};
}

// vec of U_a U_b (U_c U_d)^+ in native FP64
static __device__ __noinline__ PlaqVec plaq_vec_native(const double *q, size_t a, size_t b, size_t c, size_t d)
{
    auto mul = [&](size_t i, size_t j, double (&r)[4]) {
        const double *x = q + 4 * i, *y = q + 4 * j;
        r[0] = x[0] * y[0] - (x[1] * y[1] + x[2] * y[2] + x[3] * y[3]);
        r[1] = x[0] * y[1] + y[0] * x[1] - (x[2] * y[3] - x[3] * y[2]);
        r[2] = x[0] * y[2] + y[0] * x[2] - (x[3] * y[1] - x[1] * y[3]);
        r[3] = x[0] * y[3] + y[0] * x[3] - (x[1] * y[2] - x[2] * y[1]);
    };
    double A[4], B[4];
    mul(a, b, A);
    mul(c, d, B);
    return {{B[0] * A[1] - A[0] * B[1] + (A[2] * B[3] - A[3] * B[2]), B[0] * A[2] - A[0] * B[2] + (A[3] * B[1] - A[1] * B[3]),
             B[0] * A[3] - A[0] * B[3] + (A[1] * B[2] - A[2] * B[1])}};
}

// plane index of mu < nu: (01) (02) (03) (12) (13) (23)
__device__ __forceinline__ int plane_of(int mu, int nu)
{
    const int a = min(mu, nu), b = max(mu, nu);
    return a == 0 ? b - 1 : a + b;
}

// Vec P of the n sites from slice `first` on.  PER = 6: one thread per site, its own
// four links converted once and kept in shared memory (a conversion is some 90
// instructions, 24 of them a site were half of the kernel); 1: one per plane (blockIdx.y).
template <bool VEC, int PER>
__global__ void __launch_bounds__(128) k_plaq_vec(Geom g, const double *__restrict__ q, int first, int n,
                                                  int4 *__restrict__ pa, int2 *__restrict__ pb)
{
    constexpr int OWN = PER == 6 ? 8 : 1;
    __shared__ int4 own[OWN][128]; // this thread's slots: no other thread reads them
    __shared__ unsigned own_top[PER == 6 ? 4 : 1][128];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int V = 2 * g.vh, slice = g.d[1] * g.d[2] * g.d[3];
    int t = first * slice + i;
    if (t < 0) t += V;
    const LexSite x = lex_site(g, t);
    bool ok_own = true;
    if constexpr (PER == 6) {
#pragma unroll 1
        for (int mu = 0; mu < 4; ++mu) {
            unsigned top = 0;
            const fxq u = load_fxq<VEC>(q, (size_t)mu * V + t, ok_own, top);
            own_top[mu][threadIdx.x] = top;
            own[2 * mu][threadIdx.x] = make_int4(u.c[0].h, u.c[0].l, u.c[1].h, u.c[1].l);
            own[2 * mu + 1][threadIdx.x] = make_int4(u.c[2].h, u.c[2].l, u.c[3].h, u.c[3].l);
        }
    }
    auto own_link = [&](int mu, bool &ok, unsigned &top) -> fxq {
        if constexpr (PER == 6) {
            top = max(top, own_top[mu][threadIdx.x]);
            const int4 a = own[2 * mu][threadIdx.x], b = own[2 * mu + 1][threadIdx.x];
            return {{{a.x, a.y}, {a.z, a.w}, {b.x, b.y}, {b.z, b.w}}};
        } else {
            return load_fxq<VEC>(q, (size_t)mu * V + t, ok, top);
        }
    };
    const int p0 = PER == 6 ? 0 : blockIdx.y;
#pragma unroll 1
    for (int p = p0; p < p0 + PER; ++p) {
        const int mu = p < 3 ? 0 : p < 5 ? 1 : 2, nu = p < 3 ? p + 1 : p < 5 ? p - 1 : 3;
        int up_mu, up_nu, unused;
        lex_steps(g, x, mu, up_mu, unused);
        lex_steps(g, x, nu, up_nu, unused);
        bool ok = ok_own;
        unsigned top = 0;
        const size_t um = (size_t)mu * V + t, un = (size_t)nu * V + t;
        const fxq A = fxq_mul(own_link(mu, ok, top), load_fxq<VEC>(q, un + up_mu, ok, top));
        const fxq B = fxq_conj(fxq_mul(own_link(nu, ok, top), load_fxq<VEC>(q, um + up_nu, ok, top)));
        fxa w[3] = {};
        fxq_mac_vec(w, A, B);
        const fx v0 = fx_of(w[0]), v1 = fx_of(w[1]), v2 = fx_of(w[2]);
        int4 a = make_int4(ok ? v0.h : kPlaqBad, v0.l, v1.h, v1.l);
        int2 b = make_int2(v2.h, v2.l);
        if (ok && top < kPlaqWeak) store_marked(plaq_vec_native(q, um, un + up_mu, un, um + up_nu), a, b);
        pa[(size_t)p * n + i] = a;
        pb[(size_t)p * n + i] = b;
    }
}

// Up to this many sites k_plaq_vec runs one thread per plane, six times as many in
// flight: 16^4 15.7 us against 18.1 with one thread per site.
constexpr int kPlaqVecSplit = 1 << 17;
template <bool VEC>
inline void launch_plaq_vec(const Geom &g, const double *q, int first, int n, int4 *pa, int2 *pb, cudaStream_t s)
{
    const unsigned nb = (unsigned)((n + 127) / 128);
    if (n <= kPlaqVecSplit) k_plaq_vec<VEC, 1><<<dim3(nb, 6), 128, 0, s>>>(g, q, first, n, pa, pb);
    else k_plaq_vec<VEC, 6><<<nb, 128, 0, s>>>(g, q, first, n, pa, pb);
}

// the n vectors a plane of a slab
struct PlaqVecs {
    const int4 *a;
    const int2 *b;
    int n;
};
// what the vectors of a sum were
struct PlaqKinds {
    bool bad = false;   // one is out of range
    bool rough = false; // one is digits: links away from the identity
    unsigned top = 0;   // high word of the largest number among the doubles
};
// A vector as digits, doubles in units of 2^(E - 1022) (E = 1022 beside vectors in digits)
__device__ __forceinline__ void load_plaq(const PlaqVecs &P, int plane, int slot, int E, fx (&v)[3], PlaqKinds &kinds)
{
    const int4 a = __ldg(P.a + (size_t)plane * P.n + slot);
    const int2 b = __ldg(P.b + (size_t)plane * P.n + slot);
    v[0] = {a.x, a.y};
    v[1] = {a.z, a.w};
    v[2] = {b.x, b.y};
    if (!plaq_marked(a.x)) {
        kinds.rough = true;
    } else if (a.x == kPlaqBad) {
        kinds.bad = true;
    } else {
        const PlaqVec d = plaq_doubles(a, b);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            kinds.top = max(kinds.top, fx_abs_high(d.v[k]));
            v[k] = fx_from_double(d.v[k], E);
        }
    }
}

// A link that transports vectors: with u its vector part, t = u x v and d = |U|^2 - 1,
//   vec(U^+ v U) / |U|^2 = v + 2 (u0 t + u x t) (1 - d)
// to first order in d, which ok bounds by 2^-29.
struct Transport {
    fx u[3];
    fx w[4]; // 2 U (1 - d)
};
__device__ __forceinline__ Transport make_transport(const fxq &U, bool &ok)
{
    fxa nn = {-(1LL << 56), 0};
#pragma unroll
    for (int k = 0; k < 4; ++k) fx_mac(nn, U.c[k], U.c[k]);
    const long long d = fx_round(nn);
    ok = ok && d < (1 << 27) && d > -(1 << 27);
    Transport r;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        r.w[k] = {2 * U.c[k].h, 2 * (U.c[k].l - (int)(((long long)U.c[k].h * (int)d) >> 28))};
#pragma unroll
    for (int k = 0; k < 3; ++k) r.u[k] = U.c[k + 1];
    return r;
}
// sum += the transported v, in units of 2^-56 (|v| < 4)
__device__ __forceinline__ void transport_add(const Transport &T, const fx (&v)[3], long long (&sum)[3])
{
    fxa tc[3] = {}, acc[3];
    fx_mac_cross(tc, T.u, v);
    fx t[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        t[a] = fx_of(tc[a]);
        acc[a] = {fx_units64(v[a]), 0};
        fx_mac(acc[a], T.w[0], t[a]);
    }
    const fx wv[3] = {T.w[1], T.w[2], T.w[3]};
    fx_mac_cross(acc, wv, t);
#pragma unroll
    for (int a = 0; a < 3; ++a) sum[a] += fx_round(acc[a]);
}

} // namespace hr
