// hr_fix.cuh -- two-digit fixed-point arithmetic with FP64-class accuracy on the
// integer pipes (plain C++ as well as CUDA, HR_HD, so that the host can check it).
//
// GB300 executes native FP64 at 1.7 lane operations per clock and SM and an
// FP64 <-> FP32 conversion at 2.0 (measured; FP32 FMA 124, 32-bit integer
// multiply-add 64, 32 x 32 + 64 bit multiply-add about 30), so the kernels that
// compute on canonical doubles -- link derivatives, staples, the clover field
// strength -- were bound by the FP64 pipe at 3 to 5 % of the memory rate.
// Double-float pairs (48 bits) would be fast enough but less accurate.  A
// number here is
//   v = h 2^-28 + l 2^-56,   h, l int,
// in units of a power of two that the caller chooses: an absolute accuracy of
// 2^-56 of that unit, better than binary64's for numbers near it and worse for
// numbers below about 2^-3 of it.  Callers whose results can be that small (vector
// parts of links near the identity, sums that cancel) take a smaller unit or native
// FP64.  |l| <= 2^27 from the conversions that split at the middle (fx_split,
// fx_from_double, fx_from_pair: a little more), < 2^28 with the sign of v from
// fx_from_unit, which cuts.  A product of two numbers is three 32 x 32 -> 64 bit
// multiply-adds into two 64-bit sums that need no normalisation and no rounding:
//   a += h h' (units 2^-56),  b += h l' + l h' (units 2^-84);
// the dropped l l' is below 2^-58 for split digits, below 2^-56 and of the
// product's sign for cut ones (|q|^2 of a unit quaternion: off by at most 4.4 2^-56,
// 1.3 2^-56 on average).  That is about 0.1 clocks per SM and term against 0.59
// for a DFMA; a sum is otherwise exact until its one rounding at 2^-57.
// Callers guarantee the ranges (stated per function); blocks outside them
// (Inf, NaN, links far from unit length) take native FP64.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define HR_HD __host__ __device__
#else
#define HR_HD
#endif

namespace hr {

struct fx {
    int h, l;
};
struct fxa {
    long long a, b;
};

HR_HD inline unsigned fx_bits(float x)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    unsigned u;
    std::memcpy(&u, &x, 4);
    return u;
#endif
}
HR_HD inline float fx_float(unsigned u)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(u);
#else
    float x;
    std::memcpy(&x, &u, 4);
    return x;
#endif
}
HR_HD inline unsigned long long fx_dbits(double x)
{
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(x);
#else
    unsigned long long u;
    std::memcpy(&u, &x, 8);
    return u;
#endif
}
HR_HD inline double fx_double(unsigned long long u)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double x;
    std::memcpy(&x, &u, 8);
    return x;
#endif
}
// uncontracted FP32 operations
#ifdef __CUDA_ARCH__
__device__ __forceinline__ float fx_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fx_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fx_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fx_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
#else
inline float fx_add(float a, float b) { volatile float r = a + b; return r; }
inline float fx_sub(float a, float b) { volatile float r = a - b; return r; }
inline float fx_mul(float a, float b) { volatile float r = a * b; return r; }
inline float fx_fma(float a, float b, float c) { return std::fmaf(a, b, c); }
#endif

HR_HD inline fx fx_add(fx x, fx y) { return {x.h + y.h, x.l + y.l}; }
HR_HD inline fx fx_sub(fx x, fx y) { return {x.h - y.h, x.l - y.l}; }
HR_HD inline fx fx_neg(fx x) { return {-x.h, -x.l}; }

// s += x y.  |h| < 2^31 for any single product; the callers keep sum |h h'| < 2^63
HR_HD inline void fx_mac(fxa &s, fx x, fx y)
{
    s.a += (long long)x.h * y.h;
    s.b += (long long)x.h * y.l;
    s.b += (long long)x.l * y.h;
}

// the sum rounded to units of 2^-56
HR_HD inline long long fx_round(fxa s) { return s.a + ((s.b + (1LL << 27)) >> 28); }
// digits of t 2^-56, |t| < 2^58
HR_HD inline fx fx_split(long long t)
{
    const long long r = t + (1LL << 27);
    return {(int)(r >> 28), (int)((unsigned)r & 0xfffffffu) - (1 << 27)};
}
HR_HD inline long long fx_units64(fx v) { return (long long)v.h * (1LL << 28) + v.l; }
HR_HD inline fx fx_of(fxa s) { return fx_split(fx_round(s)); }

// t 2^-(56 + k) as a double, k <= 900: the exponent field moves, no FP64 product
HR_HD inline double fx_to_double(long long t, int k = 0)
{
    const double d = (double)t;
    return t ? fx_double(fx_dbits(d) - ((unsigned long long)(unsigned)(56 + k) << 52)) : 0.0;
}
// t 2^-56 (|t| < 2^59) as a normalised float pair: three 22-bit pieces made floats
// through the mantissa field, summed without loss until the low part is rounded, so
// the pair carries 2^-49 of the value, as one split from a double does
HR_HD inline void fx_to_pair(long long t, float &hi, float &lo)
{
    const float f2 = fx_sub(fx_float(0x4b400000u + (unsigned)(int)(t >> 44)), 12582912.f);
    const float f1 = fx_sub(fx_float(0x4b000000u | ((unsigned)(t >> 22) & 0x3fffffu)), 8388608.f);
    const float f0 = fx_sub(fx_float(0x4b000000u | ((unsigned)t & 0x3fffffu)), 8388608.f);
    const float a = fx_mul(f2, 0x1p-12f), b = fx_mul(f1, 0x1p-34f), c = fx_mul(f0, 0x1p-56f);
    const float s = fx_add(a, b), e = fx_sub(b, fx_sub(s, a)); // a + b = s + e
    hi = fx_add(s, fx_add(e, c));
    lo = fx_add(fx_sub(e, fx_sub(hi, s)), c); // (one rounding, of the low part)
}
// 2^k as a double, -1022 <= k <= 1023
HR_HD inline double fx_pow2(int k) { return fx_double((unsigned long long)(unsigned)(k + 1023) << 52); }

// ---------------------------------------------------------------- binary64 in
// Digits of a double with |x| < 4 (truncated at 2^-56): the mantissa shifted
// into place, no FP64 instruction.
HR_HD inline fx fx_from_double(double x)
{
    const unsigned long long u = fx_dbits(x);
    const int e = (int)(u >> 52) & 0x7ff;
    const unsigned long long m = ((u & 0xfffffffffffffULL) | 0x10000000000000ULL) << 10; // 2^62 <= m < 2^63 is [1, 2)
    // x = m 2^(e - 1023 - 62), so x 2^56 = m >> (1029 - e): a shift of 5 and
    // more for |x| < 4; beyond 63, and for zero and subnormals, nothing is left
    const int s = 1029 - e;
#ifdef __CUDA_ARCH__
    unsigned long long t;
    asm("shr.u64 %0, %1, %2;" : "=l"(t) : "l"(m), "r"(s)); // clamps at 64
#else
    const unsigned long long t = s > 63 ? 0 : m >> s;
#endif
    const long long sg = (long long)u >> 63;
    return fx_split((long long)(t ^ (unsigned long long)sg) - sg);
}
// Digits of a double with |x| < 2, cut instead of split at the middle (|l| < 2^28):
// 13 instead of 20 integer instructions
HR_HD inline fx fx_from_unit(double x)
{
    const unsigned long long u = fx_dbits(x);
    const unsigned long long m = ((u & 0xfffffffffffffULL) | 0x10000000000000ULL) << 4; // x 2^56 = m >> (1023 - e)
    const int s = 1023 - ((int)(u >> 52) & 0x7ff), sg = (int)(u >> 32) >> 31;
#ifdef __CUDA_ARCH__
    unsigned long long th, tl;
    asm("shr.u64 %0, %1, %2;" : "=l"(th) : "l"(m), "r"(s + 28)); // clamps at 64
    asm("shr.u64 %0, %1, %2;" : "=l"(tl) : "l"(m), "r"(s));
#else
    const unsigned long long th = s + 28 > 63 ? 0 : m >> (s + 28), tl = s > 63 ? 0 : m >> s;
#endif
    const int h = (int)(unsigned)th, l = (int)((unsigned)tl & 0xfffffffu);
    return {(h ^ sg) - sg, (l ^ sg) - sg};
}
// Digits of x / 2^(E - 1022) for |x| < 2^(E - 1022), E the biased exponent of the
// largest number of a block
HR_HD inline fx fx_from_double(double x, int E)
{
    const unsigned long long u = fx_dbits(x);
    const int e = (int)(u >> 52) & 0x7ff;
    const unsigned long long m = ((u & 0xfffffffffffffULL) | (e ? 0x10000000000000ULL : 0)) << 10;
    const int s = E - (e ? e : 1) + 7;
#ifdef __CUDA_ARCH__
    unsigned long long t;
    asm("shr.u64 %0, %1, %2;" : "=l"(t) : "l"(m), "r"(s));
#else
    const unsigned long long t = s > 63 ? 0 : m >> s;
#endif
    const long long sg = (long long)u >> 63;
    return fx_split((long long)(t ^ (unsigned long long)sg) - sg);
}
// |x| as the high word of its bits, for range tests: below fx_high(2^k) = (1023 + k) << 20
HR_HD inline unsigned fx_abs_high(double x) { return (unsigned)(fx_dbits(x) >> 32) & 0x7fffffffu; }
constexpr unsigned kFxHigh1 = 0x3ff00000u, kFxHigh2 = 0x40000000u;

// ---------------------------------------------------------------- float pairs in
// A block of float pairs (hi, lo) with the largest |hi| below 2^(E - 126), E
// its biased exponent: values are taken in units of 2^(E - 125), so |h| <= 2^27.
// E must lie in [kFxMinExp, 254]; the pairs are normalised (|lo| <= ulp(hi) / 2).
constexpr int kFxMinExp = 21, kFxPairBias = 125;
HR_HD inline float fx_pair_scale(int E) { return fx_float((unsigned)(274 - E) << 23); } // 2^(147 - E)

// hi and lo scaled to |hi| < 2^21; integer parts at 2^-22, 2^-40 and 2^-56 by
// adding and subtracting 1.5 2^23 (exact), read from the sum's mantissa bits
HR_HD inline fx fx_from_pair(float hi, float lo, float scale)
{
    const float M = 12582912.f; // 1.5 2^23
    const unsigned MB = 0x4b400000u;
    const float a = fx_mul(hi, scale), b = fx_mul(lo, scale);
    const float t0 = fx_add(a, M);
    const float r0 = fx_sub(a, fx_sub(t0, M)); // |r0| <= 1/2
    const float t1 = fx_fma(r0, 262144.f, M), t2 = fx_fma(b, 262144.f, M);
    const float r1 = fx_fma(r0, 262144.f, -fx_sub(t1, M)), r2 = fx_fma(b, 262144.f, -fx_sub(t2, M));
    const float t3 = fx_fma(fx_add(r1, r2), 65536.f, M);
    const int n12 = (int)(fx_bits(t1) + fx_bits(t2) - 2u * MB); // units 2^-40
    const int c = (n12 + (1 << 11)) >> 12;
    fx v;
    v.h = (int)((fx_bits(t0) - MB) << 6) + c;
    v.l = (int)((unsigned)(n12 - (c << 12)) << 16) + (int)(fx_bits(t3) - MB);
    return v;
}

// ---------------------------------------------------------------- common shift of a block of sums
HR_HD inline int fx_clz(unsigned long long x)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)x);
#else
    return x ? __builtin_clzll(x) : 64;
#endif
}
// bits in use by the sum (ORed over a block, for fx_block_shift)
HR_HD inline unsigned long long fx_used(fxa s)
{
    return (unsigned long long)(s.a ^ (s.a >> 63)) | ((unsigned long long)(s.b ^ (s.b >> 63)) >> 28);
}
// the left shift, -4 .. 28, that brings the largest sum of a block (|s| < 2^60) to between 2^55 and 2^57
HR_HD inline int fx_block_shift(unsigned long long used)
{
    const int s = fx_clz(used | 1u) - 8;
    return s < -4 ? -4 : (s > 28 ? 28 : s);
}
// the sum in units of 2^-(56 + s): (a 2^28 + b) >> (28 - s)
HR_HD inline long long fx_shifted(fxa s, int shift)
{
    const unsigned long long lo0 = (unsigned long long)s.a << 28, lo = lo0 + (unsigned long long)s.b;
    const long long hi = (s.a >> 36) + (s.b >> 63) + (lo < lo0 ? 1 : 0);
    const int q = 28 - shift; // 0 .. 32
#ifdef __CUDA_ARCH__
    const unsigned w0 = (unsigned)lo, w1 = (unsigned)(lo >> 32), w2 = (unsigned)hi;
    return (long long)(((unsigned long long)__funnelshift_rc(w1, w2, q) << 32) | __funnelshift_rc(w0, w1, q));
#else
    return (long long)((lo >> q) | (q ? (unsigned long long)hi << (64 - q) : 0));
#endif
}

// ---------------------------------------------------------------- quaternions
// Links: components in units of 1, |q|^2 within 1 % of 1 (fxq_near_unit), so that
// a product stays below 1.04 and a sum of six staples below 2^3.
// (a0 + i a.s)(b0 + i b.s) = (a0 b0 - a.b) + i (a0 b + b0 a - a x b).s
struct fxq {
    fx c[4];
};
HR_HD inline fxq fxq_conj(fxq q) { return {{q.c[0], fx_neg(q.c[1]), fx_neg(q.c[2]), fx_neg(q.c[3])}}; }
HR_HD inline fxq fxq_add(fxq a, fxq b)
{
    return {{fx_add(a.c[0], b.c[0]), fx_add(a.c[1], b.c[1]), fx_add(a.c[2], b.c[2]), fx_add(a.c[3], b.c[3])}};
}
// for |components| < 2, in 32-bit integers
HR_HD inline bool fxq_near_unit(const fxq &q)
{
    int n = -(1 << 26);
    for (int k = 0; k < 4; ++k) n += (q.c[k].h >> 15) * (q.c[k].h >> 15);
    return n > -(1 << 26) / 100 && n < (1 << 26) / 100;
}
// the vector part of a b into s[0..2]
HR_HD inline void fxq_mac_vec(fxa (&s)[3], const fxq &a, const fxq &b)
{
    const fx n1 = fx_neg(a.c[1]), n2 = fx_neg(a.c[2]), n3 = fx_neg(a.c[3]);
    fx_mac(s[0], a.c[0], b.c[1]); fx_mac(s[0], a.c[1], b.c[0]); fx_mac(s[0], n2, b.c[3]); fx_mac(s[0], a.c[3], b.c[2]);
    fx_mac(s[1], a.c[0], b.c[2]); fx_mac(s[1], a.c[2], b.c[0]); fx_mac(s[1], n3, b.c[1]); fx_mac(s[1], a.c[1], b.c[3]);
    fx_mac(s[2], a.c[0], b.c[3]); fx_mac(s[2], a.c[3], b.c[0]); fx_mac(s[2], n1, b.c[2]); fx_mac(s[2], a.c[2], b.c[1]);
}
// the scalar part of a b
HR_HD inline void fxq_mac_scalar(fxa &s, const fxq &a, const fxq &b)
{
    fx_mac(s, a.c[0], b.c[0]);
    fx_mac(s, fx_neg(a.c[1]), b.c[1]);
    fx_mac(s, fx_neg(a.c[2]), b.c[2]);
    fx_mac(s, fx_neg(a.c[3]), b.c[3]);
}
// s += u x v
HR_HD inline void fx_mac_cross(fxa (&s)[3], const fx (&u)[3], const fx (&v)[3])
{
    const fx n0 = fx_neg(v[0]), n1 = fx_neg(v[1]), n2 = fx_neg(v[2]);
    fx_mac(s[0], u[1], v[2]); fx_mac(s[0], u[2], n1);
    fx_mac(s[1], u[2], v[0]); fx_mac(s[1], u[0], n2);
    fx_mac(s[2], u[0], v[1]); fx_mac(s[2], u[1], n0);
}
// s += k q or q k, k = (0, k1, k2, k3) a pure vector
HR_HD inline void fxq_mac_pure_l(fxa (&s)[4], const fx (&k)[3], const fxq &q)
{
    const fx n0 = fx_neg(k[0]), n1 = fx_neg(k[1]), n2 = fx_neg(k[2]);
    fx_mac(s[0], n0, q.c[1]); fx_mac(s[0], n1, q.c[2]); fx_mac(s[0], n2, q.c[3]);
    fx_mac(s[1], k[0], q.c[0]); fx_mac(s[1], n1, q.c[3]); fx_mac(s[1], k[2], q.c[2]);
    fx_mac(s[2], k[1], q.c[0]); fx_mac(s[2], n2, q.c[1]); fx_mac(s[2], k[0], q.c[3]);
    fx_mac(s[3], k[2], q.c[0]); fx_mac(s[3], n0, q.c[2]); fx_mac(s[3], k[1], q.c[1]);
}
HR_HD inline void fxq_mac_pure_r(fxa (&s)[4], const fxq &q, const fx (&k)[3])
{
    const fx n0 = fx_neg(k[0]), n1 = fx_neg(k[1]), n2 = fx_neg(k[2]);
    fx_mac(s[0], n0, q.c[1]); fx_mac(s[0], n1, q.c[2]); fx_mac(s[0], n2, q.c[3]);
    fx_mac(s[1], k[0], q.c[0]); fx_mac(s[1], k[1], q.c[3]); fx_mac(s[1], n2, q.c[2]);
    fx_mac(s[2], k[1], q.c[0]); fx_mac(s[2], k[2], q.c[1]); fx_mac(s[2], n0, q.c[3]);
    fx_mac(s[3], k[2], q.c[0]); fx_mac(s[3], k[0], q.c[2]); fx_mac(s[3], n1, q.c[1]);
}
HR_HD inline void fxq_mac(fxa (&s)[4], const fxq &a, const fxq &b)
{
    fxa v[3] = {s[1], s[2], s[3]};
    fxq_mac_scalar(s[0], a, b);
    fxq_mac_vec(v, a, b);
    s[1] = v[0];
    s[2] = v[1];
    s[3] = v[2];
}
HR_HD inline fxq fxq_of(const fxa (&s)[4]) { return {{fx_of(s[0]), fx_of(s[1]), fx_of(s[2]), fx_of(s[3])}}; }
HR_HD inline fxq fxq_mul(const fxq &a, const fxq &b)
{
    fxa s0 = {0, 0}, s[3] = {{0, 0}, {0, 0}, {0, 0}};
    fxq_mac_scalar(s0, a, b);
    fxq_mac_vec(s, a, b);
    return {{fx_of(s0), fx_of(s[0]), fx_of(s[1]), fx_of(s[2])}};
}

} // namespace hr
