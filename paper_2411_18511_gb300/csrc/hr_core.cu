// hr_core.cu -- context, error reporting, sizes and the layout-conversion
// kernels (canonical <-> packed) of libhirep_gb300.
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "hr_cvt.cuh"
#include "hr_host.h"

using namespace hr;

// ====================================================================== errors

namespace hr {

hr_status set_error(hr_ctx *ctx, hr_status st, const char *fmt, ...)
{
    if (ctx) {
        char buf[1024];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(buf, sizeof buf, fmt, ap);
        va_end(ap);
        ctx->err = buf;
    }
    return st;
}

hr_status check_launch(hr_ctx *ctx, const char *what)
{
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_error(ctx, HR_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
    return HR_OK;
}

bool valid_rep(int rep) { return rep == HR_FUND || rep == HR_ADJ || rep == HR_ADJ_MAT; }
bool valid_prec(int prec) { return prec == HR_F64 || prec == HR_F32 || prec == HR_F16; }

static bool lattice_ok(const hr_lattice &lat, int nrhs)
{
    long long v = 1;
    for (int k = 0; k < 4; ++k) {
        if (lat.dims[k] < 2 || (lat.dims[k] & 1)) return false;
        v *= lat.dims[k];
    }
    if (nrhs < 1 || nrhs > kMaxRhs || (nrhs & (nrhs - 1))) return false;
    if (lat.bc & ~15) return false;
    // virtual-site indices and 16-byte vector indices must fit the kernels' int arithmetic
    return (v / 2) * nrhs * 12 < (1LL << 31);
}

hr_status check_buffers(hr_ctx *ctx, std::initializer_list<const void *> packed,
                        std::initializer_list<const void *> canonical, std::initializer_list<const void *> nullable)
{
    int k = 0;
    for (const void *p : packed) {
        if (!p) return set_error(ctx, HR_ERR_INVALID_ARG, "null field pointer (argument %d)", k);
        if ((uintptr_t)p & 15u) return set_error(ctx, HR_ERR_INVALID_ARG, "packed buffer %p not 16-byte aligned", p);
        ++k;
    }
    for (const void *p : canonical) {
        if (!p) return set_error(ctx, HR_ERR_INVALID_ARG, "null field pointer");
        if ((uintptr_t)p & 7u) return set_error(ctx, HR_ERR_INVALID_ARG, "canonical buffer %p not 8-byte aligned", p);
    }
    for (const void *p : nullable)
        if (p && ((uintptr_t)p & 15u)) return set_error(ctx, HR_ERR_INVALID_ARG, "work buffer %p not 16-byte aligned", p);
    return HR_OK;
}

hr_status validate_lattice(hr_ctx *ctx, const hr_lattice &lat, int nrhs)
{
    for (int k = 0; k < 4; ++k) {
        if (lat.dims[k] < 2) return set_error(ctx, HR_ERR_INVALID_ARG, "extent %d = %d < 2", k, lat.dims[k]);
        if (lat.dims[k] & 1) return set_error(ctx, HR_ERR_UNSUPPORTED, "extent %d = %d is odd (even-odd needs even extents)", k, lat.dims[k]);
    }
    if (nrhs < 1 || nrhs > kMaxRhs || (nrhs & (nrhs - 1)))
        return set_error(ctx, HR_ERR_UNSUPPORTED, "n_rhs = %d: must be a power of two in [1, %d]", nrhs, kMaxRhs);
    if (lat.bc & ~15) return set_error(ctx, HR_ERR_INVALID_ARG, "bc = %d: one bit per direction, [0, 15]", lat.bc);
    for (int k = 0; k < 4; ++k)
        if (!std::isfinite(lat.theta[k])) return set_error(ctx, HR_ERR_INVALID_ARG, "theta[%d] is not finite", k);
    if (!lattice_ok(lat, nrhs)) return set_error(ctx, HR_ERR_UNSUPPORTED, "lattice too large for 32-bit site indexing");
    return HR_OK;
}

size_t spinor_half_bytes(const Geom &g, int rep, int prec)
{
    int nc = rep_nc(rep);
    if (nc == 2) {
        if (prec == kF64) return SpinorLayout<2, kF64>::bytes(g.nblk_s);
        if (prec == kF32) return SpinorLayout<2, kF32>::bytes(g.nblk_s);
        return SpinorLayout<2, kF16>::bytes(g.nblk_s);
    }
    if (prec == kF64) return SpinorLayout<3, kF64>::bytes(g.nblk_s);
    if (prec == kF32) return SpinorLayout<3, kF32>::bytes(g.nblk_s);
    return SpinorLayout<3, kF16>::bytes(g.nblk_s);
}

// the bytes of a half that the 32-site blocks' lanes cover
static size_t packed_lane_bytes(const Geom &g, int rep, int prec)
{
    const size_t per = (size_t)8 * rep_nc(rep) * (prec == kF64 ? 8 : prec == kF32 ? 4 : 2) + (prec == kF16 ? 4 : 0);
    return (size_t)g.nblk_s * 32 * per;
}

size_t gauge_bytes(const Geom &g, int rep, int prec)
{
    size_t b;
    if (rep == HR_ADJ_MAT)
        b = prec == kF64 ? GaugeMat<kF64>::bytes(g.nblk_g) : prec == kF32 ? GaugeMat<kF32>::bytes(g.nblk_g) : GaugeMat<kF16>::bytes(g.nblk_g);
    else
        b = prec == kF64 ? GaugeQuat<kF64>::bytes(g.nblk_g) : prec == kF32 ? GaugeQuat<kF32>::bytes(g.nblk_g) : GaugeQuat<kF16>::bytes(g.nblk_g);
    return (b + 255) & ~(size_t)255;
}

} // namespace hr

// ====================================================================== kernels

namespace {

// the link U_mu(x) sits on the boundary slice x_mu = L_mu - 1 of an antiperiodic direction
__device__ __forceinline__ bool boundary_link(const Geom &g, int mu, const int (&x)[4])
{
    return ((g.bc >> mu) & 1) && x[mu] == g.d[mu] - 1;
}

// a double split on its way into a packed layout
struct PairVal {
    float h, l;
};
// x as a pair, by the FP64 pipe when it is out of the integer split's range;
// range flags into bad
struct PairFlags {
    PairVal v;
    unsigned bad;
};
__device__ __noinline__ PairFlags split_native(double x)
{
    const dd d = dd_from_double(x);
    return {{d.h, d.l}, pack_range_flags(x)};
}
__device__ __forceinline__ PairVal split_val(double x, unsigned &bad)
{
    PairVal v;
    if (!cvt_split(x, v.h, v.l)) {
        const PairFlags f = split_native(x);
        v = f.v;
        bad |= f.bad;
    }
    return v;
}
__device__ __noinline__ double join_native(float h, float l) { return (double)h + (double)l; }
__device__ __forceinline__ double join_val(dd v)
{
    double x;
    if (!cvt_join(v.h, v.l, x)) x = join_native(v.h, v.l);
    return x;
}
__device__ __forceinline__ double join_val(float v)
{
    double x;
    if (!cvt_widen(v, x)) x = join_native(v, 0.f);
    return x;
}

// 16 bytes of a canonical field (VEC: it is 16-byte aligned)
template <bool VEC> __device__ __forceinline__ double2 load_pair(const double *p)
{
    if constexpr (VEC) return *(const double2 *)p;
    else return make_double2(p[0], p[1]);
}
template <bool VEC> __device__ __forceinline__ void store_pair(double *p, double2 v)
{
    if constexpr (VEC) {
        *(double2 *)p = v;
    } else {
        p[0] = v.x;
        p[1] = v.y;
    }
}

} // namespace

namespace hr {
template <> struct Real<PairVal> {
    __device__ static dd to_dd(PairVal x) { return dd(x.h, x.l); }
    __device__ static float to_float(PairVal x) { return x.h; }
};
} // namespace hr

namespace {

// one thread per link (mu = blockIdx.y, lex site).  canon (adjoint): store the
// representative of +-q with the sign bit of q0 clear, then set it on boundary
// links; the fundamental stores -q on boundary links.  The threads beyond the
// sites zero the lanes that pad a parity's last block of 32.
template <int PREC, bool VEC>
__global__ void __launch_bounds__(256) k_gauge_pack_quat(Geom g, int canon, const double *__restrict__ can,
                                                         void *packed, unsigned *status)
{
    const unsigned V = 2u * (unsigned)g.vh, pad = (unsigned)g.nblk_g * 32u - (unsigned)g.vh;
    const unsigned x = blockIdx.x * blockDim.x + threadIdx.x;
    const int mu = blockIdx.y;
    if (x >= V + 2u * pad) return;
    if (x >= V) {
        const unsigned k = x - V;
        const PairVal z[4] = {};
        store_quat<PREC>(packed, g.nblk_g, k >= pad ? 1 : 0, mu, g.vh + (int)(k >= pad ? k - pad : k), z);
        return;
    }
    const int i = (int)(x >> 1), row = fdiv(i, g.div_h3), r1 = fdiv(row, g.div_d2);
    const int x3 = (int)(x - (unsigned)row * (unsigned)g.d[3]), x2 = row - r1 * g.d[2];
    const int x0 = fdiv(r1, g.div_d1), x1 = r1 - x0 * g.d[1];
    const int p = (x0 + x1 + x2 + x3) & 1;
    const double *src = can + ((size_t)mu * V + x) * 4;
    const double2 q01 = load_pair<VEC>(src), q23 = load_pair<VEC>(src + 2);
    double a[4] = {q01.x, q01.y, q23.x, q23.y};
    const int xc[4] = {x0, x1, x2, x3};
    const bool neg = (canon && sign_bit(a[0])) != boundary_link(g, mu, xc);
    PairVal v[4];
    unsigned bad = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = split_val(neg ? -a[k] : a[k], bad);
    if (bad) atomicOr(status, bad);
    store_quat<PREC>(packed, g.nblk_g, p, mu, i, v);
}

template <int PREC>
__global__ void k_gauge_pack_mat(Geom g, const double *__restrict__ can, void *packed, unsigned *status)
{
    long long V = 2LL * g.vh;
    long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 4 * V) return;
    int mu = (int)(t / V);
    long long x = t - (long long)mu * V;
    int x3 = (int)(x % g.d[3]);
    long long r = x / g.d[3];
    int x2 = (int)(r % g.d[2]);
    r /= g.d[2];
    int x1 = (int)(r % g.d[1]);
    int x0 = (int)(r / g.d[1]);
    int p = (x0 + x1 + x2 + x3) & 1;
    int i = (int)(x >> 1);
    double a[4] = {can[t * 4 + 0], can[t * 4 + 1], can[t * 4 + 2], can[t * 4 + 3]};
    const unsigned bad = pack_range_flags(a[0]) | pack_range_flags(a[1]) | pack_range_flags(a[2]) | pack_range_flags(a[3]);
    if (bad) atomicOr(status, bad);
    if (sign_bit(a[0]))
        for (int k = 0; k < 4; ++k) a[k] = -a[k]; // R(q) = R(-q); quat_to_adj reads the sign bit
    double R[3][3];
    quat_to_adj(a, R);
    const int xc[4] = {x0, x1, x2, x3};
    const double sg = boundary_link(g, mu, xc) ? -1.0 : 1.0;
    for (int e = 0; e < 9; ++e) {
        store_mat_entry<PREC>(packed, g.nblk_g, p, mu, i, e, sg * R[e / 3][e % 3]);
    }
}

// canonical double[nrhs][V][4][NC][2] <-> packed virtual sites, blockIdx.y-th of
// the parities from p0 on (packed halves `half` bytes apart).  A warp moves 32
// virtual sites: the packed side in 16-byte vectors of consecutive lanes, the
// canonical side in whole sites of CH 16-byte chunks (consecutive lanes, consecutive
// chunks), through a transposition in shared memory whose rows of CH + 1 chunks
// are free of bank conflicts.  Both are then bound by HBM; a thread that read or
// wrote a whole site in 8-byte steps and converted on the FP64 pipe took 590 us to
// unpack a 48^4 field.
constexpr int kConvWarps = 4;

template <int NC, int PREC, bool VEC>
__global__ void __launch_bounds__(32 * kConvWarps) k_spinor_pack(Geom g, int p0, const double *__restrict__ can,
                                                                 char *packed, size_t half, unsigned *status)
{
    constexpr int CH = 4 * NC;
    __shared__ double2 tile[kConvWarps][32][CH + 1];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nv = g.vh << g.lrhs;
    const int j0 = (blockIdx.x * kConvWarps + w) * 32, j = j0 + lane, p = p0 + blockIdx.y;
    if (j0 >= g.nblk_s * 32) return; // the whole warp
    unsigned site = 0; // r V + lex
    if (j < nv) site = (unsigned)(j & (g.nrhs - 1)) * (2u * g.vh) + (unsigned)eo_to_lex(g, j >> g.lrhs, p);
#pragma unroll
    for (int q = lane; q < 32 * CH; q += 32) {
        const int k = q / CH, c = q - k * CH;
        const unsigned s = __shfl_sync(0xffffffffu, site, k);
        if (j0 + k < nv) tile[w][k][c] = load_pair<VEC>(can + ((size_t)s * CH + c) * 2);
    }
    __syncwarp();
    cpx<PairVal> v[4][NC] = {}; // padding lanes hold zeros
    if (j < nv) {
        unsigned bad = 0;
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const double2 x = tile[w][lane][a * NC + c];
                v[a][c] = {split_val(x.x, bad), split_val(x.y, bad)};
            }
        if (bad) atomicOr(status, bad);
    }
    store_spinor<NC, PREC>(packed + blockIdx.y * half, g.nblk_s, j, v);
}

template <int NC, int PREC, bool VEC>
__global__ void __launch_bounds__(32 * kConvWarps) k_spinor_unpack(Geom g, int p0, const char *packed, size_t half,
                                                                   double *__restrict__ can)
{
    using T = typename PrecTraits<PREC>::T;
    constexpr int CH = 4 * NC;
    __shared__ double2 tile[kConvWarps][32][CH + 1];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nv = g.vh << g.lrhs;
    const int j0 = (blockIdx.x * kConvWarps + w) * 32, j = j0 + lane, p = p0 + blockIdx.y;
    if (j0 >= nv) return; // the whole warp
    unsigned site = 0;
    if (j < nv) {
        site = (unsigned)(j & (g.nrhs - 1)) * (2u * g.vh) + (unsigned)eo_to_lex(g, j >> g.lrhs, p);
        cpx<T> v[4][NC];
        load_spinor<NC, PREC>(packed + blockIdx.y * half, g.nblk_s, j, v);
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int c = 0; c < NC; ++c) tile[w][lane][a * NC + c] = make_double2(join_val(v[a][c].re), join_val(v[a][c].im));
    }
    __syncwarp();
#pragma unroll
    for (int q = lane; q < 32 * CH; q += 32) {
        const int k = q / CH, c = q - k * CH;
        const unsigned s = __shfl_sync(0xffffffffu, site, k);
        if (j0 + k < nv) store_pair<VEC>(can + ((size_t)s * CH + c) * 2, tile[w][k][c]);
    }
}

template <int NC, int PREC, bool VEC>
hr_status launch_spinor_convert(hr_ctx *ctx, const Geom &g, int p0, int np, double *can, char *packed, size_t half,
                                bool unpack, cudaStream_t s)
{
    const dim3 grid((unsigned)((g.nblk_s + kConvWarps - 1) / kConvWarps), (unsigned)np);
    if (unpack) k_spinor_unpack<NC, PREC, VEC><<<grid, 32 * kConvWarps, 0, s>>>(g, p0, packed, half, can);
    else k_spinor_pack<NC, PREC, VEC><<<grid, 32 * kConvWarps, 0, s>>>(g, p0, can, packed, half, ctx->d_counters + C_PACK);
    return check_launch(ctx, unpack ? "spinor unpack" : "spinor pack");
}

hr_status spinor_convert(hr_ctx *ctx, hr_lattice lat, int rep, int prec, int parity, int n_rhs, const double *can,
                         void *packed, bool unpack, cudaStream_t s)
{
    if (!ctx) return HR_ERR_INVALID_ARG;
    if (!valid_rep(rep) || !valid_prec(prec)) return set_error(ctx, HR_ERR_INVALID_ARG, "bad rep/prec");
    if (parity < 0 || parity > 2) return set_error(ctx, HR_ERR_INVALID_ARG, "bad parity %d", parity);
    hr_status st = validate_lattice(ctx, lat, n_rhs);
    if (st) return st;
    st = check_buffers(ctx, {packed}, {can});
    if (st) return st;
    Geom g = make_geom(lat, n_rhs);
    size_t half = spinor_half_bytes(g, rep, prec);
    int nc = rep_nc(rep);
    const int p0 = parity == HR_FULL ? 0 : parity, np = parity == HR_FULL ? 2 : 1;
    // the packed bytes that no lane covers (binary16: the scales' rounding to 256)
    const size_t used = packed_lane_bytes(g, rep, prec);
    if (!unpack && used < half) {
        for (int k = 0; k < np; ++k) {
            cudaError_t e = cudaMemsetAsync((char *)packed + k * half + used, 0, half - used, s);
            if (e != cudaSuccess) return set_error(ctx, HR_ERR_CUDA, "spinor pack: %s", cudaGetErrorString(e));
        }
    }
    const bool vec = ((uintptr_t)can & 15u) == 0;
    auto go = [&](auto nc_, auto prec_) {
        constexpr int NC = decltype(nc_)::value, PREC = decltype(prec_)::value;
        return vec ? launch_spinor_convert<NC, PREC, true>(ctx, g, p0, np, (double *)can, (char *)packed, half, unpack, s)
                   : launch_spinor_convert<NC, PREC, false>(ctx, g, p0, np, (double *)can, (char *)packed, half, unpack, s);
    };
    auto by_prec = [&](auto nc_) {
        if (prec == kF64) return go(nc_, std::integral_constant<int, kF64>());
        if (prec == kF32) return go(nc_, std::integral_constant<int, kF32>());
        return go(nc_, std::integral_constant<int, kF16>());
    };
    return nc == 2 ? by_prec(std::integral_constant<int, 2>()) : by_prec(std::integral_constant<int, 3>());
}

// packed FP64 gauge -> packed gauge of precision PD, one thread per (p, mu, site)
template <int PD, bool MAT>
__global__ void k_gauge_convert(Geom g, const void *src, void *dst)
{
    long long n = 8LL * g.nblk_g * 32;
    long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    size_t slot = (size_t)(t >> 5);
    int lane = (int)(t & 31);
    if (MAT) {
        for (int e = 0; e < 9; ++e) {
            size_t idx = (slot * 9 + e) * 32 + lane;
            float2 w = ((const float2 *)src)[idx];
            float v = __fadd_rn(w.x, w.y);
            if (PD == kF32) ((float *)dst)[idx] = v;
            else ((__half *)dst)[idx] = __float2half_rn(v);
        }
    } else {
        // FP64 packed links are double-float pairs: hi float4 then lo float4
        const float4 *q = (const float4 *)src;
        float4 hi = q[(slot * 2 + 0) * 32 + lane], lo = q[(slot * 2 + 1) * 32 + lane];
        // the sign of hi survives (-0 + 0 would round to +0 and lose the
        // adjoint links' boundary bit on a link with q0 = 0)
        float4 w0 = make_float4(copysignf(__fadd_rn(hi.x, lo.x), hi.x), copysignf(__fadd_rn(hi.y, lo.y), hi.y),
                                copysignf(__fadd_rn(hi.z, lo.z), hi.z), copysignf(__fadd_rn(hi.w, lo.w), hi.w));
        if (PD == kF32) {
            ((float4 *)dst)[slot * 32 + lane] = w0;
        } else {
            __half2 h0 = __floats2half2_rn(w0.x, w0.y);
            __half2 h1 = __floats2half2_rn(w0.z, w0.w);
            uint2 w;
            w.x = *reinterpret_cast<uint32_t *>(&h0);
            w.y = *reinterpret_cast<uint32_t *>(&h1);
            ((uint2 *)dst)[slot * 32 + lane] = w;
        }
    }
}

} // namespace

namespace hr {
hr_status consume_pack_status(hr_ctx *ctx, cudaStream_t s)
{
    unsigned flags = 0;
    cudaError_t e = cudaMemcpyAsync(&flags, ctx->d_counters + C_PACK, sizeof flags, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e == cudaSuccess && flags) e = cudaMemsetAsync(ctx->d_counters + C_PACK, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(ctx, HR_ERR_CUDA, "pack status readback: %s", cudaGetErrorString(e));
    }
    if (flags & kPackNonFinite) return set_error(ctx, HR_ERR_NUMERIC, "a packed field held a NaN or Inf");
    if (flags & kPackAboveRange)
        return set_error(ctx, HR_ERR_UNSUPPORTED,
                         "a packed value exceeded 2^120 = 1.3e36 in magnitude (the pair-of-floats FP64 layout "
                         "keeps the float exponent range): scale the field down");
    return HR_OK;
}

hr_status gauge_convert(hr_ctx *ctx, const Geom &g, int rep, int pdst, const void *src, void *dst, cudaStream_t s)
{
    long long n = 8LL * g.nblk_g * 32;
    int bs = 256;
    int grid = (int)((n + bs - 1) / bs);
    bool mat = rep == HR_ADJ_MAT;
    if (pdst == kF32) {
        if (mat) k_gauge_convert<kF32, true><<<grid, bs, 0, s>>>(g, src, dst);
        else k_gauge_convert<kF32, false><<<grid, bs, 0, s>>>(g, src, dst);
    } else if (pdst == kF16) {
        if (mat) k_gauge_convert<kF16, true><<<grid, bs, 0, s>>>(g, src, dst);
        else k_gauge_convert<kF16, false><<<grid, bs, 0, s>>>(g, src, dst);
    } else {
        return set_error(ctx, HR_ERR_UNSUPPORTED, "gauge convert target precision");
    }
    return check_launch(ctx, "gauge convert");
}
} // namespace hr

// ====================================================================== C ABI

extern "C" {

const char *hr_version(void) { return "hirep_gb300 0.1 (sm_103a)"; }

double hr_kappa_to_m0(double kappa) { return 1.0 / (2.0 * kappa) - 4.0; }
double hr_m0_to_kappa(double m0) { return 1.0 / (8.0 + 2.0 * m0); }

hr_status hr_ctx_create(hr_ctx **out, int device)
{
    if (!out) return HR_ERR_INVALID_ARG;
    *out = nullptr;
    int n = 0;
    if (cudaGetDeviceCount(&n) != cudaSuccess || device < 0 || device >= n) {
        cudaGetLastError();
        return HR_ERR_CUDA;
    }
    hr_ctx *ctx = new hr_ctx();
    ctx->device = device;
    cudaError_t e = cudaSetDevice(device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&ctx->sm_count, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess) e = cudaMalloc(&ctx->d_partials, sizeof(double) * (kMaxPartials + kFinBlocks * kMaxRhs));
    if (e == cudaSuccess) e = cudaMalloc(&ctx->d_counters, sizeof(unsigned) * kNumCounters);
    if (e == cudaSuccess) e = cudaMemset(ctx->d_counters, 0, sizeof(unsigned) * kNumCounters);
    if (e == cudaSuccess) e = cudaMalloc(&ctx->d_slab, kSlabBytes);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ctx->ev_slab, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaMalloc(&ctx->d_scal, sizeof(double) * kScalDoubles);
    if (e == cudaSuccess) e = cudaMemset(ctx->d_scal, 0, sizeof(double) * kScalDoubles);
    if (e == cudaSuccess) e = cudaMallocHost(&ctx->h_scal, sizeof(double) * kScalDoubles);
    if (e == cudaSuccess) e = cudaEventCreate(&ctx->ev0);
    if (e == cudaSuccess) e = cudaEventCreate(&ctx->ev1);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&ctx->side, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ctx->ev_fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ctx->ev_join, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        cudaGetLastError();
        hr_ctx_destroy(ctx);
        return HR_ERR_CUDA;
    }
    const char *path = getenv("HR_AUTOTUNE_CACHE");
    if (path && path[0]) {
        ctx->tune_cache_path = path;
        tune_cache_load(ctx);
    }
    const char *inj = getenv("HR_INJECT_TILE_NO_COPY");
    ctx->inject_tile_no_copy = (inj && inj[0] == '1') ? 1 : 0;
    *out = ctx;
    return HR_OK;
}

hr_status hr_ctx_destroy(hr_ctx *ctx)
{
    if (!ctx) return HR_ERR_INVALID_ARG;
    cudaSetDevice(ctx->device);
    if (ctx->d_partials) cudaFree(ctx->d_partials);
    if (ctx->d_counters) cudaFree(ctx->d_counters);
    if (ctx->d_slab) cudaFree(ctx->d_slab);
    if (ctx->ev_slab) cudaEventDestroy(ctx->ev_slab);
    if (ctx->d_scal) cudaFree(ctx->d_scal);
    if (ctx->h_scal) cudaFreeHost(ctx->h_scal);
    if (ctx->ev0) cudaEventDestroy(ctx->ev0);
    if (ctx->ev1) cudaEventDestroy(ctx->ev1);
    if (ctx->side) cudaStreamDestroy(ctx->side);
    if (ctx->ev_fork) cudaEventDestroy(ctx->ev_fork);
    if (ctx->ev_join) cudaEventDestroy(ctx->ev_join);
    for (auto &kv : ctx->graphs) {
        cudaGraphExecDestroy(kv.second.second);
        cudaGraphDestroy(kv.second.first);
    }
    delete ctx;
    return HR_OK;
}

hr_status hr_ctx_status(hr_ctx *ctx, hr_stream stream)
{
    if (!ctx) return HR_ERR_INVALID_ARG;
    return consume_pack_status(ctx, (cudaStream_t)stream);
}

const char *hr_last_error(const hr_ctx *ctx)
{
    if (!ctx) return "null context";
    return ctx->err.c_str();
}

size_t hr_gauge_packed_bytes(hr_lattice lat, hr_rep rep, hr_prec prec)
{
    if (!valid_rep(rep) || !valid_prec(prec) || !lattice_ok(lat, 1)) return 0;
    return gauge_bytes(make_geom(lat, 1), rep, prec);
}

size_t hr_spinor_packed_bytes(hr_lattice lat, hr_rep rep, hr_prec prec, hr_parity parity, int n_rhs)
{
    if (!valid_rep(rep) || !valid_prec(prec) || !lattice_ok(lat, n_rhs)) return 0;
    if (parity < 0 || parity > 2) return 0;
    size_t half = spinor_half_bytes(make_geom(lat, n_rhs), rep, prec);
    return parity == HR_FULL ? 2 * half : half;
}

hr_status hr_gauge_pack(hr_ctx *ctx, hr_lattice lat, hr_rep rep, hr_prec prec, const double *canonical, void *packed,
                        hr_stream stream)
{
    if (!ctx) return HR_ERR_INVALID_ARG;
    if (!valid_rep(rep) || !valid_prec(prec)) return set_error(ctx, HR_ERR_INVALID_ARG, "bad rep/prec");
    hr_status st = validate_lattice(ctx, lat, 1);
    if (st) return st;
    st = check_buffers(ctx, {packed}, {canonical});
    if (st) return st;
    Geom g = make_geom(lat, 1);
    cudaStream_t s = (cudaStream_t)stream;
    unsigned *status = ctx->d_counters + C_PACK;
    if (rep == HR_ADJ_MAT) {
        // zero the padding lanes so packed buffers are fully defined
        cudaMemsetAsync(packed, 0, gauge_bytes(g, rep, prec), s);
        const int bs = 256, grid = (int)((8LL * g.vh + bs - 1) / bs);
        if (prec == kF64) k_gauge_pack_mat<kF64><<<grid, bs, 0, s>>>(g, canonical, packed, status);
        else if (prec == kF32) k_gauge_pack_mat<kF32><<<grid, bs, 0, s>>>(g, canonical, packed, status);
        else k_gauge_pack_mat<kF16><<<grid, bs, 0, s>>>(g, canonical, packed, status);
    } else {
        const int canon = rep == HR_ADJ ? 1 : 0;
        const dim3 grid((unsigned)((64LL * g.nblk_g + 255) / 256), 4);
        const bool vec = ((uintptr_t)canonical & 15u) == 0;
        auto go = [&](auto prec_) {
            constexpr int PREC = decltype(prec_)::value;
            if (vec) k_gauge_pack_quat<PREC, true><<<grid, 256, 0, s>>>(g, canon, canonical, packed, status);
            else k_gauge_pack_quat<PREC, false><<<grid, 256, 0, s>>>(g, canon, canonical, packed, status);
        };
        if (prec == kF64) go(std::integral_constant<int, kF64>());
        else if (prec == kF32) go(std::integral_constant<int, kF32>());
        else go(std::integral_constant<int, kF16>());
    }
    return check_launch(ctx, "gauge pack");
}

hr_status hr_spinor_pack(hr_ctx *ctx, hr_lattice lat, hr_rep rep, hr_prec prec, hr_parity parity, int n_rhs,
                         const double *canonical, void *packed, hr_stream stream)
{
    return spinor_convert(ctx, lat, rep, prec, parity, n_rhs, canonical, packed, false, (cudaStream_t)stream);
}

hr_status hr_spinor_unpack(hr_ctx *ctx, hr_lattice lat, hr_rep rep, hr_prec prec, hr_parity parity, int n_rhs,
                           const void *packed, double *canonical, hr_stream stream)
{
    return spinor_convert(ctx, lat, rep, prec, parity, n_rhs, canonical, (void *)packed, true,
                          (cudaStream_t)stream);
}

} // extern "C"
