// hr_host.h -- host-side internals of libhirep_gb300: the context, error
// reporting, argument validation and launch helpers shared by the .cu files.
#pragma once

#include <cstdarg>
#include <cstdio>
#include <cstdint>
#include <initializer_list>
#include <map>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include <cuda_runtime.h>

#include "hirep_gb300.h"
#include "hr_internal.cuh"

// Device scratch owned by a context (allocated once in hr_ctx_create).
namespace hr {
constexpr int kMaxBlocks = 4096;      // cap on blocks of the vector kernels and of 32-RHS reducing launches
constexpr int kMaxRhs = 32;
constexpr int kMaxPartials = kMaxBlocks * kMaxRhs; // partial sums of one reducing launch
constexpr int kFinBlocks = 64;       // blocks of a finishing launch, at most
constexpr int kNumCounters = 64;
// scratch of the forces, filled slab by slab: vectors of the gauge force, digits
// of the link derivatives (bytes a site)
constexpr size_t kSlabBytes = 64u << 20, kPlaqSiteBytes = 144, kDigitSiteBytes = 264;
constexpr int kScalDoubles = 64 * kMaxRhs;

// launch shape of the hop kernel chosen by the autotuner
struct HopChoice {
    int variant; // kernel variant, 0 .. kNumHopVariants-1 (hr_hop.cu)
    int block;   // threads per block
};
constexpr int kNumHopVariants = 24;
} // namespace hr

struct hr_ctx {
    int device = 0;
    int sm_count = 0;
    std::string err;
    double *d_partials = nullptr;  // kMaxPartials, then kFinBlocks * kMaxRhs sums of a finishing launch's blocks
    unsigned *d_counters = nullptr;
    void *d_slab = nullptr;        // kSlabBytes: scratch of the forces, used under a SlabLease only
    cudaEvent_t ev_slab = nullptr; // the last lease's work
    std::mutex slab_mutex;
    double *d_scal = nullptr;      // kScalDoubles
    double *h_scal = nullptr;      // pinned mirror
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    // a finishing launch beside the next hop: its stream, fork and join
    cudaStream_t side = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    int fin_rows = 0; // rows that the last reducing hop left to its caller (HopLaunch::leave)
    std::map<std::string, hr::HopChoice> tuned; // autotuner: configuration key -> launch shape
    std::string tune_cache_path;                // JSON cache (HR_AUTOTUNE_CACHE), "" = none
    // instantiated CG iteration graphs, keyed by everything they bake in
    std::map<std::string, std::pair<cudaGraph_t, cudaGraphExec_t>> graphs;
    std::vector<std::string> graph_order;
    // failure injection for tests (HR_INJECT_TILE_NO_COPY=1 when the context is
    // created): the tiled hop's bulk copies are announced but never queued, so
    // its bounded waits run out (shortened to about half a millisecond)
    int inject_tile_no_copy = 0;
};
namespace hr {
constexpr size_t kMaxGraphs = 8;
}

namespace hr {

hr_status set_error(hr_ctx *ctx, hr_status st, const char *fmt, ...);
// Device buffers handed to an entry point: packed fields and work buffers are
// read and written as 16-byte vectors, canonical fields as doubles.  A null or
// misaligned one is an argument error, caught before any launch.  (nullable:
// only checked when not null.)
hr_status check_buffers(hr_ctx *ctx, std::initializer_list<const void *> packed,
                        std::initializer_list<const void *> canonical = {},
                        std::initializer_list<const void *> nullable = {});
hr_status check_launch(hr_ctx *ctx, const char *what);
hr_status validate_lattice(hr_ctx *ctx, const hr_lattice &lat, int nrhs);
bool valid_rep(int rep);
bool valid_prec(int prec);
inline int rep_nc(int rep) { return rep == HR_FUND ? 2 : 3; }

size_t spinor_half_bytes(const Geom &g, int rep, int prec);
size_t gauge_bytes(const Geom &g, int rep, int prec);

inline int grid_for(long long n, int block, int cap)
{
    long long b = (n + block - 1) / block;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (int)b;
}

// device counters: blocks of a finishing launch, native-path requests
// (C_PACK: the pack status word, kPack* flags of the values packed since the
// last check, read and cleared by consume_pack_status)
enum Counter { C_FIN = 0, C_FOLD = 1, C_PACK = 62, C_STATUS = 63 };

// clover site term in a hop epilogue (hr_clover.cuh): none, A(x) on the aux
// term (out = alpha A aux + beta acc), or A(x) on the result (out = A (alpha aux + beta acc))
enum ClovMode { kClovNone = 0, kClovAux = 1, kClovOut = 2 };

// Launch a kernel whose first statement is after_previous().  With `early` it may
// become resident as the previous kernel of the stream drains, which hides its
// launch latency: HMC at 16^4 27.1 -> 26.0 ms, binary16 solve at 32^4 7.6 -> 7.4 ms,
// adjoint operator at 32 x 24^3 557 -> 537 us.  Not for large fields: 16 right-hand
// sides on 26 x 22 x 18 x 20 (1.6 M sites) went from 24.3 to 24.8 ms.
constexpr long long kEarlySites = 1 << 20; // virtual sites of one parity
template <class... P, class... A>
inline void launch_after(void (*kernel)(P...), bool early, int grid, int block, size_t smem, cudaStream_t s, A... args)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &attr;
    c.numAttrs = early ? 1 : 0;
    cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}
inline bool early_start(const Geom &g) { return ((long long)g.vh << g.lrhs) <= kEarlySites; }

// A condition of the solve graph that a finishing launch sets: 1 when a reliable
// update is due, else 0 (set == 0: none).
struct FinCond {
    int set;
    unsigned long long handle;
};
// Add the `nparts` rows of nrhs partial sums in the context's scratch and run the
// scalar update `fin` on them (hr_blas.cu); skipped like the launch that wrote
// them when *gate == 0 or *done != 0.
hr_status finish_sums(hr_ctx *ctx, int nparts, int nrhs, int fin, const double *gate, const double *done,
                      cudaStream_t s, FinCond cond = {0, 0});

// Who finishes a reducing hop's rows: the launch itself; the caller; the caller if
// they are few enough for every block of the next kernel to add them (kFoldSums), else
// the launch (fin_rows = 0 then)
enum LeaveRows { kLeaveNone = 0, kLeaveAll = 1, kLeaveFew = 2 };
constexpr int kFoldSums = 1024;

// ---- hop launches (hr_hop.cu) ----
struct HopLaunch {
    int p;                 // output parity
    const void *gauge;
    const void *in;
    const void *aux;
    void *out;
    double alpha, beta;
    int g5_in, g5_out;
    int fin;               // FinishMode of the |out|^2 reduction (kFinNone: no reduction)
    const double *gate;    // skip the launch's work unless *gate != 0 (nullable)
    const double *done;    // skip the launch's work when *done != 0 (nullable)
    // fused CG update (nullable): instead of storing out, x += alpha p and
    // r -= alpha out with alpha per RHS from the scalar block, |r|^2 -> fin
    void *cg_x;
    const void *cg_p;
    void *cg_r;
    // clover site term (nullable): the half-field of the output parity
    // (clover_half) and how the epilogue applies it (ClovMode)
    const void *clov;
    int clov_mode;
    FinCond cond;
    int leave;  // of a reducing launch: kLeaveNone, or the caller finishes the rows (ctx->fin_rows)
    int joined; // the launch waits for another stream too: no early start
};
// a CG x/r update fused into the last hop of an operator (the operator's
// precision; x in FP32 when the operator runs in binary16)
struct CgFuse {
    void *x;
    const void *p;
    void *r;
    int fin; // kFinBeta or kFinBetaMixed
    FinCond cond;
    int leave; // LeaveRows of that hop
};
hr_status launch_hop(hr_ctx *ctx, const Geom &g, int rep, int prec, const HopLaunch &L, cudaStream_t s);
hr_status launch_hop_with(hr_ctx *ctx, const Geom &g, int rep, int prec, const HopLaunch &L, HopChoice c,
                          cudaStream_t s);
HopChoice hop_choice(hr_ctx *ctx, const Geom &g, int rep, int prec);
std::string tune_key(const Geom &g, int rep, int prec);
// the shape of reducing launches (aux read and |out|^2 or a fused CG update):
// their own tuned choice if there is one, else the plain one
HopChoice hop_choice_fin(hr_ctx *ctx, const Geom &g, int rep, int prec);
std::string tune_key_fin(const Geom &g, int rep, int prec);
bool hop_variant_available(int rep, int prec, int variant, int nrhs);
// autotuner cache file (hr_tune.cu)
void tune_cache_load(hr_ctx *ctx);
bool tune_cache_save(hr_ctx *ctx);
// out = op(in) on even sites, work = odd temporary (+ even temporary for NORMAL)
hr_status apply_eo_op(hr_ctx *ctx, const Geom &g, double m0, int rep, int prec, int op, const void *gauge,
                      const void *in, void *out, void *work_odd, void *work_even, int fin_schur,
                      const double *gate, const double *done, cudaStream_t s, const CgFuse *fuse = nullptr,
                      const void *clover = nullptr);

// Slabs of time slices whose data (bytes a site) fit the context's scratch, each with
// one neighbouring slice: `slots` slices fit; 0 slabs: not even two do.  Slab k of n
// holds slices [lo, hi); n == 1 is the whole lattice, without a neighbour.
struct Slabs {
    int n, T;
    int lo(int k) const { return (int)((long long)T * k / n); }
    int hi(int k) const { return lo(k + 1); }
};
inline Slabs make_slabs(const Geom &g, size_t site_bytes)
{
    const long long slice = (long long)g.d[1] * g.d[2] * g.d[3], fit = (long long)(kSlabBytes / site_bytes) / slice;
    const int T = g.d[0];
    if (fit >= T) return {1, T};
    return {fit < 2 ? 0 : (int)((T + fit - 2) / (fit - 1)), T};
}

// The context's slab scratch for the launches of one call on stream s.  The calls that
// use it (gauge force, link derivatives, clover build) touch no other scratch of
// the context, and a caller may not even choose the context (autograd keeps one per
// device and runs each backward on its forward's stream), so they must not depend on
// one stream: a lease holds the mutex while the call queues its launches, waits on
// the device for the lease before it, whatever its stream, and marks the end of its
// own launches.  Event calls alone, about 2 us of host time a call.
// mem == nullptr: not wanted, or s is being captured into a graph, which may be
// replayed beside anything (and after the context is gone); the caller then takes
// its kernels without scratch.
struct SlabLease {
    hr_ctx *ctx;
    cudaStream_t s;
    void *mem = nullptr;
    std::unique_lock<std::mutex> lock;
    SlabLease(hr_ctx *c, cudaStream_t stream, bool want) : ctx(c), s(stream)
    {
        cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
        if (!want) return;
        if (cudaStreamIsCapturing(s, &st) != cudaSuccess) { // (the launches will say why)
            cudaGetLastError();
            return;
        }
        if (st != cudaStreamCaptureStatusNone) return;
        lock = std::unique_lock<std::mutex>(ctx->slab_mutex);
        if (cudaStreamWaitEvent(s, ctx->ev_slab, 0) == cudaSuccess) mem = ctx->d_slab;
        else cudaGetLastError();
    }
    ~SlabLease()
    {
        if (mem) cudaEventRecord(ctx->ev_slab, s);
    }
    SlabLease(const SlabLease &) = delete;
    SlabLease &operator=(const SlabLease &) = delete;
};

// ---- link derivatives (hr_force.cu) ----
// out += beta dRe<a, H b> for full fields given by their even and odd halves
// (mode 0: su(2) force [4][V][3]; 1: quaternion gradient [4][V][4], no gauge field)
hr_status link_deriv(hr_ctx *ctx, hr_lattice lat, const void *gauge, const void *a_even, const void *a_odd,
                     const void *b_even, const void *b_odd, double beta, double *out, int mode, cudaStream_t s);

// ---- clover site term (hr_clover.cu) ----
// bytes of one of the four half-fields of a packed clover field (cp: kF64 / kF32)
size_t clover_half_bytes(const Geom &g, int rep, int cp);
// the half-field of A (inverse = false) or A^-1 on `parity`; nullptr for a null base
const void *clover_half(const void *base, const Geom &g, int rep, int cp, bool inverse, int parity);
// FP64 packed clover field -> FP32 packed clover field
hr_status clover_convert_f32(hr_ctx *ctx, const Geom &g, int rep, const void *src, void *dst, cudaStream_t s);
// out = A in on the sites of one parity, A from the half-field `half`
hr_status clover_apply_half(hr_ctx *ctx, const Geom &g, int rep, int prec, const void *half, const void *in,
                            void *out, cudaStream_t s);

// ---- BLAS launches (hr_blas.cu) ----
hr_status blas_norm2(hr_ctx *ctx, const Geom &g, int rep, int prec, const void *v, int fin, cudaStream_t s);
hr_status blas_p(hr_ctx *ctx, const Geom &g, int rep, int pp, int pr, void *p, const void *r, cudaStream_t s);
// the same after finishing the last hop's few rows (ctx->fin_rows) with the update `fin`
hr_status blas_p_fin(hr_ctx *ctx, const Geom &g, int rep, int prec, void *p, const void *r, int fin, const double *done,
                     FinCond cond, cudaStream_t s);
hr_status blas_convert(hr_ctx *ctx, const Geom &g, int rep, int psrc, int pdst, const void *src, void *dst,
                       const double *gate, cudaStream_t s);
// r = b - ax (FP64) with |r|^2 -> fin; also writes r in precision plo to r_lo when given
// r = b - ax (ax FP64, or FP32 with a binary16 r_lo; r nullable), |r|^2 -> fin, r_lo = r
hr_status blas_residual(hr_ctx *ctx, const Geom &g, int rep, const void *b, const void *ax, void *r, int fin,
                        const double *gate, int plo, void *r_lo, cudaStream_t s, int pax = kF64);
// packed FP64 gauge -> packed gauge of precision pdst (same rep)
hr_status gauge_convert(hr_ctx *ctx, const Geom &g, int rep, int pdst, const void *src, void *dst, cudaStream_t s);
// x_hi (FP64, or FP32) += x_lo (FP32); x_lo = 0
hr_status blas_accum(hr_ctx *ctx, const Geom &g, int rep, int plo, void *xhi, void *xlo, const double *gate,
                     cudaStream_t s, int phi = kF64);
hr_status blas_axpy(hr_ctx *ctx, const Geom &g, int rep, double a, const void *x, void *y, cudaStream_t s);
hr_status blas_gamma5(hr_ctx *ctx, const Geom &g, int rep, void *v, cudaStream_t s);
hr_status blas_zero(hr_ctx *ctx, const Geom &g, int rep, int prec, void *v, cudaStream_t s);
hr_status blas_copy(hr_ctx *ctx, const Geom &g, int rep, int prec, const void *src, void *dst, cudaStream_t s);
// per-RHS max |component| of a packed FP64 field -> scal[S_BMAX] (float bits; the slot must start at zero),
// then scal[S_SCALE] = the power of two that maps it into [0.5, 1) (1 for a zero field) and the F_RANGE
// flag when a nonzero maximum lies below 2^-100
hr_status blas_source_scale(hr_ctx *ctx, const Geom &g, int rep, const void *v, cudaStream_t s);
// dst = scal[S_SCALE] src per RHS (inverse: src / scale) on packed FP64 fields (dst may be src)
hr_status blas_scale(hr_ctx *ctx, const Geom &g, int rep, const void *src, void *dst, int inverse, cudaStream_t s);

// the pack status word (kPack* flags) since the last call, synchronising the
// stream; cleared.  HR_ERR_NUMERIC / HR_ERR_UNSUPPORTED with a message if set.
hr_status consume_pack_status(hr_ctx *ctx, cudaStream_t s);

} // namespace hr
