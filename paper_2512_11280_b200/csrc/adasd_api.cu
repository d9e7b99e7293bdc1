// C ABI of the AdaSD hot path (see include/adasd.h): context management, argument
// validation and kernel launches.  No torch types, no CPU fallback: without a CUDA
// device every call fails with ADASD_ERR_CUDA.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <type_traits>

#include "adasd_rows.cuh"
#include "adasd_cluster.cuh"
#include "adasd_spec.cuh"
#include "adasd_sweep.cuh"
#include "adasd_verify_tail.cuh"
#include "adasd_draft_stream.cuh"
#include "adasd_stream.cuh"
#include "adasd_topk.cuh"
#include "adasd_modes.cuh"

using namespace adasd;

struct adasd_ctx {
    adasd_config cfg;
    State st;
    Scratch sc;
    void* arena;              // the one device allocation, which every array of the context is a part of
    int sm_count;
    // warp-specialised verification kernel; iter == 0 means not usable for this V / dtype
    struct Fast {
        int iter;             // iterations per warp and row (template parameter)
        int cs;               // CTAs per cluster
        int smem;             // dynamic shared memory per CTA
        ClusterGeom geom;
    } fast;
    int draft_p, draft_nw, draft_it;      // draft step: CTAs per row, warps per CTA, iterations of a chunk
    bool draft_early;         // ... the next call's CTAs may be set up while one runs
    SweepTables sweep;        // verification of other rows: tables, segments
    bool cut_hist;            // the one-pass cutoff kernel got its 128 KB of shared memory
    // adjusted distribution (adasd_set_warpers) and the per-row cutoffs a call works out
    float temperature;
    int32_t top_k;
    float top_p;
    float* cut_t;             // [B,Kmax+1]
    float* cut_d;             // [B,Kmax]
    float* cut_row;           // [B] draft step
    float4* seg;              // [B (2 Kmax + 1)][2^seg_bits]: row statistics of the vanilla and greedy modes by segment
    uint32_t* stream_next;    // items its warps have drawn (0 between launches)
    int seg_bits, stream_it;  // ... of which there are 2^seg_bits; iterations of a chunk
    bool cuts_on() const { return (top_k > 0 && top_k < cfg.V) || top_p < 1.f; }
    bool warp_on() const { return cuts_on() || temperature != 1.f; }
    // The two kernels of aligned bf16 rows hold shifts and 2^t t in units of 1 / T: below this temperature a shift is off by
    // whole powers of two (logits of 10: by 8), below 4e-9 that of a masked logit overflows.  The general kernels, 7 and
    // 15 % slower on such rows, work on differences of logits.
    bool tiny_temperature() const { return temperature < 1e-6f; }
};

namespace {

#define CUDA_TRY(expr)                         \
    do {                                       \
        cudaError_t e__ = (expr);              \
        if (e__ != cudaSuccess) return ADASD_ERR_CUDA; \
    } while (0)

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

inline size_t elt_size(int dtype) { return dtype == ADASD_BF16 ? 2 : 4; }

// NULL counts as aligned: whether a pointer may be NULL is checked where it is used.
inline bool aligned_to(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }
inline bool aligned4(std::initializer_list<const void*> ps) {
    for (const void* p : ps)
        if (!aligned_to(p, 4)) return false;
    return true;
}

// The hot calls launch on the calling thread's current device with this context's pointers:
// refuse when that is another GPU.
int check_device(const adasd_ctx* c) {
    int cur = -1;
    if (cudaGetDevice(&cur) != cudaSuccess) {
        cudaGetLastError();
        return ADASD_ERR_CUDA;
    }
    return cur == c->cfg.device ? ADASD_OK : ADASD_ERR_DEVICE;
}

// Rows can take 16-byte loads when the base and every stride are 16-byte multiples.
inline bool vec_ok(const void* base, int dtype, std::initializer_list<long long> strides) {
    if (!aligned16(base)) return false;
    for (long long s : strides)
        if ((s * (long long)elt_size(dtype)) % 16 != 0) return false;
    return true;
}

template <typename P>
int launch_cluster(void (*kernel)(P), const P& params, long long clusters, int cs,
                   cudaStream_t stream) {
    cudaLaunchConfig_t lc;
    memset(&lc, 0, sizeof(lc));
    lc.gridDim = dim3((unsigned)(clusters * cs), 1, 1);
    lc.blockDim = dim3(kThreads, 1, 1);
    lc.dynamicSmemBytes = 0;
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    CUDA_TRY(cudaLaunchKernelEx(&lc, kernel, params));
    return ADASD_OK;
}

// ---- warp-specialised verification kernel: configuration and launch ----------------------
template <typename K>
int kernel_occupancy(K kern, int threads, int cs, int smem) {
    cudaLaunchConfig_t lc;
    memset(&lc, 0, sizeof(lc));
    lc.gridDim = dim3((unsigned)(cs * 64), 1, 1);
    lc.blockDim = dim3((unsigned)threads, 1, 1);
    lc.dynamicSmemBytes = (size_t)smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &lc) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

template <typename K>
int kernel_static_smem(K kern) {
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess) {
        cudaGetLastError();
        return -1;
    }
    return (int)fa.sharedSizeBytes;
}

// The limit on dynamic shared memory is one value per function and device, not per context: it is set to the
// most any vocabulary of this ITER can ask for, so that no context lowers it under another's launches.
template <int ITER, bool WARPED>
cudaError_t fast_allow(int smem_optin) {
    const int st = kernel_static_smem(spec_verify_kernel<ITER, WARPED>);
    if (st < 0) return cudaErrorInvalidDeviceFunction;
    return cudaFuncSetAttribute(spec_verify_kernel<ITER, WARPED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                std::min(kSW * ITER * kSIterBytes, smem_optin - st));
}
template <int ITER>
int fast_occupancy(int cs, int smem, int smem_optin) {
    if (fast_allow<ITER, false>(smem_optin) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return kernel_occupancy(spec_verify_kernel<ITER>, kSThreads, cs, smem);
}
template <int ITER>
int fast_static_smem() {
    return kernel_static_smem(spec_verify_kernel<ITER>);
}

#define ADASD_ITER_SWITCH(iter, CALL, fail)  \
    switch (iter) {                          \
        case 1: return CALL(1);              \
        case 2: return CALL(2);              \
        case 3: return CALL(3);              \
        case 4: return CALL(4);              \
        case 5: return CALL(5);              \
        case 6: return CALL(6);              \
        case 7: return CALL(7);              \
        case 8: return CALL(8);              \
        case 9: return CALL(9);              \
        case 10: return CALL(10);            \
        default: return fail;                \
    }

int fast_occupancy_iter(int iter, int cs, int smem, int smem_optin) {
#define CALL(I) fast_occupancy<I>(cs, smem, smem_optin)
    ADASD_ITER_SWITCH(iter, CALL, 0)
#undef CALL
}
cudaError_t fast_allow_warped_iter(int iter, int smem_optin) {
#define CALL(I) fast_allow<I, true>(smem_optin)
    ADASD_ITER_SWITCH(iter, CALL, cudaErrorInvalidValue)
#undef CALL
}
int fast_static_smem_iter(int iter) {
#define CALL(I) fast_static_smem<I>()
    ADASD_ITER_SWITCH(iter, CALL, -1)
#undef CALL
}

// Verification kernel of aligned bf16 rows: chooses the cluster size that covers the most SMs among those whose per-CTA
// slice fits on chip: two position buffers per compute warp, iter * 512 bytes per row (the
// 2^t values live in registers or are worked out again).  bf16 rows of a multiple of 8
// elements only.
void fast_setup(adasd_ctx* c, size_t smem_optin) {
    adasd_ctx::Fast& f = c->fast;
    f.iter = 0;
    const int V = c->cfg.V;
    if (c->cfg.dtype != ADASD_BF16 || (V & 7) != 0 || V < 8192) return;
    const int NU = V >> 3;
    int best_score = 0;
    for (int cs = kCMaxCluster; cs >= 1; --cs) {
        if (c->cfg.cluster_size != 0 && c->cfg.cluster_size != cs) continue;
        const int ncu = (NU + cs - 1) / cs, nwi = (ncu + 31) / 32;
        const int I_lo = nwi / kSW, rem = nwi % kSW, iter = I_lo + (rem ? 1 : 0);
        if (iter < 1 || iter > kSMaxIter) continue;
        const int st = fast_static_smem_iter(iter);
        if (st < 0) continue;
        const int smem = nwi * kSIterBytes;
        if (smem > (int)smem_optin - st - 1024) continue;
        const int ncl = fast_occupancy_iter(iter, cs, smem, (int)smem_optin);
        const int score = ncl * cs;
        if (score > best_score) {
            best_score = score;
            f.iter = iter;
            f.cs = cs;
            f.smem = smem;
            f.geom.ncl = ncl;
        }
    }
    if (f.iter > 0 && fast_allow_warped_iter(f.iter, (int)smem_optin) != cudaSuccess) {
        cudaGetLastError();
        f.iter = 0;
    }
}
void cutoff_setup(adasd_ctx* c) {
    c->cut_hist = cudaFuncSetAttribute(row_cutoff_hist_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kHistWords * 4) == cudaSuccess;
    if (!c->cut_hist) cudaGetLastError();
}

// Chunk length and segments of a row in the vanilla and greedy modes.
// Chunks of 8 iterations (4 KB) cost a warp 0.42 us, of 2 iterations 0.33: the short ones only where a row does
// not fill a long one, or where segments of long ones would be so few that shorter ones spread the launch over
// more warps: less than one for four warps (vanilla, bf16 V=8200 B=8 K=5, 352 of them: 10.0 us with short chunks, 10.5
// with long ones; V=16384, 704: 10.6 and 9.4), five where a row is a single chunk (greedy, fp32 V=1000 B=64 K=4, 576:
// 5.4 and 4.7).
// Segments: with four chunks or more for every warp of the grid, at least two chunks each while that gives the
// warps six items each (half as long measured 33 instead of 31.8 us on 544 rows of 128256); with fewer long
// chunks, as many as leave every warp with one item at most (greedy, 512 rows of 8200 bf16, 1024 / 2048 / 4096
// items: 7.2 / 7.8 / 9.5 us); short chunks: an item for every warp at least.
void stream_setup(adasd_ctx* c) {
    const int N = c->cfg.dtype == ADASD_BF16 ? 8 : 4, NU = (c->cfg.V + N - 1) / N;
    const long long rows = (long long)c->cfg.B * (2 * c->cfg.Kmax + 1), warps = 2LL * c->sm_count * kRW;
    const int nc8 = (NU + 255) / 256;
    long long items8 = rows;
    for (int k = 2; k <= std::min(kMaxSegs, nc8); k *= 2) items8 *= 2;
    c->stream_it = NU >= 224 && items8 * (nc8 == 1 ? 5 : 4) >= warps ? 8 : 2;
    const int NC = c->stream_it == 8 ? nc8 : (NU + 63) / 64;
    auto more = [&](int bits) -> bool {
        const long long items = rows << bits;
        if (c->stream_it == 8 && rows * nc8 < 4 * warps) return items * 2 <= warps;
        return items < warps || (items < 6 * warps && (NC >> bits) >= 4);
    };
    int bits = 0;
    while ((2 << bits) <= std::min(kMaxSegs, NC) && more(bits)) ++bits;
    c->seg_bits = bits;
}

template <typename T, bool ALIGNED, int IT>
cudaError_t stream_prepare_it() {
    cudaError_t e = cudaFuncSetAttribute(row_stream_kernel<T, ALIGNED, OP_LSE, false, IT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(row_stream_kernel<T, ALIGNED, OP_LSE, true, IT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(row_stream_kernel<T, ALIGNED, OP_ARGMAX, false, IT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRSmem);
    return e;
}
template <typename T, bool ALIGNED>
cudaError_t stream_prepare(int it) { return it == 8 ? stream_prepare_it<T, ALIGNED, 8>() : stream_prepare_it<T, ALIGNED, 2>(); }

// early: launch with programmatic stream serialisation: the kernel may become resident while the one ahead of
// it is still running (it waits before it reads what that one wrote).  cs: CTAs per cluster; 0: the kernel
// uses no cluster.  (A kernel that uses cluster-scope instructions gets the attribute even for clusters of one.)
template <typename K, typename... Args>
int launch_kernel(bool early, K kernel, int grid, int threads, int smem, int cs, cudaStream_t stream, const Args&... args) {
    cudaLaunchConfig_t lc;
    memset(&lc, 0, sizeof(lc));
    lc.gridDim = dim3((unsigned)grid, 1, 1);
    lc.blockDim = dim3((unsigned)threads, 1, 1);
    lc.dynamicSmemBytes = (size_t)smem;
    lc.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = early ? 1 : 0;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cs;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = cs > 0 ? 2 : 1;
    CUDA_TRY(cudaLaunchKernelEx(&lc, kernel, args...));
    return ADASD_OK;
}
template <typename K, typename... Args>
int launch_pdl(K kernel, int grid, int threads, int smem, int cs, cudaStream_t stream, const Args&... args) {
    return launch_kernel(true, kernel, grid, threads, smem, cs, stream, args...);
}

template <typename T, bool ALIGNED, int IT>
int launch_stream_it(adasd_ctx* c, const StreamParams& p, int op, cudaStream_t stream) {
    const long long rows = (long long)p.B * (p.zd ? 2 * p.Kmax + 1 : p.Kmax + 1);
    const int grid = (int)std::min<long long>(((rows << p.seg_bits) + kRW - 1) / kRW, 2LL * c->sm_count);
    if (op == OP_ARGMAX) return launch_pdl(row_stream_kernel<T, ALIGNED, OP_ARGMAX, false, IT>, grid, kRThreads, kRSmem, 0, stream, p);
    return c->warp_on() ? launch_pdl(row_stream_kernel<T, ALIGNED, OP_LSE, true, IT>, grid, kRThreads, kRSmem, 0, stream, p)
                        : launch_pdl(row_stream_kernel<T, ALIGNED, OP_LSE, false, IT>, grid, kRThreads, kRSmem, 0, stream, p);
}
template <typename T, bool ALIGNED>
int launch_stream(adasd_ctx* c, const StreamParams& p, int op, cudaStream_t stream) {
    return c->stream_it == 8 ? launch_stream_it<T, ALIGNED, 8>(c, p, op, stream) : launch_stream_it<T, ALIGNED, 2>(c, p, op, stream);
}
int launch_stream(adasd_ctx* c, const StreamParams& p, int op, bool aligned, cudaStream_t stream) {
    if (c->cfg.dtype == ADASD_BF16)
        return aligned ? launch_stream<__nv_bfloat16, true>(c, p, op, stream) : launch_stream<__nv_bfloat16, false>(c, p, op, stream);
    return aligned ? launch_stream<float, true>(c, p, op, stream) : launch_stream<float, false>(c, p, op, stream);
}

// ---- draft step: configuration and launch -----------------------------------------------------
// CTAs per row until they cover three quarters of the SMs.  16 warps per CTA, one CTA per SM, where that
// takes all of a call's CTAs at once (clusters of 4: 33 fit, of 8: 15); else 8 warps and two CTAs per SM.
void draft_setup(adasd_ctx* c) {
    int P = 1;
    if (c->cfg.cluster_size == 1 || c->cfg.cluster_size == 2 || c->cfg.cluster_size == 4 || c->cfg.cluster_size == 8)
        P = c->cfg.cluster_size;
    else
        while (P < kDMaxP && (long long)c->cfg.B * P * 4 < 3LL * c->sm_count) P *= 2;
    c->draft_p = P;
    const long long grid = (long long)c->cfg.B * P;
    c->draft_nw = P <= 4 && grid <= (P == 4 ? 132 : c->sm_count) ? kDWBig : kDW;
    // dependents early: where the SMs hold two CTAs and a call needs at most half of them, or where they hold one
    c->draft_early = c->draft_nw == kDWBig || grid * 2 <= c->sm_count;
    const int N = c->cfg.dtype == ADASD_BF16 ? 8 : 4, NI = ((c->cfg.V + N - 1) / N + 31) / 32;
    c->draft_it = NI >= 16 * P * c->draft_nw ? 8 : 4;
}
// Large batches of aligned bf16 rows: the kernel whose warps split a row to 16 bytes.
bool draft_rows(const adasd_ctx* c) {
    return c->cfg.dtype == ADASD_BF16 && (c->cfg.V & 7) == 0 && c->cfg.V >= 8192 && c->draft_p <= 2 && !c->tiny_temperature() &&
           c->cfg.V <= kDMaxChunks * kDChunkUnits * 8 * c->draft_p * c->draft_nw;
}
template <int NW>
cudaError_t draft_rows_prepare() {
    cudaError_t e = cudaFuncSetAttribute(draft_stream_kernel<NW, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, NW * 2 * kDChunkBytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(draft_stream_kernel<NW, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, NW * 2 * kDChunkBytes);
    return e;
}
template <int NW>
int launch_draft_rows(adasd_ctx* c, const DraftParams& p, cudaStream_t stream) {
    const int grid = p.B * c->draft_p, smem = NW * 2 * kDChunkBytes;
    return c->warp_on() ? launch_pdl(draft_stream_kernel<NW, true>, grid, NW * 32, smem, c->draft_p, stream, p)
                        : launch_pdl(draft_stream_kernel<NW, false>, grid, NW * 32, smem, c->draft_p, stream, p);
}

template <typename T, bool ALIGNED, int NW, int IT>
cudaError_t draft_prepare_it() {
    cudaError_t e = cudaFuncSetAttribute(draft_step_kernel<T, ALIGNED, NW, IT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, NW * kDRingB);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(draft_step_kernel<T, ALIGNED, NW, IT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, NW * kDRingB);
    return e;
}
template <typename T, bool ALIGNED>
cudaError_t draft_prepare(const adasd_ctx* c) {
    if (c->draft_nw == kDW) return c->draft_it == 8 ? draft_prepare_it<T, ALIGNED, kDW, 8>() : draft_prepare_it<T, ALIGNED, kDW, 4>();
    return c->draft_it == 8 ? draft_prepare_it<T, ALIGNED, kDWBig, 8>() : draft_prepare_it<T, ALIGNED, kDWBig, 4>();
}
template <typename T, bool ALIGNED, int NW, int IT>
int launch_draft_it(adasd_ctx* c, const DraftParams& p, cudaStream_t stream) {
    const int grid = p.B * c->draft_p;
    return c->warp_on() ? launch_pdl(draft_step_kernel<T, ALIGNED, NW, IT, true>, grid, NW * 32, NW * kDRingB, c->draft_p, stream, p)
                        : launch_pdl(draft_step_kernel<T, ALIGNED, NW, IT, false>, grid, NW * 32, NW * kDRingB, c->draft_p, stream, p);
}
template <typename T, bool ALIGNED>
int launch_draft(adasd_ctx* c, const DraftParams& p, cudaStream_t stream) {
    if (c->draft_nw == kDW)
        return c->draft_it == 8 ? launch_draft_it<T, ALIGNED, kDW, 8>(c, p, stream) : launch_draft_it<T, ALIGNED, kDW, 4>(c, p, stream);
    return c->draft_it == 8 ? launch_draft_it<T, ALIGNED, kDWBig, 8>(c, p, stream) : launch_draft_it<T, ALIGNED, kDWBig, 4>(c, p, stream);
}
template <typename T>
int launch_draft(adasd_ctx* c, const DraftParams& p, bool aligned, cudaStream_t stream) {
    return aligned ? launch_draft<T, true>(c, p, stream) : launch_draft<T, false>(c, p, stream);
}

template <int ITER, bool WARPED>
int fast_launch(adasd_ctx* c, const VerifyParams& p, cudaStream_t stream) {
    const long long positions = (long long)p.B * (p.Kmax + 1);
    const adasd_ctx::Fast& f = c->fast;
    ClusterGeom gq = f.geom;
    if (positions < gq.ncl) gq.ncl = (int)positions;
    return launch_pdl(spec_verify_kernel<ITER, WARPED>, gq.ncl * f.cs, kSThreads, f.smem, f.cs, stream, p, gq);
}

int fast_launch_iter(adasd_ctx* c, const VerifyParams& p, cudaStream_t stream) {
    if (c->warp_on()) {
#define CALL(I) fast_launch<I, true>(c, p, stream)
        ADASD_ITER_SWITCH(c->fast.iter, CALL, ADASD_ERR_SHAPE)
#undef CALL
    }
#define CALL(I) fast_launch<I, false>(c, p, stream)
    ADASD_ITER_SWITCH(c->fast.iter, CALL, ADASD_ERR_SHAPE)
#undef CALL
}

int check_strides(const adasd_ctx* c, long long seq, long long row) {
    if (row < c->cfg.V || seq < 0) return ADASD_ERR_SHAPE;
    return ADASD_OK;
}

int fill_verify_params(adasd_ctx* ctx, VerifyParams& p, const void* zd, const void* zt,
                       int64_t d_seq, int64_t d_row, int64_t t_seq, int64_t t_row,
                       const int32_t* x, const int32_t* draft_len) {
    if (!ctx || !zd || !zt || !x) return ADASD_ERR_NULL;
    int rc;
    if ((rc = check_device(ctx)) != ADASD_OK) return rc;
    const size_t es = elt_size(ctx->cfg.dtype);
    if (!aligned_to(zd, es) || !aligned_to(zt, es) || !aligned4({x, draft_len})) return ADASD_ERR_ALIGN;
    if ((rc = check_strides(ctx, d_seq, d_row)) != ADASD_OK) return rc;
    if ((rc = check_strides(ctx, t_seq, t_row)) != ADASD_OK) return rc;
    memset(&p, 0, sizeof(p));
    p.zd = zd;
    p.zt = zt;
    p.d_seq = d_seq;
    p.d_row = d_row;
    p.t_seq = t_seq;
    p.t_row = t_row;
    p.x = x;
    p.draft_len = draft_len;
    p.sc = ctx->sc;
    p.st = ctx->st;
    p.B = ctx->cfg.B;
    p.V = ctx->cfg.V;
    p.Kmax = ctx->cfg.Kmax;
    p.inv_temp = 1.f / ctx->temperature;
    p.c1 = kLog2e / ctx->temperature;
    if (ctx->cuts_on()) {
        p.cut_t = ctx->cut_t;
        p.cut_d = ctx->cut_d;
    }
    return ADASD_OK;
}

// One cutoff logit per needed row (top-k / top-p of the adjusted distribution) of one or two arrays of rows.
CutParams cut_params(const adasd_ctx* ctx, const void* z, long long seq_stride, long long row_stride, int R, int extra,
                     const int32_t* draft_len, const uint8_t* active, float* cut) {
    CutParams c;
    memset(&c, 0, sizeof(c));
    c.z = z;
    c.seq_stride = seq_stride;
    c.row_stride = row_stride;
    c.draft_len = draft_len;
    c.active = active;
    c.cut = cut;
    c.status = ctx->st.status;
    c.B = ctx->cfg.B;
    c.R = R;
    c.V = ctx->cfg.V;
    c.extra = extra;
    c.c1 = 1.4426950408889634 / (double)ctx->temperature;
    c.top_k = ctx->top_k;
    c.top_p = ctx->top_p;
    return c;
}
int launch_cutoffs(adasd_ctx* ctx, CutParams c, const CutParams* second, cudaStream_t stream) {
    const bool bf = ctx->cfg.dtype == ADASD_BF16;
    const bool vec1 = vec_ok(c.z, ctx->cfg.dtype, {c.seq_stride, c.row_stride});
    const bool vec2 = !second || vec_ok(second->z, ctx->cfg.dtype, {second->seq_stride, second->row_stride});
    CutParams c2 = second ? *second : c;
    const long long rows = (long long)c.B * (c.R + (second ? second->R : 0));
    // top-k on: selection, a row over as many CTAs as are resident at once; it flags what it cannot do
    int P = 1;
    while (P < kSelMaxP && rows * P * 2 <= 3LL * ctx->sm_count) P *= 2;
    // ... up to a k where it is the faster one.  It compares its candidates, a few times k, with one another; the histogram of
    // aligned bf16 rows depends little on k, but takes a CTA a row and a launch an array.  Selection / histogram, us a call,
    // temperature 0.8, rows of s N(0, 1) - ln(rank), inputs beyond L2:
    // - a top-p cut behind it, draft calls: V=128256, 32 rows, k=200 41 / 46; V=32000, 8 rows k=200 28 / 34, 32 rows k=100
    //   28 / 34 and k=200 37 / 36, 256 rows k=200 46 / 67 (the worst: V=8192, 111 rows, k=200 41 / 36);
    // - verification of 16 sequences, K=5: V=32000, with top-p k=200 59 / 84, without it k=64 42 / 50;
    // - draft calls without top-p, where the histogram is a count: V=128256, 32 rows k=100 27 / 30, 256 rows k=100 54 / 62;
    //   V=32000, 8 rows k=64 18 / 18, 256 rows k=64 29 / 35.  Here the limits are beyond the crossing while the histogram is
    //   one wave of more than 16 rows: V=8192, 55 rows, k=40 24 / 17; V=32000, 32 rows, k=40 23 / 19; V=128256, 111 rows,
    //   k=200 47 / 36.  A line through that range is not drawn yet.
    // Up to 200 the candidates fit the list even of a row sorted by its logits, which has the most (five times k); such rows
    // lose (2 N(0, 1), V=32000, 8 rows, top-p, k=64 32 / 31, k=200 124 / 32).  Against the radix descent: always, unless the
    // few groups of a row with one CTA leave so many candidates that it hands rows over (the same, 256 fp32 rows, not sorted,
    // k=400 114 / 221, k=448 140 / 222, k=512 293 / 225).
    const bool histogram = bf && vec1 && vec2 && ctx->cut_hist;
    const int k_most = !histogram ? std::min(kSelMaxK, 448 * P) : c.V >= 65536 || c.top_p < 1.f || P == 1 ? 200 : 64;
    const bool select = c.top_k > 0 && c.top_k < c.V && c.top_k <= k_most && c.V >= kSelMinV && rows <= 0x7FFFFFFF / kSelMaxP;
    if (select) {
        const int g = (int)(rows * P);
        const bool aligned = vec1 && vec2;
        int rc;
        if (bf)
            rc = aligned ? launch_pdl(row_cutoff_select_kernel<__nv_bfloat16, true>, g, kSelThreads, 0, P, stream, c, c2)
                         : launch_pdl(row_cutoff_select_kernel<__nv_bfloat16, false>, g, kSelThreads, 0, P, stream, c, c2);
        else
            rc = aligned ? launch_pdl(row_cutoff_select_kernel<float, true>, g, kSelThreads, 0, P, stream, c, c2)
                         : launch_pdl(row_cutoff_select_kernel<float, false>, g, kSelThreads, 0, P, stream, c, c2);
        if (rc != ADASD_OK) return rc;
    }
    for (int k = 0; k < (second ? 2 : 1); ++k) {
        CutParams& q = k ? c2 : c;
        const bool vec = k ? vec2 : vec1;
        const long long n = (long long)q.B * q.R;
        q.only_flagged = select ? 1 : 0;
        if (!select && bf && vec && ctx->cut_hist) {
            // one pass per row over a histogram of the 65536 bf16 values; a row it cannot do (a value
            // that occurs 65536 times or more) is left flagged for the radix kernel
            row_cutoff_hist_kernel<<<(unsigned)std::min<long long>(n, (long long)ctx->sm_count), kHistThreads, kHistWords * 4, stream>>>(q);
            CUDA_TRY(cudaGetLastError());
            q.only_flagged = 1;
        }
        const int grid = (int)std::min<long long>(n, 2LL * ctx->sm_count);
        // (early only where it has next to nothing to do: 64 rows of 128256 fp32 logits took 904 instead of 400 us, packed on the
        // SMs beside the draft step ahead)
        const bool early = q.only_flagged != 0;
        int rc;
        if (bf)
            rc = vec ? launch_kernel(early, row_cutoff_kernel<__nv_bfloat16, true>, grid, kCutThreads, 0, 0, stream, q)
                     : launch_kernel(early, row_cutoff_kernel<__nv_bfloat16, false>, grid, kCutThreads, 0, 0, stream, q);
        else
            rc = vec ? launch_kernel(early, row_cutoff_kernel<float, true>, grid, kCutThreads, 0, 0, stream, q)
                     : launch_kernel(early, row_cutoff_kernel<float, false>, grid, kCutThreads, 0, 0, stream, q);
        if (rc != ADASD_OK) return rc;
    }
    return ADASD_OK;
}
// ... of the rows of a verification round
int launch_round_cutoffs(adasd_ctx* ctx, const VerifyParams& p, cudaStream_t stream) {
    if (!ctx->cuts_on()) return ADASD_OK;
    const CutParams d = cut_params(ctx, p.zd, p.d_seq, p.d_row, p.Kmax, 0, p.draft_len, nullptr, ctx->cut_d);
    return launch_cutoffs(ctx, cut_params(ctx, p.zt, p.t_seq, p.t_row, p.Kmax + 1, 1, p.draft_len, nullptr, ctx->cut_t), &d, stream);
}

// ---- verification of rows the warp-specialised kernel does not take ---------------------------
// Segments of a position: as many as make the most loaded warp of a grid that fills the chip take the fewest
// chunks, an item (its description, the folding of statistics, a drained ring) counting as two chunks more.
void sweep_setup(adasd_ctx* c) {
    const int N = c->cfg.dtype == ADASD_BF16 ? 8 : 4;
    const int NC = ((c->cfg.V + N - 1) / N + 32 * kSweepIt - 1) / (32 * kSweepIt);
    const long long P = (long long)c->cfg.B * (c->cfg.Kmax + 1), warps = 2LL * c->sm_count * kSweepW;
    long long best = 0;
    for (int segs = 1; segs <= std::min(NC, kSweepMaxSegs) && P * segs < 0x40000000LL; ++segs) {
        const long long load = ((P * segs + warps - 1) / warps) * ((NC + segs - 1) / segs + 2);
        if (segs == 1 || load < best) {
            best = load;
            c->sweep.segs = segs;
        }
    }
}
template <typename T, bool ALIGNED>
cudaError_t sweep_prepare() {
    cudaError_t e = cudaFuncSetAttribute(sweep_kernel<T, ALIGNED, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSweepSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(sweep_kernel<T, ALIGNED, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSweepSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(sweep_kernel<T, ALIGNED, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSweepSmem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(sweep_kernel<T, ALIGNED, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSweepSmem);
    return e;
}
template <typename T, bool ALIGNED, bool WARPED>
int launch_sweep(adasd_ctx* c, const VerifyParams& p, cudaStream_t stream) {
    const long long items = (long long)p.B * (p.Kmax + 1) * c->sweep.segs;
    const int grid = (int)std::min<long long>(items, 2LL * c->sm_count);
    if (int rc = launch_pdl(sweep_kernel<T, ALIGNED, WARPED, false>, grid, kSweepThreads, kSweepSmem, 0, stream, p, c->sweep)) return rc;
    return launch_pdl(sweep_kernel<T, ALIGNED, WARPED, true>, grid, kSweepThreads, kSweepSmem, 0, stream, p, c->sweep);
}
template <typename T>
int launch_sweep(adasd_ctx* c, const VerifyParams& p, bool aligned, cudaStream_t stream) {
    if (aligned) return c->warp_on() ? launch_sweep<T, true, true>(c, p, stream) : launch_sweep<T, true, false>(c, p, stream);
    return c->warp_on() ? launch_sweep<T, false, true>(c, p, stream) : launch_sweep<T, false, false>(c, p, stream);
}

int launch_verify(adasd_ctx* ctx, const VerifyParams& p, cudaStream_t stream) {
    const bool vec = vec_ok(p.zd, ctx->cfg.dtype, {p.d_seq, p.d_row}) &&
                     vec_ok(p.zt, ctx->cfg.dtype, {p.t_seq, p.t_row});
    if (int rc = launch_round_cutoffs(ctx, p, stream)) return rc;
    if (vec && ctx->fast.iter > 0 && !ctx->tiny_temperature()) return fast_launch_iter(ctx, p, stream);
    return ctx->cfg.dtype == ADASD_BF16 ? launch_sweep<__nv_bfloat16>(ctx, p, vec, stream) : launch_sweep<float>(ctx, p, vec, stream);
}

// CTAs per sequence of the tail kernel: a list entry costs every candidate one exponential, so a
// sequence whose lists can hold more than a few entries per thread gets more threads, as long as the
// sequences leave room for them.
int tail_cluster(const adasd_ctx* c) {
    int S = 1;
    while (S < kTailMaxS && (long long)c->cfg.list_capacity > 4LL * kTailThreads * S &&
           (long long)c->cfg.B * S * 2 <= 4LL * c->sm_count)
        S *= 2;
    return S;
}

struct DeviceGuard {
    int prev = -1;
    bool ok = false;
    explicit DeviceGuard(int dev) {
        if (cudaGetDevice(&prev) != cudaSuccess) return;
        ok = (prev == dev) || (cudaSetDevice(dev) == cudaSuccess);
    }
    ~DeviceGuard() {
        if (ok && prev >= 0) {
            int cur = -1;
            if (cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
        }
    }
};

constexpr size_t kExportHeader = 24;

}  // namespace

// ---- allocation-free vanilla verification -------------------------------------------
// Scratch of adasd_vanilla_verify_static: lives in the library image, one copy per GPU
// that loads it, shared by every call.  Words: per-candidate accept flags, per-position
// candidate tokens, per-sequence arrival counters, one status word.
static __device__ __align__(256) uint32_t g_static_scratch[2 * ADASD_STATIC_MAX_POSITIONS +
                                                           ADASD_STATIC_MAX_B + 64];

namespace {
constexpr int kMaxDevices = 64;
struct StaticSetup {
    uint32_t* base = nullptr;   // device address of g_static_scratch on this device
    int sm_count = 0;
};
StaticSetup g_static_setup[kMaxDevices];
std::mutex g_static_mutex;

// Device address of the scratch array on the CURRENT device.  The array's name is only a
// host-side handle: the address a kernel can use comes from cudaGetSymbolAddress, asked
// once per device with that device current.
int static_setup(int dev, StaticSetup& out) {
    std::lock_guard<std::mutex> lock(g_static_mutex);
    StaticSetup& s = g_static_setup[dev];
    if (!s.base) {
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || !ptr) {
            cudaGetLastError();
            return ADASD_ERR_CUDA;
        }
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            return ADASD_ERR_CUDA;
        }
        s.sm_count = sms;
        s.base = static_cast<uint32_t*>(ptr);
    }
    out = s;
    return ADASD_OK;
}
}  // namespace

extern "C" {

int adasd_create(adasd_ctx** out, const adasd_config* cfg) {
    if (!out || !cfg) return ADASD_ERR_NULL;
    *out = nullptr;
    if (cfg->B < 1 || cfg->V < 1 || cfg->Kmax < 1 || cfg->Kmax > ADASD_KMAX_LIMIT ||
        cfg->list_capacity < 1)
        return ADASD_ERR_SHAPE;
    if ((long long)cfg->B * (cfg->Kmax + 1) > 0x3FFFFFFFLL) return ADASD_ERR_SHAPE;
    if (cfg->dtype != ADASD_BF16 && cfg->dtype != ADASD_FP32) return ADASD_ERR_DTYPE;
    if (cfg->kde_bandwidth < 0 || cfg->kde_bandwidth > 1 || cfg->reject_rule < 0 ||
        cfg->reject_rule > 1)
        return ADASD_ERR_DTYPE;
    if (cfg->cluster_size < 0 || cfg->cluster_size > kMaxCluster) return ADASD_ERR_SHAPE;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || cfg->device < 0 || cfg->device >= ndev)
        return ADASD_ERR_CUDA;
    DeviceGuard guard(cfg->device);
    if (!guard.ok) return ADASD_ERR_CUDA;

    adasd_ctx* c = new (std::nothrow) adasd_ctx();
    if (!c) return ADASD_ERR_CUDA;
    c->cfg = *cfg;
    if (c->cfg.min_kde_samples < 2) c->cfg.min_kde_samples = 2;
    // (two attributes: cudaGetDeviceProperties takes 2.7 ms, the rest of this function 0.2)
    int smem_optin = 0;
    if (cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, cfg->device) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, cfg->device) != cudaSuccess) {
        delete c;
        return ADASD_ERR_CUDA;
    }
    memset(&c->st, 0, sizeof(c->st));
    memset(&c->sc, 0, sizeof(c->sc));

    const size_t B = (size_t)cfg->B, K = (size_t)cfg->Kmax, cap = (size_t)cfg->list_capacity;
    int rc = ADASD_OK;
    State& s = c->st;
    Scratch& t = c->sc;
    s.cap = cfg->list_capacity;
    sweep_setup(c);
    stream_setup(c);
    // one zeroed allocation for all arrays: laid out once for its size, once at its address
    auto carve = [&](unsigned char* base) -> size_t {
        size_t at = 0;
        auto take = [&](auto*& ptr, size_t n) {
            ptr = reinterpret_cast<std::remove_reference_t<decltype(ptr)>>(base + at);
            at += (n * sizeof(*ptr) + 255) & ~(size_t)255;
        };
        take(s.T_G, B);
        take(s.sumE, B);
        take(s.nE, B);
        take(s.nA, B);
        take(s.nR, B);
        take(s.sumA, B);
        take(s.sumA2, B);
        take(s.sumR, B);
        take(s.sumR2, B);
        take(s.LE, B * cap);
        take(s.LA, B * cap);
        take(s.LR, B * cap);
        take(s.status, 1);
        take(t.H_d, B * K);
        take(t.dist, B * K);
        take(t.y, B * (K + 1));
        take(c->cut_t, B * (K + 1));
        take(c->cut_d, B * K);
        take(c->cut_row, B);
        take(c->stream_next, 1);
        take(c->sweep.seg1, B * (K + 1) * c->sweep.segs);
        take(c->sweep.seg2, B * (K + 1) * c->sweep.segs);
        take(c->sweep.done, B * (K + 1));
        take(c->sweep.next, 2);
        take(c->seg, (B * (2 * K + 1)) << c->seg_bits);
        return at;
    };
    const size_t arena_bytes = carve(nullptr);
    if (cudaMalloc(&c->arena, arena_bytes) != cudaSuccess) {
        cudaGetLastError();
        delete c;
        return ADASD_ERR_CUDA;
    }
    carve(static_cast<unsigned char*>(c->arena));
    if (cudaMemset(c->arena, 0, arena_bytes) != cudaSuccess) rc = ADASD_ERR_CUDA;
    c->temperature = 1.f;
    c->top_k = 0;
    c->top_p = 1.f;
    if (rc == ADASD_OK) {
        fast_setup(c, (size_t)smem_optin);
        cutoff_setup(c);
    }
    if (rc == ADASD_OK) {
        const cudaError_t e1 = cfg->dtype == ADASD_BF16 ? stream_prepare<__nv_bfloat16, true>(c->stream_it) : stream_prepare<float, true>(c->stream_it);
        const cudaError_t e2 = cfg->dtype == ADASD_BF16 ? stream_prepare<__nv_bfloat16, false>(c->stream_it) : stream_prepare<float, false>(c->stream_it);
        draft_setup(c);
        const cudaError_t e3 = cfg->dtype == ADASD_BF16 ? draft_prepare<__nv_bfloat16, true>(c) : draft_prepare<float, true>(c);
        const cudaError_t e4 = cfg->dtype == ADASD_BF16 ? draft_prepare<__nv_bfloat16, false>(c) : draft_prepare<float, false>(c);
        const cudaError_t e5 = c->draft_nw == kDW ? draft_rows_prepare<kDW>() : draft_rows_prepare<kDWBig>();
        const cudaError_t e6 = cfg->dtype == ADASD_BF16 ? sweep_prepare<__nv_bfloat16, true>() : sweep_prepare<float, true>();
        const cudaError_t e7 = cfg->dtype == ADASD_BF16 ? sweep_prepare<__nv_bfloat16, false>() : sweep_prepare<float, false>();
        if (e6 != cudaSuccess || e7 != cudaSuccess) rc = ADASD_ERR_CUDA;
        if (e1 != cudaSuccess || e2 != cudaSuccess || e3 != cudaSuccess || e4 != cudaSuccess || e5 != cudaSuccess) rc = ADASD_ERR_CUDA;
    }
    if (rc == ADASD_OK && cudaDeviceSynchronize() != cudaSuccess) rc = ADASD_ERR_CUDA;
    if (rc != ADASD_OK) {
        cudaFree(c->arena);
        delete c;
        return rc;
    }
    *out = c;
    return ADASD_OK;
}

int adasd_destroy(adasd_ctx* ctx) {
    if (!ctx) return ADASD_ERR_NULL;
    DeviceGuard guard(ctx->cfg.device);
    int rc = ADASD_OK;
    if (cudaDeviceSynchronize() != cudaSuccess) rc = ADASD_ERR_CUDA;
    if (cudaFree(ctx->arena) != cudaSuccess) rc = ADASD_ERR_CUDA;
    delete ctx;
    return rc;
}

int adasd_reset(adasd_ctx* ctx, const int32_t* seq_ids_dev, int32_t n, void* stream) {
    if (!ctx) return ADASD_ERR_NULL;
    if (int rc = check_device(ctx)) return rc;
    if (!aligned4({seq_ids_dev})) return ADASD_ERR_ALIGN;
    if (!seq_ids_dev) n = ctx->cfg.B;
    if (n < 0) return ADASD_ERR_SHAPE;
    if (n == 0) return ADASD_OK;
    reset_kernel<<<(n + 127) / 128, 128, 0, (cudaStream_t)stream>>>(ctx->st, seq_ids_dev, n,
                                                                    ctx->cfg.B);
    CUDA_TRY(cudaGetLastError());
    return ADASD_OK;
}

// adasd_draft_entropy, optionally (expire_row >= 0) as the self-test of the bounded waits
static int draft_entropy_impl(adasd_ctx* ctx, const void* logits_dev, int64_t row_stride,
                              const float* u_dev, uint8_t* active_inout_dev, float* H_out_dev,
                              float* lse_out_dev, int32_t* token_out_dev, uint8_t* stop_out_dev,
                              int32_t* draft_len_inout_dev, void* stream, int32_t expire_row) {
    if (!ctx || !logits_dev || !H_out_dev) return ADASD_ERR_NULL;
    if (u_dev != nullptr && token_out_dev == nullptr) return ADASD_ERR_NULL;
    if (int rc = check_device(ctx)) return rc;
    if (!aligned_to(logits_dev, elt_size(ctx->cfg.dtype)) ||
        !aligned4({u_dev, H_out_dev, lse_out_dev, token_out_dev, draft_len_inout_dev}))
        return ADASD_ERR_ALIGN;
    if (row_stride < ctx->cfg.V) return ADASD_ERR_SHAPE;
    DraftParams p;
    memset(&p, 0, sizeof(p));
    p.z = logits_dev;
    p.row_stride = row_stride;
    p.u = u_dev;
    p.active = active_inout_dev;
    p.H_out = H_out_dev;
    p.lse_out = lse_out_dev;
    p.token_out = token_out_dev;
    p.argmax = (!u_dev && token_out_dev) ? 1 : 0;
    p.early = ctx->draft_early ? 1 : 0;
    p.stop_out = stop_out_dev;
    p.draft_len = draft_len_inout_dev;
    p.st = ctx->st;
    p.B = ctx->cfg.B;
    p.V = ctx->cfg.V;
    p.expire_row = expire_row;
    p.c1 = kLog2e / ctx->temperature;
    if (ctx->cuts_on()) p.cut = ctx->cut_row;
    const bool aligned = vec_ok(logits_dev, ctx->cfg.dtype, {row_stride});
    // (the self-test is kept to the rows its header names)
    if (expire_row >= 0 && !(aligned && ctx->cfg.dtype == ADASD_BF16 && (p.V & 7) == 0 && p.V >= 8192 && expire_row < p.B))
        return ADASD_ERR_SHAPE;
    cudaStream_t st = (cudaStream_t)stream;
    if (ctx->cuts_on()) {
        if (int rc = launch_cutoffs(ctx, cut_params(ctx, logits_dev, row_stride, 0, 1, 1, nullptr, active_inout_dev, ctx->cut_row), nullptr, st))
            return rc;
    }
    if (aligned && !p.argmax && draft_rows(ctx))
        return ctx->draft_nw == kDW ? launch_draft_rows<kDW>(ctx, p, st) : launch_draft_rows<kDWBig>(ctx, p, st);
    return ctx->cfg.dtype == ADASD_BF16 ? launch_draft<__nv_bfloat16>(ctx, p, aligned, st) : launch_draft<float>(ctx, p, aligned, st);
}

int adasd_draft_entropy(adasd_ctx* ctx, const void* logits_dev, int64_t row_stride,
                        const float* u_dev, uint8_t* active_inout_dev, float* H_out_dev,
                        float* lse_out_dev, int32_t* token_out_dev, uint8_t* stop_out_dev,
                        int32_t* draft_len_inout_dev, void* stream) {
    return draft_entropy_impl(ctx, logits_dev, row_stride, u_dev, active_inout_dev, H_out_dev, lse_out_dev,
                              token_out_dev, stop_out_dev, draft_len_inout_dev, stream, -1);
}

int adasd_selftest_expired_wait(adasd_ctx* ctx, const void* logits_dev, int64_t row_stride, int32_t row,
                                const float* u_dev, float* H_out_dev, int32_t* token_out_dev, void* stream) {
    if (row < 0) return ADASD_ERR_SHAPE;
    return draft_entropy_impl(ctx, logits_dev, row_stride, u_dev, nullptr, H_out_dev, nullptr, token_out_dev,
                              nullptr, nullptr, stream, row);
}

int adasd_verify(adasd_ctx* ctx, const void* draft_logits_dev, const void* target_logits_dev,
                 int64_t d_seq_stride, int64_t d_row_stride, int64_t t_seq_stride,
                 int64_t t_row_stride, const int32_t* draft_tokens_dev,
                 const int32_t* draft_len_dev, const float* u_target_dev,
                 const float* u_accept_dev, int32_t* accept_len_dev, int32_t* next_token_dev,
                 const adasd_round_record* record, uint32_t flags, void* stream) {
    VerifyParams p;
    int rc = fill_verify_params(ctx, p, draft_logits_dev, target_logits_dev, d_seq_stride,
                                d_row_stride, t_seq_stride, t_row_stride, draft_tokens_dev,
                                draft_len_dev);
    if (rc != ADASD_OK) return rc;
    if (!u_target_dev || !u_accept_dev || !accept_len_dev || !next_token_dev)
        return ADASD_ERR_NULL;
    if (!aligned4({u_target_dev, u_accept_dev, accept_len_dev, next_token_dev})) return ADASD_ERR_ALIGN;
    if (record && !aligned4({record->H_d, record->H_t, record->lse_d, record->lse_t, record->jsd,
                             record->dist, record->p_acc, record->y, record->draft_len,
                             record->accept_len, record->rejected}))
        return ADASD_ERR_ALIGN;
    if (flags & ~ADASD_FUSE_UPDATE) return ADASD_ERR_SHAPE;
    p.u_target = u_target_dev;
    p.u_accept = u_accept_dev;
    p.accept_len = accept_len_dev;
    p.next_token = next_token_dev;
    if (record) p.user = *record;
    cudaStream_t st = (cudaStream_t)stream;
    if ((rc = launch_verify(ctx, p, st)) != ADASD_OK) return rc;
    TailParams t;
    memset(&t, 0, sizeof(t));
    t.cfg.Kmax = ctx->cfg.Kmax;
    t.cfg.min_samples = ctx->cfg.min_kde_samples;
    t.cfg.bw_rule = ctx->cfg.kde_bandwidth;
    t.cfg.reject_rule = ctx->cfg.reject_rule;
    t.cfg.update = (flags & ADASD_FUSE_UPDATE) ? 1u : 0u;
    t.st = ctx->st;
    t.H_d = ctx->sc.H_d;
    t.dist = ctx->sc.dist;
    t.y = ctx->sc.y;
    t.x = p.x;
    t.u_accept = p.u_accept;
    t.draft_len = p.draft_len;
    t.p_acc = p.user.p_acc;
    t.accept_len_rec = p.user.accept_len;
    t.rejected_rec = p.user.rejected;
    t.draft_len_rec = p.user.draft_len;
    t.accept_len = p.accept_len;
    t.next_token = p.next_token;
    const int S = tail_cluster(ctx);
    return launch_pdl(verify_tail_kernel, ctx->cfg.B * S, kTailThreads, 0, S, st, t);
}

int adasd_update_thresholds(adasd_ctx* ctx, const adasd_round_record* record, void* stream) {
    if (!ctx || !record) return ADASD_ERR_NULL;
    if (!record->H_d || !record->dist || !record->draft_len || !record->accept_len ||
        !record->rejected)
        return ADASD_ERR_NULL;
    if (int rc = check_device(ctx)) return rc;
    if (!aligned4({record->H_d, record->dist, record->draft_len, record->accept_len, record->rejected}))
        return ADASD_ERR_ALIGN;
    const int B = ctx->cfg.B;
    update_kernel<<<(B + 127) / 128, 128, 0, (cudaStream_t)stream>>>(ctx->st, *record, B,
                                                                     ctx->cfg.Kmax);
    CUDA_TRY(cudaGetLastError());
    return ADASD_OK;
}

int adasd_vanilla_verify(adasd_ctx* ctx, const void* draft_logits_dev,
                         const void* target_logits_dev, int64_t d_seq_stride,
                         int64_t d_row_stride, int64_t t_seq_stride, int64_t t_row_stride,
                         const int32_t* draft_tokens_dev, const int32_t* draft_len_dev,
                         const float* u_accept_dev, const float* u_resample_dev,
                         int32_t* accept_len_dev, int32_t* next_token_dev, float* alpha_out_dev,
                         void* stream) {
    VerifyParams p;
    int rc = fill_verify_params(ctx, p, draft_logits_dev, target_logits_dev, d_seq_stride,
                                d_row_stride, t_seq_stride, t_row_stride, draft_tokens_dev,
                                draft_len_dev);
    if (rc != ADASD_OK) return rc;
    if (!u_accept_dev || !u_resample_dev || !accept_len_dev || !next_token_dev)
        return ADASD_ERR_NULL;
    if (!aligned4({u_accept_dev, u_resample_dev, accept_len_dev, next_token_dev, alpha_out_dev}))
        return ADASD_ERR_ALIGN;
    p.u_accept = u_accept_dev;
    p.u_resample = u_resample_dev;
    p.accept_len = accept_len_dev;
    p.next_token = next_token_dev;
    p.alpha_out = alpha_out_dev;
    cudaStream_t st = (cudaStream_t)stream;
    const bool aligned = vec_ok(p.zd, ctx->cfg.dtype, {p.d_seq, p.d_row}) && vec_ok(p.zt, ctx->cfg.dtype, {p.t_seq, p.t_row});
    if ((rc = launch_round_cutoffs(ctx, p, st))) return rc;
    StreamParams sp;
    memset(&sp, 0, sizeof(sp));
    sp.zd = p.zd;
    sp.zt = p.zt;
    sp.d_seq = p.d_seq;
    sp.d_row = p.d_row;
    sp.t_seq = p.t_seq;
    sp.t_row = p.t_row;
    sp.draft_len = p.draft_len;
    sp.seg = ctx->seg;
    sp.status = ctx->st.status;
    sp.next = ctx->stream_next;
    sp.B = p.B;
    sp.V = p.V;
    sp.Kmax = p.Kmax;
    sp.seg_bits = ctx->seg_bits;
    sp.c1 = p.c1;
    sp.cut_t = p.cut_t;
    sp.cut_d = p.cut_d;
    if ((rc = launch_stream(ctx, sp, OP_LSE, aligned, st))) return rc;
    VanillaParams vp;
    vp.v = p;
    vp.seg = ctx->seg;
    vp.next = ctx->stream_next;
    vp.seg_bits = ctx->seg_bits;
    // CTAs per sequence: until the SMs carry two each, as long as a warp keeps an iteration or two
    const int NI = (ctx->cfg.V / (ctx->cfg.dtype == ADASD_BF16 ? 8 : 4) + 31) / 32;
    int S = 1;
    while (S < kVMaxS && (long long)p.B * S * 2 <= 4LL * ctx->sm_count && NI >= 2 * S * kVWarps) S *= 2;
    const int grid = p.B * S;
    if (ctx->cfg.dtype == ADASD_BF16)
        return aligned ? launch_pdl(vanilla_finish_kernel<__nv_bfloat16, true>, grid, kVThreads, 0, S, st, vp)
                       : launch_pdl(vanilla_finish_kernel<__nv_bfloat16, false>, grid, kVThreads, 0, S, st, vp);
    return aligned ? launch_pdl(vanilla_finish_kernel<float, true>, grid, kVThreads, 0, S, st, vp)
                   : launch_pdl(vanilla_finish_kernel<float, false>, grid, kVThreads, 0, S, st, vp);
}

int adasd_greedy_verify(adasd_ctx* ctx, const void* target_logits_dev, int64_t t_seq_stride,
                        int64_t t_row_stride, const int32_t* draft_tokens_dev,
                        const int32_t* draft_len_dev, int32_t* accept_len_dev, int32_t* next_token_dev,
                        int32_t* argmax_out_dev, void* stream) {
    if (!ctx || !target_logits_dev || !draft_tokens_dev || !accept_len_dev || !next_token_dev)
        return ADASD_ERR_NULL;
    if (int rc = check_device(ctx)) return rc;
    if (!aligned_to(target_logits_dev, elt_size(ctx->cfg.dtype)) ||
        !aligned4({draft_tokens_dev, draft_len_dev, accept_len_dev, next_token_dev, argmax_out_dev}))
        return ADASD_ERR_ALIGN;
    if (int rc = check_strides(ctx, t_seq_stride, t_row_stride)) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const int B = ctx->cfg.B, K = ctx->cfg.Kmax;
    StreamParams sp;
    memset(&sp, 0, sizeof(sp));
    sp.zt = target_logits_dev;
    sp.t_seq = t_seq_stride;
    sp.t_row = t_row_stride;
    sp.draft_len = draft_len_dev;
    sp.seg = ctx->seg;
    sp.status = ctx->st.status;
    sp.next = ctx->stream_next;
    sp.B = B;
    sp.V = ctx->cfg.V;
    sp.Kmax = K;
    sp.seg_bits = ctx->seg_bits;
    sp.c1 = kLog2e;
    const bool aligned = vec_ok(target_logits_dev, ctx->cfg.dtype, {t_seq_stride, t_row_stride});
    if (int rc = launch_stream(ctx, sp, OP_ARGMAX, aligned, st)) return rc;
    GreedyParams g;
    g.seg = ctx->seg;
    g.x = draft_tokens_dev;
    g.draft_len = draft_len_dev;
    g.accept_len = accept_len_dev;
    g.next_token = next_token_dev;
    g.argmax_out = argmax_out_dev;
    g.status = ctx->st.status;
    g.next = ctx->stream_next;
    g.Kmax = K;
    g.seg_bits = ctx->seg_bits;
    return launch_pdl(greedy_finish_kernel, B, kGThreads, 0, 0, st, g);
}

int adasd_gen_only_update(adasd_ctx* ctx, const float* H_draft_dev, const int32_t* draft_len_dev,
                          const int32_t* accept_len_dev, void* stream) {
    if (!ctx || !H_draft_dev || !accept_len_dev) return ADASD_ERR_NULL;
    if (int rc = check_device(ctx)) return rc;
    if (!aligned4({H_draft_dev, draft_len_dev, accept_len_dev})) return ADASD_ERR_ALIGN;
    const int B = ctx->cfg.B;
    gen_only_update_kernel<<<(B + 127) / 128, 128, 0, (cudaStream_t)stream>>>(ctx->st, H_draft_dev, draft_len_dev,
                                                                             accept_len_dev, B, ctx->cfg.Kmax);
    CUDA_TRY(cudaGetLastError());
    return ADASD_OK;
}

int adasd_set_warpers(adasd_ctx* ctx, float temperature, int32_t top_k, float top_p) {
    if (!ctx) return ADASD_ERR_NULL;
    if (!(temperature > 0.f) || !std::isfinite(temperature)) return ADASD_ERR_SHAPE;
    if (!(top_p > 0.f) || top_p > 1.f) return ADASD_ERR_SHAPE;
    ctx->temperature = temperature;
    ctx->top_k = top_k < 0 ? 0 : top_k;
    ctx->top_p = top_p;
    return ADASD_OK;
}

int adasd_get_thresholds(adasd_ctx* ctx, float* T_G_dev, int32_t* nE_dev, int32_t* nA_dev,
                         int32_t* nR_dev, void* stream) {
    if (!ctx) return ADASD_ERR_NULL;
    if (int rc = check_device(ctx)) return rc;
    if (!aligned4({T_G_dev, nE_dev, nA_dev, nR_dev})) return ADASD_ERR_ALIGN;
    const int B = ctx->cfg.B;
    get_thresholds_kernel<<<(B + 127) / 128, 128, 0, (cudaStream_t)stream>>>(
        ctx->st, T_G_dev, nE_dev, nA_dev, nR_dev, B);
    CUDA_TRY(cudaGetLastError());
    return ADASD_OK;
}

int adasd_state_export(adasd_ctx* ctx, int32_t seq, void* host_buf, size_t* bytes) {
    if (!ctx || !bytes) return ADASD_ERR_NULL;
    if (seq < 0 || seq >= ctx->cfg.B) return ADASD_ERR_SHAPE;
    DeviceGuard guard(ctx->cfg.device);
    CUDA_TRY(cudaDeviceSynchronize());
    const State& s = ctx->st;
    int32_t n[3];
    float tg;
    CUDA_TRY(cudaMemcpy(&n[0], s.nE + seq, 4, cudaMemcpyDeviceToHost));
    CUDA_TRY(cudaMemcpy(&n[1], s.nA + seq, 4, cudaMemcpyDeviceToHost));
    CUDA_TRY(cudaMemcpy(&n[2], s.nR + seq, 4, cudaMemcpyDeviceToHost));
    CUDA_TRY(cudaMemcpy(&tg, s.T_G + seq, 4, cudaMemcpyDeviceToHost));
    if (n[0] > s.cap) n[0] = s.cap;   // entropies beyond the capacity were only summed
    const size_t need = kExportHeader + 4 * ((size_t)n[0] + n[1] + n[2]);
    if (!host_buf) {
        *bytes = need;
        return ADASD_OK;
    }
    if (*bytes < need) {
        *bytes = need;
        return ADASD_ERR_CAPACITY;
    }
    char* o = static_cast<char*>(host_buf);
    int32_t hdr[4] = {n[0], n[1], n[2], 0};
    float fh[2] = {tg, 0.f};
    memcpy(o, hdr, 16);
    memcpy(o + 16, fh, 8);
    o += kExportHeader;
    const float* lists[3] = {s.LE, s.LA, s.LR};
    for (int k = 0; k < 3; ++k) {
        if (n[k] > 0)
            CUDA_TRY(cudaMemcpy(o, lists[k] + (size_t)seq * s.cap, 4 * (size_t)n[k],
                                cudaMemcpyDeviceToHost));
        o += 4 * (size_t)n[k];
    }
    *bytes = need;
    return ADASD_OK;
}

int adasd_state_import(adasd_ctx* ctx, int32_t seq, const void* host_buf, size_t bytes) {
    if (!ctx || !host_buf) return ADASD_ERR_NULL;
    if (seq < 0 || seq >= ctx->cfg.B || bytes < kExportHeader) return ADASD_ERR_SHAPE;
    const char* in = static_cast<const char*>(host_buf);
    int32_t hdr[4];
    float fh[2];
    memcpy(hdr, in, 16);
    memcpy(fh, in + 16, 8);
    const State& s = ctx->st;
    for (int k = 0; k < 3; ++k)
        if (hdr[k] < 0 || hdr[k] > s.cap) return ADASD_ERR_CAPACITY;
    if (bytes < kExportHeader + 4 * ((size_t)hdr[0] + hdr[1] + hdr[2])) return ADASD_ERR_SHAPE;
    DeviceGuard guard(ctx->cfg.device);
    CUDA_TRY(cudaDeviceSynchronize());
    const float* src = reinterpret_cast<const float*>(in + kExportHeader);
    float* lists[3] = {s.LE, s.LA, s.LR};
    double sums[3] = {0, 0, 0}, sums2[3] = {0, 0, 0};
    for (int k = 0; k < 3; ++k) {
        for (int j = 0; j < hdr[k]; ++j) {
            float v;
            memcpy(&v, src + j, 4);
            sums[k] += (double)v;
            sums2[k] += (double)v * (double)v;
        }
        if (hdr[k] > 0)
            CUDA_TRY(cudaMemcpy(lists[k] + (size_t)seq * s.cap, src, 4 * (size_t)hdr[k],
                                cudaMemcpyHostToDevice));
        src += hdr[k];
    }
    float tg = hdr[0] > 0 ? (float)(sums[0] / (double)hdr[0]) : fh[0];
    CUDA_TRY(cudaMemcpy(s.nE + seq, &hdr[0], 4, cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMemcpy(s.nA + seq, &hdr[1], 4, cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMemcpy(s.nR + seq, &hdr[2], 4, cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMemcpy(s.T_G + seq, &tg, 4, cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMemcpy(s.sumE + seq, &sums[0], 8, cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMemcpy(s.sumA + seq, &sums[1], 8, cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMemcpy(s.sumA2 + seq, &sums2[1], 8, cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMemcpy(s.sumR + seq, &sums[2], 8, cudaMemcpyHostToDevice));
    CUDA_TRY(cudaMemcpy(s.sumR2 + seq, &sums2[2], 8, cudaMemcpyHostToDevice));
    return ADASD_OK;
}

int adasd_status(adasd_ctx* ctx, uint32_t* status_out) {
    if (!ctx || !status_out) return ADASD_ERR_NULL;
    DeviceGuard guard(ctx->cfg.device);
    CUDA_TRY(cudaDeviceSynchronize());
    CUDA_TRY(cudaMemcpy(status_out, ctx->st.status, 4, cudaMemcpyDeviceToHost));
    CUDA_TRY(cudaMemset(ctx->st.status, 0, 4));
    return ADASD_OK;
}

int adasd_vanilla_verify_static(int32_t B, int32_t V, int32_t Kmax, int32_t dtype,
                                const void* draft_logits_dev, const void* target_logits_dev,
                                int64_t d_seq_stride, int64_t d_row_stride, int64_t t_seq_stride,
                                int64_t t_row_stride, const int32_t* draft_tokens_dev,
                                const int32_t* draft_len_dev, const float* u_accept_dev,
                                const float* u_resample_dev, int32_t* accept_len_dev,
                                int32_t* next_token_dev, float* alpha_out_dev,
                                uint32_t* status_out_dev, void* stream) {
    if (!draft_logits_dev || !target_logits_dev || !draft_tokens_dev || !u_accept_dev ||
        !u_resample_dev || !accept_len_dev || !next_token_dev)
        return ADASD_ERR_NULL;
    if (dtype != ADASD_BF16 && dtype != ADASD_FP32) return ADASD_ERR_DTYPE;
    if (B < 1 || V < 1 || Kmax < 1 || Kmax > ADASD_KMAX_LIMIT) return ADASD_ERR_SHAPE;
    if (B > ADASD_STATIC_MAX_B || (long long)B * (Kmax + 1) > ADASD_STATIC_MAX_POSITIONS)
        return ADASD_ERR_CAPACITY;
    if (d_row_stride < V || t_row_stride < V || d_seq_stride < 0 || t_seq_stride < 0)
        return ADASD_ERR_SHAPE;
    if (!aligned_to(draft_logits_dev, elt_size(dtype)) || !aligned_to(target_logits_dev, elt_size(dtype)) ||
        !aligned4({draft_tokens_dev, draft_len_dev, u_accept_dev, u_resample_dev, accept_len_dev,
                   next_token_dev, alpha_out_dev, status_out_dev}))
        return ADASD_ERR_ALIGN;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
        cudaGetLastError();
        return ADASD_ERR_CUDA;
    }
    StaticSetup su;
    int rc = static_setup(dev, su);
    if (rc != ADASD_OK) return rc;

    cudaStream_t st = (cudaStream_t)stream;
    uint32_t* flag = su.base;
    uint32_t* tok = su.base + ADASD_STATIC_MAX_POSITIONS;
    uint32_t* ticket = su.base + 2 * ADASD_STATIC_MAX_POSITIONS;
    uint32_t* status = status_out_dev ? status_out_dev : ticket + ADASD_STATIC_MAX_B;
    // the array keeps whatever the previous call left: counters and status start at zero
    CUDA_TRY(cudaMemsetAsync(ticket, 0, sizeof(uint32_t) * (size_t)B, st));
    CUDA_TRY(cudaMemsetAsync(status, 0, sizeof(uint32_t), st));

    VerifyParams p;
    memset(&p, 0, sizeof(p));
    p.inv_temp = 1.f;                        // no context, no adjusted distribution
    p.c1 = kLog2e;
    p.zd = draft_logits_dev;
    p.zt = target_logits_dev;
    p.d_seq = d_seq_stride;
    p.d_row = d_row_stride;
    p.t_seq = t_seq_stride;
    p.t_row = t_row_stride;
    p.x = draft_tokens_dev;
    p.draft_len = draft_len_dev;
    p.u_accept = u_accept_dev;
    p.u_resample = u_resample_dev;
    p.accept_len = accept_len_dev;
    p.next_token = next_token_dev;
    p.alpha_out = alpha_out_dev;
    p.sc.van_flag = reinterpret_cast<int32_t*>(flag);
    p.sc.van_tok = reinterpret_cast<int32_t*>(tok);
    p.sc.ticket = ticket;
    p.st.status = status;
    p.B = B;
    p.V = V;
    p.Kmax = Kmax;

    const long long positions = (long long)B * (Kmax + 1);
    int cs = kMaxCluster;
    for (int c = 1; c <= kMaxCluster; c *= 2)
        if (positions * c >= 2LL * su.sm_count) {
            cs = c;
            break;
        }
    const bool vec = vec_ok(draft_logits_dev, dtype, {d_seq_stride, d_row_stride}) &&
                     vec_ok(target_logits_dev, dtype, {t_seq_stride, t_row_stride});
    if (dtype == ADASD_BF16)
        return vec ? launch_cluster(static_vanilla_kernel<__nv_bfloat16, true>, p, positions, cs, st)
                   : launch_cluster(static_vanilla_kernel<__nv_bfloat16, false>, p, positions, cs, st);
    return vec ? launch_cluster(static_vanilla_kernel<float, true>, p, positions, cs, st)
               : launch_cluster(static_vanilla_kernel<float, false>, p, positions, cs, st);
}

const char* adasd_strerror(int code) {
    switch (code) {
        case ADASD_OK: return "ok";
        case ADASD_ERR_NULL: return "a required pointer is NULL";
        case ADASD_ERR_ALIGN: return "a pointer is not aligned to its element type";
        case ADASD_ERR_SHAPE: return "size, stride or window out of range";
        case ADASD_ERR_DTYPE: return "unknown dtype or rule";
        case ADASD_ERR_CAPACITY: return "size beyond a stated maximum";
        case ADASD_ERR_CUDA: return "a CUDA runtime call failed";
        case ADASD_ERR_DEVICE: return "the current device is not the context's device";
        default: return "unknown error";
    }
}

}  // extern "C"
