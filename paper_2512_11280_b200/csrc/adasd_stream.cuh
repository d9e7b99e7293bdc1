// Streaming row statistics for sm_100a: what vanilla speculative sampling and greedy decoding need of
// the rows of a round, read from HBM once.  bf16 or fp32 rows of any length, alignment and stride.
//
// The accept test of a vanilla candidate needs only the softmax normalisers of its two rows,
// alpha = min(1, p(x) / q(x)), as the largest logit m and S = sum 2^((z - m) log2 e): log2 p(x) = (z[x] - m) log2 e - log2 S
// stays as accurate for rows whose logits share a large offset, where a log-sum-exp would round to a
// multiple of its own last bit (logits around 5000: 4e-4 in alpha).  Only ONE position of a sequence needs more,
// the first rejected one (its residual max(0, p - q) is sampled) or, if none is rejected, the bonus
// row.  The greedy test needs the target rows' argmax.  So:
//
//  1. row_stream_kernel streams every needed row once: the row is cut into segments, a WARP takes a
//     segment at a time and leaves its largest logit and the sum of 2^t under it, or its index, in
//     a table.  No warp waits for another: the rounding of a row to warps costs nothing but its
//     last, shorter, copy, and one row of one sequence spreads over the chip as well as a batch does.
//  2. vanilla_finish_kernel (a cluster per sequence) folds the segments, forms the alphas, finds the
//     first rejection and samples the one position that is left;
//     greedy_finish_kernel (a CTA per sequence) folds the segments and scans for the first mismatch.
//
// What bounds step 1 is HBM (one exponential and about 6 instructions per logit): 16 warps per SM with
// three 4 KB bulk copies each in flight, running on across segment and row borders.  Measured, a call on
// 4224 rows of 151936 bf16 logits (1.28 GB): 222 us, of which step 1 is about 209 (6.1 TB/s); 544 rows of
// 128256 (140 MB): 43 us, of which step 1 is 31 and step 2, a chain of dependent loads, 11.
#pragma once

#include "adasd_async.cuh"

namespace adasd {

constexpr int kRW = 8;                           // warps per CTA, two CTAs per SM
constexpr int kRThreads = kRW * 32;
constexpr int kRRing = 3;
constexpr int kRStage = 8 * 512 + 16;            // a chunk of 8 iterations (+ one unit: rows off a 16-byte boundary)
constexpr int kRSmem = kRW * kRRing * kRStage;
constexpr int kMaxSegs = 64;                     // segments of a row, at most
constexpr float kRBig = 1e7f;                    // shifts up to it are exact to 0.5
constexpr int kRItems = 4;                       // items of a warp that may be between their first copy and their end

constexpr int OP_LSE = 0, OP_ARGMAX = 1;

struct StreamParams {
    const void* zd;                              // draft rows (null: target rows only)
    const void* zt;
    long long d_seq, d_row, t_seq, t_row;
    const int32_t* draft_len;                    // nullable: Kmax
    float4* seg;                                 // [rows][2^seg_bits]: rows of sequence b from b (2 Kmax + 1): target, then draft
    uint32_t* status;
    uint32_t* next;                              // items drawn so far beyond the first two of every warp (the finish kernel puts it back to 0)
    int32_t B, V, Kmax, seg_bits;                // 2^seg_bits segments a row
    float c1;                                    // log2 e / temperature (adjusted distribution)
    const float* cut_t;                          // nullable [B, Kmax + 1]: logit below which a row's tokens are cut
    const float* cut_d;                          // nullable [B, Kmax]
};

// A row is cut into NC chunks of IT iterations (32 lanes x 16 bytes each), and these into at most NC
// segments of whole chunks: segment s starts at this one.
__device__ __forceinline__ int seg_begin(int s, int NC, int seg_bits) { return (int)(((long long)s * NC) >> seg_bits); }

// What a warp needs of an item it has asked for: written when its first copy is issued.
struct __align__(16) StreamItem {
    int32_t slot;                                // row in the table; -1: no more items
    int32_t seg, ch0, ch1;                       // segment and its chunks
    int32_t shift;                               // elements between the row's 16-byte boundary and the row
    float cut;
    int32_t pad[2];
};

// Largest logit of elements [e0, e1) of a row and the sum of 2^((z - m) log2 e / T), by a warp, element by element
// from memory: logits or 1 / T so large (1e7 and more between them) that a shift fl(m log2 e / T) is off by whole
// powers of two.
template <typename T>
__device__ __noinline__ float2 big_segment(const T* row, int e0, int e1, float c1, float cut) {
    const int lane = threadIdx.x & 31;
    float m = kFloorL, S = 0.f;
    for (int e = e0 + lane; e < e1; e += 32) m = fmaxf(m, to_f32(row[e]));
    m = warp_max_f32(m);
    for (int e = e0 + lane; e < e1; e += 32) {
        const float z = to_f32(row[e]);
        if (z >= cut) S += ex2((z - m) * c1);
    }
    return make_float2(m, warp_sum(S));
}

// IT: 8 iterations a chunk, or 2 where the launch has too few chunks of 8 for its warps.
// (bounds of 320 threads: at most 96 registers a thread)
template <typename T, bool ALIGNED, int OP, bool WARPED, int IT>
__global__ void __launch_bounds__(320, 2) row_stream_kernel(StreamParams p) {
    using U = Unit<T>;
    constexpr int N = U::N, NP = N / 2;
    const float floor_v = N == 8 ? ADASD_FLOOR_BF : kFloor;
    extern __shared__ __align__(128) unsigned char dyn_smem[];
    __shared__ unsigned long long bars[kRW][kRRing];
    __shared__ StreamItem items[kRW][kRItems];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int K = p.Kmax, K1 = K + 1, R = 2 * K + 1;
    const int rows_of_d = p.zd ? 1 : 0;
    const int NU = (p.V + N - 1) / N, NC = (NU + 32 * IT - 1) / (32 * IT);
    const int GW = (int)gridDim.x * kRW, gw = (int)blockIdx.x * kRW + warp;
    const float c1 = WARPED ? p.c1 : kLog2e, inv_c1 = 1.f / c1;
    auto row_of = [&](int slot) -> const T* {    // (of the table)
        const int b = slot / R, i = slot - b * R;
        return i <= K ? reinterpret_cast<const T*>(p.zt) + (long long)b * p.t_seq + (long long)i * p.t_row
                      : reinterpret_cast<const T*>(p.zd) + (long long)b * p.d_seq + (long long)(i - K1) * p.d_row;
    };
    unsigned char* const ring = dyn_smem + (size_t)warp * (kRRing * kRStage);
    if (lane == 0) {
        for (int s = 0; s < kRRing; ++s) mbar_init(reinterpret_cast<uint64_t*>(&bars[warp][s]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    pdl_wait();
    pdl_trigger();

    // Items are the segments of the needed rows, sequence by sequence (target rows 0 .. K_b, then draft
    // rows 0 .. K_b - 1).  A warp starts with numbers gw and gw + GW and draws the others (dealt in turn
    // they would leave up to a whole item's time idle at the end: 246 against 232 us for a call that
    // streams 1.28 GB); a number is drawn two items ahead of its use, so that nothing waits for it.  A block of 32 sequences at a
    // time: lane l holds the number of rows of sequence blk_b + l and their running total.
    long long item = gw, blk_rank = 0;           // the next item; rows before the block
    uint32_t drawn = 0;
    bool first = true;
    auto draw = [&]() {
        if (lane == 0) drawn = atomicAdd(p.next, 1u);
    };
    draw();
    int blk_b = 0, blk_cnt = 0, blk_incl = 0, blk_tot = 0;
    auto load_block = [&]() {
        const int b = blk_b + lane;
        int kt = K;
        if (b < p.B && p.draft_len) kt = max(0, min(__ldcg(p.draft_len + b), K));
        blk_cnt = b < p.B ? kt + 1 + (rows_of_d ? kt : 0) : 0;
        blk_incl = blk_cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xFFFFFFFFu, blk_incl, o);
            if (lane >= o) blk_incl += t;
        }
        blk_tot = __shfl_sync(0xFFFFFFFFu, blk_incl, 31);
    };
    load_block();
    // the item being asked for
    const unsigned char* base = nullptr;         // its row, rounded down to 16 bytes
    int g1 = 0, ich = 0, ich1 = 0, n_items = 0;  // granules that hold elements: [0, g1); its next chunk, its end
    bool more = true;
    auto next_item = [&]() {
        StreamItem d;
        d.slot = -1;
        const long long rank = item >> p.seg_bits;
        const int seg = (int)(item - (rank << p.seg_bits));
        while (blk_b < p.B && rank >= blk_rank + blk_tot) {
            blk_rank += blk_tot;
            blk_b += 32;
            if (blk_b < p.B) load_block();
        }
        more = blk_b < p.B;
        if (more) {
            if (first) {
                item += GW;
            } else {
                item = 2LL * GW + __shfl_sync(0xFFFFFFFFu, drawn, 0);
                draw();
            }
            first = false;
            ich = seg_begin(seg, NC, p.seg_bits);
            ich1 = seg_begin(seg + 1, NC, p.seg_bits);
            const int o = (int)(rank - blk_rank);
            const int src = __ffs(__ballot_sync(0xFFFFFFFFu, blk_incl > o)) - 1;
            const int cnt = __shfl_sync(0xFFFFFFFFu, blk_cnt, src);
            const int j = o - (__shfl_sync(0xFFFFFFFFu, blk_incl, src) - cnt);
            const int kt = rows_of_d ? (cnt - 1) >> 1 : cnt - 1;
            const int b = blk_b + src;
            const bool tgt = j <= kt;
            const int i = tgt ? j : j - kt - 1;
            const T* row = tgt ? reinterpret_cast<const T*>(p.zt) + (long long)b * p.t_seq + (long long)i * p.t_row
                               : reinterpret_cast<const T*>(p.zd) + (long long)b * p.d_seq + (long long)i * p.d_row;
            const unsigned long long a = reinterpret_cast<unsigned long long>(row);
            base = reinterpret_cast<const unsigned char*>(ALIGNED ? a : a & ~15ull);
            d.shift = ALIGNED ? 0 : (int)((a & 15ull) / sizeof(T));
            g1 = (d.shift + p.V + N - 1) / N;
            d.slot = b * R + (tgt ? i : K1 + i);
            d.seg = seg;
            d.ch0 = ich;
            d.ch1 = ich1;
            d.cut = -INFINITY;
            if (WARPED && p.cut_t) d.cut = tgt ? __ldcg(p.cut_t + (size_t)b * K1 + i) : __ldcg(p.cut_d + (size_t)b * K + i);
        }
        if (lane == 0) items[warp][n_items & (kRItems - 1)] = d;
        ++n_items;
        __syncwarp();
    };
    const float2 L2 = pair2(c1);
    bool alive = true;
    int is = 0, n_issued = 0, n_taken = 0;
    auto issue = [&]() {                         // the next chunk
        if (!alive || !more) return;
        if (lane == 0) {
            const int u0 = 32 * IT * ich, u1 = u0 + 32 * IT;
            const uint32_t bytes = (uint32_t)(min(ALIGNED ? u1 : u1 + 1, g1) - u0) * 16u;
            uint64_t* bar = reinterpret_cast<uint64_t*>(&bars[warp][is]);
            mbar_expect_tx(bar, bytes);
            bulk_g2s(ring + is * kRStage, base + (size_t)u0 * 16, bytes, bar);
        }
        ++n_issued;
        is = is + 1 == kRRing ? 0 : is + 1;
        if (++ich == ich1) next_item();
    };
    next_item();
    for (int k = 0; k < kRRing; ++k) issue();

    int rs = 0;
    uint32_t rph = 0;
    for (int n = 0;; ++n) {
        const StreamItem c = items[warp][n & (kRItems - 1)];
        if (c.slot < 0) break;
        float v = kFloorL;                       // the segment's shift fl(z log2 e / T), z its largest logit (kFloorL: nothing finite)
        float2 S2 = make_float2(0.f, 0.f);
        // argmax: this lane's largest logit so far, its unit (the first that has it) and what is in it.  Any finite
        // logit counts, also one that has no probability (a mask of the type's lowest value)
        float top = -INFINITY;
        int top_u = -1;
        uint4 top_w = U::none4();
        uint32_t bad = 0u;
        const typename U::Cut cut = U::make_cut(c.cut);
        // One chunk; EDGE: the last one of the row.  The maximum first, then the sum, each from shared
        // memory: held in registers between the two, a chunk would take the kernel to 112 a thread, and
        // with 96 or fewer a CTA of the finish kernel is resident beside two of this one and past its
        // first loads when this kernel ends.
        auto chunk = [&](auto edge_c, int ch, const unsigned char* sb) {
            constexpr bool EDGE = decltype(edge_c)::value;
            auto load = [&](int k) -> uint4 {
                uint4 w = *reinterpret_cast<const uint4*>(sb + k * 512);
                if (!ALIGNED) w = U::realign(w, *reinterpret_cast<const uint4*>(sb + k * 512 + 16), c.shift);
                if (EDGE) {
                    const int v0 = (32 * (ch * IT + k) + lane) * N;
                    if (v0 + N > p.V) U::mask(w, 0, p.V - v0);
                }
                return w;
            };
            typename U::Max mx = U::max0();
            if (OP == OP_ARGMAX) {
#pragma unroll
                for (int k = 0; k < IT; ++k) {
                    const uint4 w = load(k);
                    const typename U::Max h = U::unit_max(w);
                    U::max_join(mx, h);
                    const float t = U::top(h);
                    if (t > top) {
                        top = t;
                        top_u = 32 * (ch * IT + k) + lane;
                        top_w = w;
                    }
                }
                U::max_val(mx, bad);
            } else {
#pragma unroll
                for (int k = 0; k < IT; ++k) U::max_add(mx, load(k));
                const float x = warp_max_f32(U::max_val(mx, bad));
                if (x == INFINITY) bad = 1u;
                if (x > floor_v && x * c1 > v) { // raise the shift, rescale what is summed
                    const float m = x * c1, f = ex2(v - m);
                    S2.x *= f;
                    S2.y *= f;
                    v = m;
                }
                const float nv = v > kFloorL ? -v : 0.f;
                const float2 nv2 = pair2(nv);
#pragma unroll 4
                for (int k = 0; k < IT; ++k) {
                    uint4 w = load(k);
                    if (WARPED) U::cut(w, cut);
                    float2 z[NP];
                    U::unpack_raw(w, z);
#pragma unroll
                    for (int j = 0; j < NP; ++j) {
                        const float2 t = __ffma2_rn(z[j], L2, nv2);
                        S2 = __fadd2_rn(S2, make_float2(ex2(t.x), ex2(t.y)));
                    }
                }
            }
            __syncwarp();
            issue();                             // the chunk has been read, its slot is free
        };
        for (int ch = c.ch0; ch < c.ch1; ++ch) {
            if (alive) {
                bool ok = mbar_wait_bounded(reinterpret_cast<uint64_t*>(&bars[warp][rs]), rph);
                ok = __all_sync(0xFFFFFFFFu, ok);
                if (!ok) {
                    alive = false;
                    if (lane == 0) atomicOr(p.status, ADASD_STATUS_TIMEOUT);
                } else {
                    ++n_taken;
                }
            }
            const unsigned char* sb = ring + rs * kRStage + lane * 16;
            if (++rs == kRRing) {
                rs = 0;
                rph ^= 1u;
            }
            if (!alive) bad = 1u;
            else if (ch == NC - 1) chunk(std::true_type{}, ch, sb);
            else chunk(std::false_type{}, ch, sb);
        }
        float S = 0.f;
        int idx = 0x7FFFFFFF;
        if (OP == OP_ARGMAX) {                   // lowest index of the largest logit: that of the lowest unit that has it
            v = warp_max_f32(top);
            if (v == INFINITY) bad = 1u;
            if (top_u >= 0 && top == v) {
                float2 z[NP];
                U::unpack_raw(top_w, z);
#pragma unroll
                for (int j = NP - 1; j >= 0; --j) {
                    if (z[j].y == v) idx = top_u * N + 2 * j + 1;
                    if (z[j].x == v) idx = top_u * N + 2 * j;
                }
            }
            idx = __reduce_min_sync(0xFFFFFFFFu, idx);
        } else {
            // The table holds a logit m next to the largest and the sum under it: the exponents z log2 e / T - v are all off by
            // the same residue m log2 e / T - v
            S = warp_sum(S2.x + S2.y);
            if (v > kFloorL) {
                if (fabsf(v) < kRBig) {
                    const float m = v * inv_c1;
                    S *= ex2(-fmaf(m, c1, -v));
                    v = m;
                } else {
                    const float2 ms = big_segment(row_of(c.slot), 32 * IT * N * c.ch0, min(32 * IT * N * c.ch1, p.V), c1, c.cut);
                    v = ms.x;
                    S = ms.y;
                }
            }
        }
        bad = __reduce_or_sync(0xFFFFFFFFu, bad);
        if (lane == 0) p.seg[((size_t)c.slot << p.seg_bits) + c.seg] = make_float4(v, S, __int_as_float(idx), __uint_as_float(bad));
        if (!alive) {
            // a copy never landed: nothing more is asked for, the rest of this warp's items are reported
            // unusable, and whatever is still in flight is waited for (bounded)
            for (int q = n_taken; q < n_issued; ++q)
                mbar_wait_bounded(reinterpret_cast<uint64_t*>(&bars[warp][q % kRRing]), (uint32_t)(q / kRRing) & 1u);
            for (int m = n + 1; m < n_items || more; ++m) {
                if (m >= n_items) next_item();
                const StreamItem d = items[warp][m & (kRItems - 1)];
                if (d.slot < 0) break;
                if (lane == 0) p.seg[((size_t)d.slot << p.seg_bits) + d.seg] = make_float4(kFloorL, 0.f, __int_as_float(-1), __uint_as_float(1u));
                __syncwarp();
            }
            break;
        }
    }
}

// The segments of a row, two to a lane, and what a whole warp makes of them.
struct SegPair {
    float4 a, b;
};
// (v_none: the maximum of a segment that does not exist)
__device__ __forceinline__ SegPair load_segments(const float4* seg, int segs, bool on, float v_none) {
    const int lane = threadIdx.x & 31;
    const float4 none = make_float4(v_none, 0.f, __int_as_float(-1), 0.f);
    SegPair r;
    r.a = on && lane < segs ? __ldcg(seg + lane) : none;
    r.b = on && lane + 32 < segs ? __ldcg(seg + lane + 32) : none;
    return r;
}
__device__ __forceinline__ bool segments_bad(const SegPair& s, float v, float v_none) {
    return __any_sync(0xFFFFFFFFu, (__float_as_uint(s.a.w) | __float_as_uint(s.b.w)) & 1u) || !(v > v_none);
}

// ---- vanilla: accept test and the one sampled position of every sequence ---------------------
//
// A cluster of S CTAs per sequence.  Each CTA folds the normalisers of the round's rows and finds the
// first rejection for itself; the row pair of that position is then read a second time (from L2 where
// the round is small), spread over the cluster's warps: with the normalisers known, p and q are final
// as they are read, so sums of the residual max(0, p - q) (and of p, for the bonus row and for a
// residual without mass) over blocks of a warp's share locate the crossing of u, and rank 0 scans that
// block again.  Latency bounds it: the caller's tokens, their logits and the uniforms are read before
// the wait for step 1.
constexpr int kVThreads = 256;
constexpr int kVWarps = kVThreads / 32;
constexpr int kVMaxS = 8;
constexpr int kVBlocks = 16;                     // blocks of a warp's share, at most

struct VanillaParams {
    VerifyParams v;
    const float4* seg;
    uint32_t* next;                              // row_stream_kernel's counter, put back to 0 here
    int32_t seg_bits;
};

struct VanillaShared {
    float2 row[2 * ADASD_KMAX_LIMIT + 1];        // largest logit and log2 S of the rows (NaN: unusable): target, then draft
    float2 tab[kVMaxS * kVWarps * kVBlocks];     // rank 0: (residual, target) mass of every block, warp by warp of the cluster
    int32_t w;
};

template <typename T, bool ALIGNED>
__global__ void __launch_bounds__(kVThreads, 4) vanilla_finish_kernel(VanillaParams q) {
    using U = Unit<T>;
    constexpr int N = U::N, NP = N / 2;
    const VerifyParams& p = q.v;
    __shared__ VanillaShared sh;
    cg::cluster_group cluster = cg::this_cluster();
    const int S = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int b = blockIdx.x / S;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int K = p.Kmax, K1 = K + 1, R = 2 * K + 1;
    const float c1 = p.c1;
    pdl_trigger();

    int kt = p.draft_len ? __ldcg(p.draft_len + b) : K;
    kt = max(0, min(kt, K));
    const T* const rt = reinterpret_cast<const T*>(p.zt) + (long long)b * p.t_seq;
    const T* const rd = reinterpret_cast<const T*>(p.zd) + (long long)b * p.d_seq;
    float u_acc = 0.f, ztx = 0.f, zdx = 0.f;
    bool x_ok = false;
    const float u_res = __ldcg(p.u_resample + b);
    if (warp == 0 && lane < kt) {
        const size_t idd = (size_t)b * K + lane;
        u_acc = __ldcg(p.u_accept + idd);
        const int xi = __ldcg(p.x + idd);
        x_ok = xi >= 0 && xi < p.V;
        if (x_ok) {
            ztx = to_f32(rt[(long long)lane * p.t_row + xi]);
            zdx = to_f32(rd[(long long)lane * p.d_row + xi]);
        }
    }
    if (S > 1) cluster.sync();                   // every CTA of the cluster runs: rank 0 may be written to
    pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0) *q.next = 0u;

    // row r: target 0 .. kt, draft 0 .. kt - 1; three rows of a warp are asked for before the first is folded
    const int segs = 1 << q.seg_bits;
    for (int r0 = warp; r0 < 2 * kt + 1; r0 += 3 * kVWarps) {
        SegPair sp[3];
        auto slot_of = [&](int r) -> int { return r <= kt ? r : K1 + (r - kt - 1); };
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int r = r0 + k * kVWarps;
            sp[k] = load_segments(q.seg + (((size_t)b * R + slot_of(r)) << q.seg_bits), segs, r < 2 * kt + 1, kFloorL);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int r = r0 + k * kVWarps;
            if (r < 2 * kt + 1) {
                const float v = warp_max_f32(fmaxf(sp[k].a.x, sp[k].b.x));
                const float sum = warp_sum(ex2((sp[k].a.x - v) * c1) * sp[k].a.y + ex2((sp[k].b.x - v) * c1) * sp[k].b.y);
                const float lS = segments_bad(sp[k], v, kFloorL) ? NAN : lg2(sum);
                if (lane == 0) sh.row[r <= kt ? r : ADASD_KMAX_LIMIT + 1 + (r - kt - 1)] = make_float2(v, lS);
            }
        }
    }
    __syncthreads();
    if (warp == 0) {
        bool reject = false, bad = false;
        if (lane < kt) {
            const size_t idd = (size_t)b * K + lane;
            const float2 mt = sh.row[lane], md = sh.row[ADASD_KMAX_LIMIT + 1 + lane];
            bad = (mt.y != mt.y) || (md.y != md.y);
            float alpha = 0.f;
            if (x_ok) {
                // log2 p(x) and log2 q(x): -inf for a logit below its row's cutoff; equal, and alpha exactly 1, where
                // the rows are
                if (p.cut_t && ztx < p.cut_t[(size_t)b * K1 + lane]) ztx = -INFINITY;
                if (p.cut_d && zdx < p.cut_d[idd]) zdx = -INFINITY;
                const float lp = fmaf(ztx - mt.x, c1, -mt.y), lq = fmaf(zdx - md.x, c1, -md.y);
                alpha = fminf(1.f, ex2(lp - lq));
                if (!(ex2(lq) > 0.f)) alpha = 1.f;       // q(x) = 0 cannot have been drafted
            }
            reject = bad || !(u_acc < alpha);
            if (rank == 0 && p.alpha_out) p.alpha_out[idd] = bad ? NAN : alpha;
        }
        const unsigned mr = __ballot_sync(0xFFFFFFFFu, reject), mb = __ballot_sync(0xFFFFFFFFu, bad);
        if (lane == 0) {
            const float lb = sh.row[kt].y;         // the bonus row
            if (rank == 0 && (mb || lb != lb)) atomicOr(p.st.status, ADASD_STATUS_NAN);
            sh.w = mr ? (__ffs(mr) - 1) : kt;
        }
    }
    __syncthreads();
    const int i = sh.w;
    const bool bonus = (i >= kt);
    const float2 mt = sh.row[i], md = bonus ? make_float2(0.f, 0.f) : sh.row[ADASD_KMAX_LIMIT + 1 + i];
    const bool rowbad = (mt.y != mt.y) || (md.y != md.y);

    // p and max(0, p - q) of unit u of the two rows
    const float2 c2 = pair2(c1), nmt2 = pair2(-mt.x), nst2 = pair2(-mt.y), nmd2 = pair2(-md.x), nsd2 = pair2(-md.y);
    const typename U::Cut cut_t = U::make_cut(p.cut_t ? __ldcg(p.cut_t + (size_t)b * K1 + i) : -INFINITY);
    const typename U::Cut cut_d = U::make_cut((p.cut_d && !bonus) ? __ldcg(p.cut_d + (size_t)b * K + i) : -INFINITY);
    const int NU = (p.V + N - 1) / N, NI = (NU + 31) >> 5;
    struct Row {
        const uint4* base;
        int shift, g1;
    };
    auto row_of = [&](const T* r) -> Row {
        const unsigned long long a = reinterpret_cast<unsigned long long>(r);
        Row o;
        o.base = reinterpret_cast<const uint4*>(ALIGNED ? a : a & ~15ull);
        o.shift = ALIGNED ? 0 : (int)((a & 15ull) / sizeof(T));
        o.g1 = (o.shift + p.V + N - 1) / N;
        return o;
    };
    const Row row_t = row_of(rt + (long long)i * p.t_row), row_d = row_of(rd + (long long)min(i, K - 1) * p.d_row);
    auto load = [&](const Row& r, int u) -> uint4 {
        uint4 w = u < r.g1 ? r.base[u] : U::none4();
        if (!ALIGNED) w = U::realign(w, u + 1 < r.g1 ? r.base[u + 1] : U::none4(), r.shift);
        return w;
    };
    auto weights = [&](uint4 a, uint4 d, int u, float (&pv)[N], float (&rv)[N]) {
        const int v0 = u * N;
        if (v0 + N > p.V) {
            U::mask(a, 0, p.V - v0);
            U::mask(d, 0, p.V - v0);
        }
        U::cut(a, cut_t);
        U::cut(d, cut_d);
        float2 z[NP], y[NP];
        U::unpack(a, z);
        U::unpack(d, y);
#pragma unroll
        for (int j = 0; j < NP; ++j) {
            const float2 lp = __ffma2_rn(__fadd2_rn(z[j], nmt2), c2, nst2), lq = __ffma2_rn(__fadd2_rn(y[j], nmd2), c2, nsd2);
            pv[2 * j] = ex2(lp.x);
            pv[2 * j + 1] = ex2(lp.y);
            const float q0 = bonus ? 0.f : ex2(lq.x), q1 = bonus ? 0.f : ex2(lq.y);
            rv[2 * j] = fmaxf(pv[2 * j] - q0, 0.f);
            rv[2 * j + 1] = fmaxf(pv[2 * j + 1] - q1, 0.f);
        }
    };
    const int G = S * kVWarps;
    // warp g's share: iterations [g NI / G, (g + 1) NI / G), in blocks of `per` (a multiple of 4)
    const int per_max = (NI + G - 1) / G;
    const int per = ((per_max + kVBlocks - 1) / kVBlocks + 3) & ~3;
    const int nblk = (per_max + per - 1) / per;      // blocks of a share
    if (!rowbad) {
        const int g = rank * kVWarps + warp;
        const int it0 = (int)((long long)g * NI / G), it1 = (int)((long long)(g + 1) * NI / G);
        float2* tab = &cluster.map_shared_rank(&sh, 0)->tab[g * nblk];
        float rs = 0.f, ps = 0.f;
        int blk = 0;
        for (int it = it0; it < it1; it += 4) {
            uint4 a[4], d[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int u = 32 * (it + k) + lane;
                a[k] = it + k < it1 ? load(row_t, u) : U::none4();
                d[k] = (it + k < it1 && !bonus) ? load(row_d, u) : U::none4();
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (it + k < it1) {
                    float pv[N], rv[N];
                    weights(a[k], d[k], 32 * (it + k) + lane, pv, rv);
#pragma unroll
                    for (int j = 0; j < N; ++j) {
                        ps += pv[j];
                        rs += rv[j];
                    }
                }
            }
            if (it + 4 >= it1 || it + 4 - it0 == (blk + 1) * per) {      // the block is complete
                rs = warp_sum(rs);
                ps = warp_sum(ps);
                if (lane == 0) tab[blk] = make_float2(rs, ps);
                rs = ps = 0.f;
                ++blk;
            }
        }
        if (lane >= blk && lane < nblk) tab[lane] = make_float2(0.f, 0.f);
    }
    if (S > 1) cluster.sync();
    else __syncthreads();
    if (rank != 0 || warp != 0) return;

    int tok = -1;
    if (!rowbad) {
        // lane l takes consecutive blocks: index order is warp by warp, block by block, lane by lane
        const int E = G * nblk, per_lane = (E + 31) / 32;
        const float2* tf = sh.tab;
        float rl = 0.f, pl = 0.f;
        for (int e = lane * per_lane; e < min(E, (lane + 1) * per_lane); ++e) {
            rl += tf[e].x;
            pl += tf[e].y;
        }
        const float RM = warp_sum(rl), PM = warp_sum(pl);
        const bool use_r = !bonus && RM > 0.f;       // a residual without mass: draw from p
        const float wl = use_r ? rl : pl;
        float target = u_res * (use_r ? RM : PM);
        float incl = wl;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += t;
        }
        float run = incl - wl;
        int hit = -1, last = -1;
        float hbase = 0.f, lbase = 0.f;
        for (int e = lane * per_lane; e < min(E, (lane + 1) * per_lane); ++e) {
            const float w = use_r ? tf[e].x : tf[e].y;
            if (w > 0.f) {
                last = e;
                lbase = run;
                if (hit < 0 && run + w > target) {
                    hit = e;
                    hbase = run;
                }
            }
            run += w;
        }
        const unsigned mh = __ballot_sync(0xFFFFFFFFu, hit >= 0), ml = __ballot_sync(0xFFFFFFFFu, last >= 0);
        int ent = -1;
        float base = 0.f;
        if (mh) {
            const int l = __ffs(mh) - 1;
            ent = __shfl_sync(0xFFFFFFFFu, hit, l);
            base = __shfl_sync(0xFFFFFFFFu, hbase, l);
        } else if (ml) {          // rounding left no crossing: last block with mass, last token with mass
            const int l = 31 - __clz(ml);
            ent = __shfl_sync(0xFFFFFFFFu, last, l);
            base = __shfl_sync(0xFFFFFFFFu, lbase, l);
            target = INFINITY;
        }
        if (ent >= 0) {
            const int g = ent / nblk, blk = ent - g * nblk;
            const int a0 = (int)((long long)g * NI / G) + blk * per, a1 = min((int)((long long)(g + 1) * NI / G), a0 + per);
            float runw = base;
            int last_pos = -1;
            for (int it = a0; it < a1 && tok < 0; it += 4) {
                uint4 a[4], d[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int u = 32 * (it + k) + lane;
                    a[k] = it + k < a1 ? load(row_t, u) : U::none4();
                    d[k] = (it + k < a1 && !bonus) ? load(row_d, u) : U::none4();
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (tok < 0 && it + k < a1) {          // same for the whole warp
                        const int u = 32 * (it + k) + lane;
                        float pv[N], rv[N];
                        weights(a[k], d[k], u, pv, rv);
                        float ls = 0.f;
#pragma unroll
                        for (int j = 0; j < N; ++j) {
                            if (!use_r) rv[j] = pv[j];
                            ls += rv[j];
                        }
                        float li = ls;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const float t = __shfl_up_sync(0xFFFFFFFFu, li, o);
                            if (lane >= o) li += t;
                        }
                        float cc = runw + (li - ls);
                        int h = -1;
#pragma unroll
                        for (int j = 0; j < N; ++j) {
                            cc += rv[j];
                            if (rv[j] > 0.f) {
                                last_pos = u * N + j;
                                if (h < 0 && cc > target) h = u * N + j;
                            }
                        }
                        const unsigned m2 = __ballot_sync(0xFFFFFFFFu, h >= 0);
                        if (m2) tok = __shfl_sync(0xFFFFFFFFu, h, __ffs(m2) - 1);
                        runw += __shfl_sync(0xFFFFFFFFu, li, 31);
                    }
                }
            }
            if (tok < 0) tok = __reduce_max_sync(0xFFFFFFFFu, last_pos);
        }
    }
    if (lane == 0) {
        p.accept_len[b] = i;
        p.next_token[b] = tok;
    }
}

// ---- greedy: one CTA per sequence --------------------------------------------------------------
// Longest prefix of candidates that equal the target's choice argmax p_i (lowest index among equal
// maxima; a row with NaN, +inf or no finite logit has no choice, -1, and matches nothing).
struct GreedyParams {
    const float4* seg;
    const int32_t* x;
    const int32_t* draft_len;
    int32_t* accept_len;
    int32_t* next_token;
    int32_t* argmax_out;                         // nullable
    uint32_t* status;
    uint32_t* next;                              // row_stream_kernel's counter, put back to 0 here
    int32_t Kmax, seg_bits;
};

constexpr int kGThreads = 256;

__global__ void __launch_bounds__(kGThreads) greedy_finish_kernel(GreedyParams p) {
    __shared__ int32_t choice[ADASD_KMAX_LIMIT + 1];
    const int b = (int)blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int K = p.Kmax, K1 = K + 1, R = 2 * K + 1, segs = 1 << p.seg_bits;
    pdl_trigger();
    int kt = p.draft_len ? __ldcg(p.draft_len + b) : K;
    kt = max(0, min(kt, K));
    const int x = lane < kt ? __ldcg(p.x + (size_t)b * K + lane) : 0;
    pdl_wait();
    if (b == 0 && threadIdx.x == 0) *p.next = 0u;
    constexpr int W = kGThreads / 32;
    for (int i0 = warp; i0 <= kt; i0 += 3 * W) {     // three rows of a warp asked for before the first is folded
        SegPair sp[3];
#pragma unroll
        for (int k = 0; k < 3; ++k)
            sp[k] = load_segments(p.seg + (((size_t)b * R + i0 + k * W) << p.seg_bits), segs, i0 + k * W <= kt, -INFINITY);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int i = i0 + k * W;
            if (i <= kt) {
                const float v = warp_max_f32(fmaxf(sp[k].a.x, sp[k].b.x));
                // segments are in index order: the lowest index of those that have the maximum
                const int ia = sp[k].a.x == v ? __float_as_int(sp[k].a.z) : 0x7FFFFFFF, ib = sp[k].b.x == v ? __float_as_int(sp[k].b.z) : 0x7FFFFFFF;
                int am = __reduce_min_sync(0xFFFFFFFFu, min(ia, ib));
                if (segments_bad(sp[k], v, -INFINITY)) am = -1;
                if (lane == 0) {
                    choice[i] = am;
                    if (p.argmax_out) p.argmax_out[(size_t)b * K1 + i] = am;
                    if (am < 0) atomicOr(p.status, ADASD_STATUS_NAN);
                }
            }
        }
    }
    __syncthreads();
    if (warp != 0) return;
    const unsigned m = __ballot_sync(0xFFFFFFFFu, lane < kt && x != choice[lane]);
    const int w = m ? (__ffs(m) - 1) : kt;
    if (lane == 0) {
        p.accept_len[b] = w;
        p.next_token[b] = choice[w];
    }
}

}  // namespace adasd
