// Verification kernels for sm_100a for rows the warp-specialised kernel does not take (adasd_verify on fp32
// rows, rows off 16-byte boundaries, short ones): every candidate position (b,i) = target row p_i + draft row
// q_i of a round, bf16 or fp32, any length, alignment and stride.
//
// A position is swept twice, by two launches of sweep_kernel.  Sweep 1 forms 2^t, t = (z - max) log2 e, with a
// running maximum and adds up S = sum 2^t and T = sum 2^t t of both rows; sweep 2, with the row totals known,
// forms the divergence from non-negative terms of p = 2^t_p / S_p and q, and scans for the token y_i ~ p_i.
//
// Either sweep of a position is cut into segments; a WARP takes a segment at a time (an "item"), its rows
// coming through a ring of bulk copies that runs on across items.  The warps never meet: sweep 1 leaves every
// segment's statistics in a table, a warp of sweep 2 folds those of its position when it takes the item on,
// and the last warp of a position (a counter in device memory) publishes its distance.  Nothing in
// a launch waits for anything but its own copies.
//
// What bounds them: sweep 1 HBM, sweep 2 issue slots and the special-function pipe, for few rows the latency of
// two launches and the tail's.  adasd_verify, three-pass cluster kernel before -> now: fp32 V=128256
// B=16 K=5 125 -> 51 us (90 MB), B=64 K=4 356 -> 132 (297 MB), fp32 V=32000 B=1 K=5 24.6 -> 17.5,
// bf16 V=50257 B=8 K=5 59.7 -> 26.9, B=64 160 -> 68.  (One launch in which sweep 2 follows sweep 1 at a distance
// that keeps the rows in L2 was slower, 84 to 110 us for the first: warps in different sweeps evict one
// another's instructions, and those that wait hold up items that others wait for.)
#pragma once

#include "adasd_async.cuh"

namespace adasd {

constexpr int kSweepW = 8;                       // warps per CTA, two CTAs per SM
constexpr int kSweepThreads = kSweepW * 32;
constexpr int kSweepIt = 4;                      // iterations (32 lanes x 16 bytes of each row) per chunk
constexpr int kSweepRing = 3;
constexpr int kSweepRowB = kSweepIt * 512 + 16;  // one row's chunk (+ one unit: unaligned draft rows)
constexpr int kSweepStage = 2 * kSweepRowB;
constexpr int kSweepSmem = kSweepW * kSweepRing * kSweepStage;
constexpr int kSweepMaxSegs = 64;                // segments of a position, two to a lane of the folding warp
constexpr int kSweepItems = 8;                   // descriptions of items a warp keeps (it holds at most five)

// Statistics of both rows over a segment: largest logits (kFloorL: none), S and T under them.
struct __align__(16) SegStats {
    float vt, St, Tt, vd;
    float Sd, Td;
    uint32_t bad;                 // 1: NaN / +inf / expired wait
    uint32_t pad;
};

struct SweepTables {
    SegStats* seg1;               // [positions][segments]
    float2* seg2;                 // [positions][segments] sweep-2 sums: of s phi(u), of 2^t_p 2^t_q
    uint32_t* done;               // [positions] items done of sweep 2 (0 between rounds)
    uint32_t* next;               // [2] items drawn so far by either sweep (0 before its launch)
    int32_t segs;                 // segments of a position, each of one chunk or more
};

// An item as its warp describes it to itself when it asks for the first copy.
struct __align__(16) SweepItem {
    int32_t pos;                  // b (Kmax + 1) + i; -1: no more items
    int32_t mt;                   // elements between the target row's 16-byte boundary (its unit 0) and the row
    int32_t sd;                   // draft row: elements between a 16-byte boundary and the element that pairs with unit 0's first
    int32_t seg, ch0, ch1;        // segment, and its chunks
    int32_t bonus;                // the sequence's bonus row (target row only)
    float cut_t, cut_d;           // adjusted distribution: the rows' cutoff logits
    // sweep 2, bonus row: largest logit; this segment holds the crossing of u S: weight (under vt) before it, and where that lies
    float vt, base, target;
};
// A warp's place among the items.
struct __align__(16) SweepWarp {
    SweepItem items[kSweepItems];
    unsigned long long bar[kSweepRing];
    uint32_t blk_rank;            // positions before the block of 32 sequences it is in, the block
    int32_t blk_b;
    int32_t n_items;              // items described
};
// What the copies of an item need (lane 0: target row, lane 1: draft row): base, the granules that hold
// elements, chunks.
struct ItemRows {
    unsigned long long src;
    int32_t glo, ghi, ch, ch1;    // ch < 0: no more items
};

// A position's totals from its segments, by a whole warp.
struct PosTotals {
    float vt, St, vd, Sd, base, target;
    int32_t sel;                  // the segment with the crossing of u S, -1: the position is unusable
};
template <bool WARPED>
__device__ __forceinline__ PosTotals fold_position(const VerifyParams& p, const SweepTables& q, int pos, float u) {
    const int lane = threadIdx.x & 31, segs = q.segs;
    const float c1 = WARPED ? p.c1 : kLog2e;
    const float4* sp = reinterpret_cast<const float4*>(q.seg1 + (size_t)pos * segs);
    const float4 none0 = make_float4(kFloorL, 0.f, 0.f, kFloorL), none1 = make_float4(0.f, 0.f, 0.f, 0.f);
    const bool in0 = lane < segs, in1 = lane + 32 < segs;
    const float4 a0 = in0 ? __ldcg(sp + 2 * lane) : none0, a1 = in0 ? __ldcg(sp + 2 * lane + 1) : none1;
    const float4 b0 = in1 ? __ldcg(sp + 2 * (lane + 32)) : none0, b1 = in1 ? __ldcg(sp + 2 * (lane + 32) + 1) : none1;
    PosTotals t;
    t.vt = warp_max_f32(fmaxf(a0.x, b0.x));
    t.vd = warp_max_f32(fmaxf(a0.w, b0.w));
    const float w0 = ex2((a0.x - t.vt) * c1) * a0.y, w1 = ex2((b0.x - t.vt) * c1) * b0.y;
    float d0 = ex2((a0.w - t.vd) * c1) * a1.x, d1 = ex2((b0.w - t.vd) * c1) * b1.x;
    const bool bad = __any_sync(0xFFFFFFFFu, (__float_as_uint(a1.z) | __float_as_uint(b1.z)) & 1u) || !(t.vt > kFloorL) || !(t.vd > kFloorL);
    // running weights: lane by lane over the first 32 segments, then over the others.  Lane 31's prefix adds the same
    // pairs as the exchange of the draft row's sums, so that identical rows have identical totals and a distance of
    // exactly 0
    float i0 = w0, i1 = w1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const float t0 = __shfl_up_sync(0xFFFFFFFFu, i0, o), t1 = __shfl_up_sync(0xFFFFFFFFu, i1, o);
        d0 += __shfl_xor_sync(0xFFFFFFFFu, d0, o);
        d1 += __shfl_xor_sync(0xFFFFFFFFu, d1, o);
        if (lane >= o) {
            i0 += t0;
            i1 += t1;
        }
    }
    i1 += __shfl_sync(0xFFFFFFFFu, i0, 31);
    t.St = __shfl_sync(0xFFFFFFFFu, i1, 31);
    t.Sd = d1 + d0;
    t.sel = -1;
    t.base = 0.f;
    t.target = u * t.St;
    if (!bad) {
        // the segment with the crossing of u S in index order; if rounding leaves none, the last with mass
        const unsigned h0 = __ballot_sync(0xFFFFFFFFu, w0 > 0.f && i0 > t.target), h1 = __ballot_sync(0xFFFFFFFFu, w1 > 0.f && i1 > t.target);
        if (h0) t.sel = __ffs(h0) - 1;
        else if (h1) t.sel = 32 + __ffs(h1) - 1;
        else {
            const unsigned m0 = __ballot_sync(0xFFFFFFFFu, w0 > 0.f), m1 = __ballot_sync(0xFFFFFFFFu, w1 > 0.f);
            t.sel = m1 ? 32 + 31 - __clz(m1) : 31 - __clz(m0);
            t.target = INFINITY;
        }
        t.base = __shfl_sync(0xFFFFFFFFu, t.sel < 32 ? i0 - w0 : i1 - w1, t.sel & 31);
    }
    return t;
}

// Entropies and log-sum-exps of one position, worked out in float64 by a whole warp (its first segment's).
// none: the position is unusable.
template <bool WARPED>
__device__ __noinline__ void publish_entropies(const VerifyParams& p, const SweepTables& q, int pos, bool bonus, bool none, float vt, float vd) {
    const int lane = threadIdx.x & 31, segs = q.segs;
    const double c1 = (double)(WARPED ? p.c1 : kLog2e);
    const SegStats* const seg = q.seg1 + (size_t)pos * segs;
    // S = sum f_c S_c, T = sum f_c (T_c + d_c S_c) with d_c = (v_c - v) log2 e / T, f_c = 2^d_c
    double St = 0.0, Tt = 0.0, Sd = 0.0, Td = 0.0;
    for (int s = lane; s < segs; s += 32) {
        const float4 e0 = __ldcg(reinterpret_cast<const float4*>(seg + s)), e1 = __ldcg(reinterpret_cast<const float4*>(seg + s) + 1);
        if (e0.x > kFloorL) {
            const double d = ((double)e0.x - (double)vt) * c1, f = exp2(d);
            St += f * (double)e0.y;
            Tt += f * ((double)e0.z + d * (double)e0.y);
        }
        if (e0.w > kFloorL) {
            const double d = ((double)e0.w - (double)vd) * c1, f = exp2(d);
            Sd += f * (double)e1.x;
            Td += f * ((double)e1.y + d * (double)e1.x);
        }
    }
    St = warp_sum_f64(St);
    Tt = warp_sum_f64(Tt);
    Sd = warp_sum_f64(Sd);
    Td = warp_sum_f64(Td);
    // lane 0: the target row, lane 1: the draft row
    if (lane >= (bonus ? 1 : 2)) return;
    const double kLn2d = 0.69314718055994530942, S = lane ? Sd : St, lS = log2(S);
    const float H = none ? NAN : (float)(kLn2d * (lS - (lane ? Td : Tt) / S));
    const float lse = none ? NAN : (float)(kLn2d * ((double)(lane ? vd : vt) * c1 + lS));
    const size_t id = (size_t)(pos / (p.Kmax + 1)) * p.Kmax + pos % (p.Kmax + 1);
    if (lane == 0) {
        if (p.user.H_t) p.user.H_t[pos] = H;
        if (p.user.lse_t) p.user.lse_t[pos] = lse;
    } else {
        p.sc.H_d[id] = H;
        if (p.user.H_d) p.user.H_d[id] = H;
        if (p.user.lse_d) p.user.lse_d[id] = lse;
    }
}

// D_JS and the distance of one position, by one lane.  A: sum s phi(u), PQ: 0 where the supports are disjoint.
__device__ __forceinline__ void publish_distance(const VerifyParams& p, int pos, bool none, double A, float PQ) {
    float jsd = fminf((float)(0.25 * A), kLn2);
    if (!(PQ > 0.f)) jsd = kLn2;                                // disjoint supports: ln 2
    float dist = jsd >= kLn2 ? 1.f : fminf(sqrtf(jsd / kLn2), 1.f);
    if (none) jsd = dist = NAN;
    const size_t id = (size_t)(pos / (p.Kmax + 1)) * p.Kmax + pos % (p.Kmax + 1);
    p.sc.dist[id] = dist;
    if (p.user.jsd) p.user.jsd[id] = jsd;
    if (p.user.dist) p.user.dist[id] = dist;
}

// Row sums of sweep 1 under the running maximum v (warp-wide; kFloorL: nothing finite so far).  Under a temperature T
// adds up 2^t (z - v) and is scaled once a segment: z - v is finite, t for small temperatures is not.
template <bool WARPED>
struct RowSums {
    float v;
    float2 S, T;
    __device__ __forceinline__ void raise(float x, float floor_v, float c1) {      // a larger maximum: rescale
        if (x > v && x > floor_v) {
            const float dz = v > kFloorL ? v - x : kFloorL, d = WARPED ? dz : dz * c1, f = ex2(dz * c1);
            T.x = f * fmaf(d, S.x, T.x);
            T.y = f * fmaf(d, S.y, T.y);
            S.x *= f;
            S.y *= f;
            v = x;
        }
    }
    // t is exactly 0 for the largest logit, so that a one-hot row gets S = 1, T = 0 and H = 0 exactly
    template <typename U>
    __device__ __forceinline__ void add(const uint4& w, float2 nv2, float2 L2) {
        float2 z[U::N / 2];
        U::unpack(w, z);
#pragma unroll
        for (int j = 0; j < U::N / 2; ++j) {
            const float2 d = __fadd2_rn(z[j], nv2), t = __fmul2_rn(d, L2);
            const float2 e = make_float2(ex2(t.x), ex2(t.y));
            S = __fadd2_rn(S, e);
            T = __ffma2_rn(e, WARPED ? d : t, T);
        }
    }
};

// Sweep-2 terms of one unit of both rows: the overlap indicator PQ += 2^t_p 2^t_q, and the divergence from
// non-negative terms, D_JS = 1/4 sum s phi(u) with s = p + q, u = |q - p| / s and
// phi(u) = (1-u) ln(1-u) + (1+u) ln(1+u), which do not cancel however close the rows are:
//   u < 1/2: u^2 + u^4/6 + u^6/15 + u^8/28 + u^10/45 (low by at most 1.7e-5 of phi, at u = 1/2);
//   else   : 2 ln(1+u) - (1-u) |ln(p / q)|, the logarithm of p / q from the logits and 1 - u = 2 min(p,q) / s.
// Four special-function results a pair.
struct PairConsts {
    float2 nt2, nd2, at2, ad2, L2;
    float dl;                     // log2 (rd / rt): log2 (q / p) = t_q - t_p + dl
};
template <typename U>
__device__ __forceinline__ void pair_add(const uint4& Tw, const uint4& Dw, const PairConsts& c, float2& A2, float2& PQ2) {
    float2 z[U::N / 2], y[U::N / 2];
    U::unpack_raw(Tw, z);
    U::unpack_raw(Dw, y);
#pragma unroll
    for (int j = 0; j < U::N / 2; ++j) {
        const float2 t = __fmul2_rn(__fadd2_rn(z[j], c.nt2), c.L2), r = __fmul2_rn(__fadd2_rn(y[j], c.nd2), c.L2);
        const float2 a = make_float2(ex2(t.x), ex2(t.y)), d = make_float2(ex2(r.x), ex2(r.y));
        const float2 pp = __fmul2_rn(a, c.at2), qq = __fmul2_rn(d, c.ad2);
        const float2 ss = __fadd2_rn(__fadd2_rn(pp, pair2(kTiny)), qq);
        const float2 df = __ffma2_rn(pp, pair2(-1.f), qq);                                // q - p
        const float2 rs = make_float2(rcp_approx(ss.x), rcp_approx(ss.y));
        const float2 u = __fmul2_rn(df, rs), w = __fmul2_rn(u, u);
        float2 f = __ffma2_rn(w, pair2(1.f / 45.f), pair2(1.f / 28.f));
        f = __ffma2_rn(f, w, pair2(1.f / 15.f));
        f = __ffma2_rn(f, w, pair2(1.f / 6.f));
        f = __ffma2_rn(f, w, pair2(1.f));
        f = __fmul2_rn(f, w);
        // (fminf: the difference of two logits of -inf is NaN, and 0 times it has to be 0)
        const float hx = fminf(pp.x, qq.x) * rs.x * fminf(fabsf(r.x - t.x + c.dl), 1e30f);
        const float hy = fminf(pp.y, qq.y) * rs.y * fminf(fabsf(r.y - t.y + c.dl), 1e30f);
        const float gx = 2.f * kLn2 * (lg2(1.f + fabsf(u.x)) - hx), gy = 2.f * kLn2 * (lg2(1.f + fabsf(u.y)) - hy);
        A2 = __ffma2_rn(ss, make_float2(w.x < 0.25f ? f.x : gx, w.y < 0.25f ? f.y : gy), A2);
        PQ2 = __ffma2_rn(a, d, PQ2);
    }
}

// Describes item number j (of P segs; position by position, sequence by sequence) to the warp, in sweep 2 the
// next one that has something to do: a bonus row only needs the scan of one segment.  (A function of its
// own, like publish_entropies: the loops keep the registers.)
template <typename T, bool ALIGNED, bool WARPED, bool SECOND>
__device__ __noinline__ ItemRows sweep_item(const VerifyParams& p, const SweepTables& q, SweepWarp* w, uint32_t P, int NC, uint32_t j) {
    constexpr int N = Unit<T>::N;
    const int lane = threadIdx.x & 31, K = p.Kmax, K1 = K + 1;
    const uint32_t segs = (uint32_t)q.segs;
    SweepItem d;
    ItemRows r;
    d.pos = -1;
    r.src = 0ull;
    r.glo = r.ghi = r.ch1 = 0;
    r.ch = -1;
    for (; j < P * segs;) {
        const uint32_t rank = j / segs;
        const int seg = (int)(j - rank * segs);
        int b, i;
        bool bonus;
        if (!p.draft_len) {
            b = (int)(rank / (uint32_t)K1);
            i = (int)rank - b * K1;
            bonus = i == K;
        } else {                                     // a block of 32 sequences at a time; the ranks only go up
            uint32_t blk_rank = w->blk_rank;
            int blk_b = w->blk_b, cnt, incl;
            for (;;) {
                cnt = blk_b + lane < p.B ? max(0, min(__ldcg(p.draft_len + blk_b + lane), K)) + 1 : 0;
                incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                    if (lane >= o) incl += t;
                }
                const uint32_t tot = (uint32_t)__shfl_sync(0xFFFFFFFFu, incl, 31);
                if (rank < blk_rank + tot) break;    // (rank < P: the block exists)
                blk_rank += tot;
                blk_b += 32;
            }
            __syncwarp();
            if (lane == 0) {
                w->blk_rank = blk_rank;
                w->blk_b = blk_b;
            }
            __syncwarp();
            const int o = (int)(rank - blk_rank);
            const int src = __ffs(__ballot_sync(0xFFFFFFFFu, incl > o)) - 1;
            const int n = __shfl_sync(0xFFFFFFFFu, cnt, src);
            b = blk_b + src;
            i = o - (__shfl_sync(0xFFFFFFFFu, incl, src) - n);
            bonus = i == n - 1;
        }
        const int pos = b * K1 + i;
        if (SECOND && bonus) {
            pdl_wait();                              // (the warp's first item is described before the wait)
            const PosTotals t = fold_position<WARPED>(p, q, pos, __ldcg(p.u_target + pos));
            const bool none = t.sel < 0;
            if (seg == 0) {
                publish_entropies<WARPED>(p, q, pos, true, none, t.vt, t.vd);
                if (none && lane == 0) {
                    atomicOr(p.st.status, ADASD_STATUS_NAN);
                    p.sc.y[pos] = -1;
                    if (p.user.y) p.user.y[pos] = -1;
                }
            }
            if (t.sel != seg) {
                if (lane == 0) j = gridDim.x * kSweepW + atomicAdd(q.next + 1, 1u);
                j = __shfl_sync(0xFFFFFFFFu, j, 0);
                continue;
            }
            d.vt = t.vt;
            d.base = t.base;
            d.target = t.target;
        }
        d.pos = pos;
        d.seg = seg;
        d.bonus = bonus ? 1 : 0;
        d.ch0 = (int)((uint32_t)(seg * NC) / segs);
        d.ch1 = (int)((uint32_t)((seg + 1) * NC) / segs);
        const unsigned long long at = reinterpret_cast<unsigned long long>(
            reinterpret_cast<const T*>(p.zt) + (long long)b * p.t_seq + (long long)i * p.t_row);
        const unsigned long long ad = reinterpret_cast<unsigned long long>(
            reinterpret_cast<const T*>(p.zd) + (long long)b * p.d_seq + (long long)(bonus ? 0 : i) * p.d_row);
        const unsigned long long bt = ALIGNED ? at : at & ~15ull;
        d.mt = ALIGNED ? 0 : (int)((at & 15ull) / sizeof(T));
        const unsigned long long qd = ad - (unsigned long long)d.mt * sizeof(T);
        const unsigned long long bd = ALIGNED ? ad : qd & ~15ull;
        d.sd = ALIGNED ? 0 : (int)((qd & 15ull) / sizeof(T));
        d.cut_t = (WARPED && p.cut_t) ? __ldcg(p.cut_t + pos) : -INFINITY;
        d.cut_d = (WARPED && p.cut_d && !bonus) ? __ldcg(p.cut_d + (size_t)b * K + i) : -INFINITY;
        const int e0 = d.sd + d.mt;                  // elements between bd and the draft row
        r.src = lane == 0 ? bt : bd;
        r.glo = lane == 0 || ALIGNED ? 0 : e0 / N;
        r.ghi = lane == 0 ? (d.mt + p.V + N - 1) / N : (bonus ? 0 : (e0 + p.V + N - 1) / N);
        r.ch = d.ch0;
        r.ch1 = d.ch1;
        break;
    }
    if (lane == 0) {
        w->items[w->n_items & (kSweepItems - 1)] = d;
        ++w->n_items;
    }
    __syncwarp();
    return r;
}

// ALIGNED: every row starts on a 16-byte boundary.  WARPED: an adjusted distribution is set (Sec. 2.1.1); the
// ordinary instantiation carries none of its code.
// A wait that expires (a copy that never lands) sets ADASD_STATUS_TIMEOUT; the warp stops copying, waits
// (bounded) for the copies it has in flight, and reports the items it still holds as unusable.
template <typename T, bool ALIGNED, bool WARPED, bool SECOND>
__global__ void __launch_bounds__(kSweepThreads, 2) sweep_kernel(const __grid_constant__ VerifyParams p, const __grid_constant__ SweepTables q) {
    using U = Unit<T>;
    constexpr int N = U::N, NP = N / 2, IT = kSweepIt;
    const float floor_v = N == 8 ? ADASD_FLOOR_BF : kFloor;
    extern __shared__ __align__(128) unsigned char dyn_smem[];
    __shared__ SweepWarp warps_s[kSweepW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int K = p.Kmax;
    const float c1 = WARPED ? p.c1 : kLog2e;         // log2 e / temperature
    // chunks of a position (unaligned rows: one unit more, wherever the row starts)
    const int NC = ((ALIGNED ? (p.V + N - 1) / N : (p.V + 2 * N - 2) / N) + 32 * IT - 1) / (32 * IT);
    // (few items: spread over the SMs)
    const uint32_t GW = gridDim.x * kSweepW, gw = (uint32_t)warp * gridDim.x + blockIdx.x;
    unsigned char* const ring = dyn_smem + (size_t)warp * (kSweepRing * kSweepStage);
    SweepWarp* const sw = warps_s + warp;
    if (lane == 0) {
        for (int s = 0; s < kSweepRing; ++s) mbar_init(reinterpret_cast<uint64_t*>(&sw->bar[s]), 2);   // (one arrival per row)
        sw->blk_rank = 0u;
        sw->blk_b = 0;
        sw->n_items = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    if (!SECOND) {
        pdl_wait();
        pdl_trigger();
    }
    // active positions of the round (i <= K_b)
    uint32_t P = 0;
    if (p.draft_len) {
        for (int b = lane; b < p.B; b += 32) P += (uint32_t)max(0, min(__ldcg(p.draft_len + b), K)) + 1u;
        P = __reduce_add_sync(0xFFFFFFFFu, P);
    } else {
        P = (uint32_t)p.B * (uint32_t)(K + 1);
    }

    // ---- asking for rows ------------------------------------------------------------------
    // A warp starts with item gw and draws the others, a few chunks before it needs them.
    uint32_t drawn = 0u;                             // (in lane 0)
    bool alive = true, pending = false;
    auto draw = [&]() {
        if (lane == 0) drawn = atomicAdd(q.next + (SECOND ? 1 : 0), 1u) + GW;
        pending = true;
    };
    ItemRows rows = sweep_item<T, ALIGNED, WARPED, SECOND>(p, q, sw, P, NC, gw);
    int is = 0, n_issued = 0, n_taken = 0;
    auto ask = [&](int ch) {                         // ring slot `is` gets a chunk of both rows
        if (lane < 2) {
            // (unaligned draft rows: one granule more)
            const int u0 = 32 * IT * ch, a = ALIGNED ? u0 : max(u0, rows.glo), e = min(u0 + 32 * IT + (ALIGNED ? 0 : lane), rows.ghi);
            const uint32_t bytes = (uint32_t)max(e - a, 0) * 16u;
            uint64_t* bar = reinterpret_cast<uint64_t*>(&sw->bar[is]);
            mbar_expect_tx(bar, bytes);
            if (bytes)
                bulk_g2s(ring + is * kSweepStage + lane * kSweepRowB + (a - u0) * 16,
                         reinterpret_cast<const unsigned char*>(rows.src) + (size_t)a * 16, bytes, bar);
        }
        __syncwarp();
        ++n_issued;
        is = is + 1 == kSweepRing ? 0 : is + 1;
    };
    auto issue = [&](bool asked) {                   // the next chunk
        if (rows.ch < 0) return;
        if (!asked) ask(rows.ch);
        if (++rows.ch == rows.ch1) {
            if (!pending) draw();
            pending = false;
            rows = sweep_item<T, ALIGNED, WARPED, SECOND>(p, q, sw, P, NC, __shfl_sync(0xFFFFFFFFu, drawn, 0));
        } else if (rows.ch + 2 >= rows.ch1 && !pending) {
            draw();
        }
    };
    // Sweep 2 asks for its first copies before it waits for sweep 1: logits and window lengths were there
    // before that one began.
    int early = 0;
    if (SECOND) {
#pragma unroll 1
        for (; early < kSweepRing && rows.ch >= 0 && rows.ch + early < rows.ch1; ++early) ask(rows.ch + early);
        pdl_wait();
        pdl_trigger();
    }
    if (gw == 0 && lane == 0) q.next[SECOND ? 0 : 1] = 0u;       // the other sweep's counter, for its next launch
#pragma unroll 1
    for (int k = 0; k < kSweepRing; ++k) issue(k < early);

    int rs = 0;                                      // ring slot and phase of the next chunk to take
    uint32_t rph = 0;
    auto take = [&]() -> const unsigned char* {
        const unsigned char* sb = ring + rs * kSweepStage + lane * 16;
        bool ok = mbar_wait_bounded(reinterpret_cast<uint64_t*>(&sw->bar[rs]), rph);
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (!ok) {
            alive = false;
            rows.ch = -1;
            if (lane == 0) atomicOr(p.st.status, ADASD_STATUS_TIMEOUT);
        } else {
            ++n_taken;
        }
        if (++rs == kSweepRing) {
            rs = 0;
            rph ^= 1u;
        }
        return sb;
    };
    const float2 L2 = pair2(c1);

    for (int n = 0;; ++n) {
        if (!alive && n == *reinterpret_cast<volatile int32_t*>(&sw->n_items)) {     // one more number may have been drawn
            if (!pending) break;
            pending = false;
            sweep_item<T, ALIGNED, WARPED, SECOND>(p, q, sw, P, NC, __shfl_sync(0xFFFFFFFFu, drawn, 0));
        }
        const SweepItem& c = sw->items[n & (kSweepItems - 1)];
        const int pos = c.pos;
        if (pos < 0) break;
        const bool bonus = c.bonus != 0;
        const int seg = c.seg, ch0 = c.ch0, ch1 = c.ch1, mt = c.mt, sd = c.sd;
        const typename U::Cut cut_t = U::make_cut(WARPED ? c.cut_t : -INFINITY), cut_d = U::make_cut(WARPED ? c.cut_d : -INFINITY);
        // a chunk's units; at an edge, elements that do not exist (before the row, past its end) may be among them
        auto is_edge = [&](int ch) -> bool { return ch >= NC - (ALIGNED ? 1 : 2) || (!ALIGNED && ch == 0); };
        auto mask = [&](uint4& w, int ch, int k) {
            const int v0 = (32 * (ch * IT + k) + lane) * N - mt;           // first element of this lane's unit
            if (v0 < 0 || v0 + N > p.V) U::mask(w, -v0, p.V - v0);
        };
        auto unit_t = [&](const unsigned char* sb, int k) -> uint4 { return *reinterpret_cast<const uint4*>(sb + k * 512); };
        auto unit_d = [&](const unsigned char* sb, int k) -> uint4 {
            uint4 w = *reinterpret_cast<const uint4*>(sb + kSweepRowB + k * 512);
            if (!ALIGNED) w = U::realign(w, *reinterpret_cast<const uint4*>(sb + kSweepRowB + k * 512 + 16), sd);
            return w;
        };

        if (!SECOND) {
            RowSums<WARPED> rt = {kFloorL, make_float2(0.f, 0.f), make_float2(0.f, 0.f)}, rd = rt;
            uint32_t bad = 0u;
            auto chunk = [&](auto bonus_c, auto edge_c, int ch, const unsigned char* sb) {
                constexpr bool BONUS = decltype(bonus_c)::value, edge = decltype(edge_c)::value;
                typename U::Max m1 = U::max0(), m2 = U::max0();
#pragma unroll
                for (int k = 0; k < IT; ++k) {
                    uint4 w = unit_t(sb, k);
                    if (edge) mask(w, ch, k);
                    U::max_add(m1, w);
                    if (!BONUS) {
                        w = unit_d(sb, k);
                        if (edge) mask(w, ch, k);
                        U::max_add(m2, w);
                    }
                }
                const float xt = warp_max_f32(U::max_val(m1, bad));
                const float xd = BONUS ? xt : warp_max_f32(U::max_val(m2, bad));
                if (xt == INFINITY || xd == INFINITY) bad = 1u;
                rt.raise(xt, floor_v, c1);
                if (!BONUS) rd.raise(xd, floor_v, c1);
                const float2 nt2 = pair2(rt.v > kFloorL ? -rt.v : 0.f), nd2 = pair2(rd.v > kFloorL ? -rd.v : 0.f);
#pragma unroll 2
                for (int k = 0; k < IT; ++k) {
                    uint4 Tw = unit_t(sb, k);
                    if (edge) mask(Tw, ch, k);
                    if (WARPED) U::cut(Tw, cut_t);
                    rt.template add<U>(Tw, nt2, L2);
                    if (!BONUS) {
                        uint4 Dw = unit_d(sb, k);
                        if (edge) mask(Dw, ch, k);
                        if (WARPED) U::cut(Dw, cut_d);
                        rd.template add<U>(Dw, nd2, L2);
                    }
                }
            };
            for (int ch = ch0; ch < ch1 && alive; ++ch) {
                const unsigned char* sb = take();
                if (!alive) break;
                if (is_edge(ch)) {
                    if (bonus) chunk(std::true_type{}, std::true_type{}, ch, sb);
                    else chunk(std::false_type{}, std::true_type{}, ch, sb);
                } else {
                    if (bonus) chunk(std::true_type{}, std::false_type{}, ch, sb);
                    else chunk(std::false_type{}, std::false_type{}, ch, sb);
                }
                __syncwarp();
                issue(false);                        // the chunk has been read, its slot is free
            }
            if (!alive) bad = 1u;
            const float sc = WARPED ? c1 : 1.f, St = warp_sum(rt.S.x + rt.S.y), Tt = sc * warp_sum(rt.T.x + rt.T.y);
            const float Sd = bonus ? St : warp_sum(rd.S.x + rd.S.y), Td = bonus ? Tt : sc * warp_sum(rd.T.x + rd.T.y);
            bad = __reduce_or_sync(0xFFFFFFFFu, bad);
            if (lane == 0) {
                float4* w = reinterpret_cast<float4*>(q.seg1 + (size_t)pos * q.segs + seg);
                __stcg(w, make_float4(rt.v, St, Tt, bonus ? rt.v : rd.v));
                __stcg(w + 1, make_float4(Sd, Td, __uint_as_float(bad), 0.f));
            }
            continue;
        }

        // ================================== sweep 2 =========================================
        float vt, run, target;                       // scan: weight before the chunk, where the sample's crossing lies
        bool scan = true, none = false;
        PairConsts pc;
        if (bonus) {
            vt = c.vt;
            run = c.base;
            target = c.target;
        } else {
            const PosTotals t = fold_position<WARPED>(p, q, pos, __ldcg(p.u_target + pos));
            none = t.sel < 0;
            vt = t.vt;
            run = t.base;
            target = t.target;
            scan = t.sel == seg;
            const float rt = __fdiv_rn(1.f, t.St), rd = __fdiv_rn(1.f, t.Sd);
            pc.nt2 = pair2(-vt);
            pc.nd2 = pair2(-t.vd);
            pc.at2 = pair2(rt);
            pc.ad2 = pair2(rd);
            pc.L2 = L2;
            pc.dl = lg2(t.St) - lg2(t.Sd);
            if (seg == 0) {
                publish_entropies<WARPED>(p, q, pos, false, none, vt, t.vd);
                if (none && lane == 0) {
                    publish_distance(p, pos, true, 0.0, 1.f);
                    atomicOr(p.st.status, ADASD_STATUS_NAN);
                    p.sc.y[pos] = -1;
                    if (p.user.y) p.user.y[pos] = -1;
                }
            }
        }
        float2 A2 = make_float2(0.f, 0.f), PQ2 = A2;
        int tok = -1, last = -1;
        // y_i: the first element (index order) where the running weight exceeds the target, else the last
        // one of the segment with weight.  A chunk's weight first, element by element only in the chunk that
        // holds the crossing.
        auto scan_unit = [&](const unsigned char* sb, int ch, int k, float (&e)[N]) {
            uint4 w = unit_t(sb, k);
            mask(w, ch, k);
            if (WARPED) U::cut(w, cut_t);
            float2 z[NP];
            U::unpack_raw(w, z);
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                e[2 * j] = ex2((z[j].x - vt) * c1);
                e[2 * j + 1] = ex2((z[j].y - vt) * c1);
            }
        };
        auto scan_chunk = [&](const unsigned char* sb, int ch) {
            float tot = 0.f, e[N];
#pragma unroll 1
            for (int k = 0; k < IT; ++k) {
                scan_unit(sb, ch, k, e);
                const int e0 = (32 * (ch * IT + k) + lane) * N - mt;
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    tot += e[j];
                    if (e[j] > 0.f) last = e0 + j;
                }
            }
            tot = warp_sum(tot);
            if (!(run + tot > target)) {
                run += tot;
                return;
            }
#pragma unroll 1
            for (int k = 0; k < IT && tok < 0; ++k) {
                scan_unit(sb, ch, k, e);
                float s = 0.f;
#pragma unroll
                for (int j = 0; j < N; ++j) s += e[j];
                float incl = s;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const float t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                    if (lane >= o) incl += t;
                }
                float cc = run + (incl - s);
                int hit = -1;
                const int e0 = (32 * (ch * IT + k) + lane) * N - mt;
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    cc += e[j];
                    if (e[j] > 0.f && hit < 0 && cc > target) hit = e0 + j;
                }
                const unsigned mh = __ballot_sync(0xFFFFFFFFu, hit >= 0);
                if (mh) tok = __shfl_sync(0xFFFFFFFFu, hit, __ffs(mh) - 1);
                run += __shfl_sync(0xFFFFFFFFu, incl, 31);
            }
        };
        auto chunk = [&](auto edge_c, int ch, const unsigned char* sb) {
            constexpr bool edge = decltype(edge_c)::value;
#pragma unroll 2
            for (int k = 0; k < IT; ++k) {
                uint4 Tw = unit_t(sb, k), Dw = unit_d(sb, k);
                if (edge) {
                    mask(Tw, ch, k);
                    mask(Dw, ch, k);
                }
                if (WARPED) {
                    U::cut(Tw, cut_t);
                    U::cut(Dw, cut_d);
                }
                pair_add<U>(Tw, Dw, pc, A2, PQ2);
            }
        };
        for (int ch = ch0; ch < ch1 && alive; ++ch) {
            const unsigned char* sb = take();
            if (!alive) break;
            if (scan && tok < 0) scan_chunk(sb, ch);
            if (!bonus && !none) {
                if (is_edge(ch)) chunk(std::true_type{}, ch, sb);
                else chunk(std::false_type{}, ch, sb);
            }
            __syncwarp();
            issue(false);                            // the chunk has been read, its slot is free
        }
        if (scan) {
            if (tok < 0) tok = __reduce_max_sync(0xFFFFFFFFu, last);
            if (!alive) tok = -1;
            if (lane == 0) {
                p.sc.y[pos] = tok;
                if (p.user.y) p.user.y[pos] = tok;
            }
        }
        if (bonus || none) continue;
        const float A = warp_sum(A2.x + A2.y), PQ = warp_sum(PQ2.x + PQ2.y);
        float2* const seg2 = q.seg2 + (size_t)pos * q.segs;
        uint32_t old = 0u;
        if (lane == 0) {
            __stcg(seg2 + seg, alive ? make_float2(A, PQ) : make_float2(NAN, 0.f));
            __threadfence();
            old = atomicAdd(q.done + pos, 1u);
        }
        if (__shfl_sync(0xFFFFFFFFu, old, 0) + 1u != (uint32_t)q.segs) continue;
        // the position's last segment
        __threadfence();
        if (lane == 0) q.done[pos] = 0u;             // ready for the next round
        const float2 s0 = lane < q.segs ? __ldcg(seg2 + lane) : make_float2(0.f, 0.f);
        const float2 s1 = lane + 32 < q.segs ? __ldcg(seg2 + lane + 32) : make_float2(0.f, 0.f);
        const double At = warp_sum_f64((double)s0.x + (double)s1.x);
        const float PQt = warp_sum(s0.y + s1.y);
        if (lane == 0) publish_distance(p, pos, At != At, At, PQt);
        __syncwarp();
    }
    // a warp that gave up still waits (bounded) for whatever it had in flight
    if (!alive)
        for (int k = n_taken; k < n_issued; ++k)
            mbar_wait_bounded(reinterpret_cast<uint64_t*>(&sw->bar[k % kSweepRing]), (uint32_t)(k / kSweepRing) & 1u);
}

}  // namespace adasd
