// Draft-step kernel for sm_100a (adasd_draft_entropy): bf16 or fp32 rows of any length, alignment and
// stride, every row read from HBM once.
//
//  * One cluster of P CTAs per row (P = 1, 2, 4 or 8, chosen so that the launch fills the SMs); the
//    warps of the cluster split the row into contiguous shares and stream them through a ring of
//    three 2 KB bulk copies each (bounded mbarrier waits).
//  * Per chunk: packed maximum, then 2^((z - max) log2 e) with the warp's running maximum (the sums
//    are rescaled when a chunk raises it), accumulating S = sum 2^t and T = sum 2^t t.  Sums over
//    short runs of chunks are kept in a table for sampling.  Greedy drafting: the index of the
//    maximum is looked up when a chunk raises it.
//  * The warps send their totals and tables to rank 0 over DSMEM; after one cluster barrier rank 0
//    forms H(q) = ln 2 (log2 S - T / S), the log-sum-exp and the stop flag H > T_G, finds the run of
//    chunks that holds the inverse-CDF crossing of u and scans just that again (from L2).
//
// What bounds it: a call is a few microseconds, of which the stream itself is about half; the rest is
// start-up, the first copy's latency and the serial end on one warp.  So the copies are asked for before
// the cluster's CTAs have met, what the end needs from global memory is asked for at the start, and a call
// signals its dependents at once: the next call's CTAs are set up while this one runs, and wait before
// they read anything.  Where the grid does not leave half of the SMs free, a second CTA per SM would put
// two rows of the same call on one SM and none on another (31 instead of 13 us a call for 128 rows of
// 151936 bf16 logits): draft_setup allows it only where it cannot.
#pragma once

#include "adasd_async.cuh"

namespace adasd {

constexpr int kDW = 8;                         // warps per CTA
constexpr int kDWBig = 16;                     // ... when the grid has one CTA per SM at most
constexpr int kDRingB = 6 * (4 * 512 + 16);     // bytes of a warp's ring: six chunks of 4 iterations (32 lanes x 16 bytes;
                                               // + one unit: rows off a 16-byte boundary) or three of 8
constexpr int kDMaxRing = 6;
constexpr int kDRuns = 8;                      // runs of chunks a warp's table holds
constexpr int kDMaxP = 8;
constexpr int kDMaxEntries = 64;               // warps per cluster, at most: two table entries per lane

template <int NW>
struct __align__(16) DraftShared {
    float2 run[kDMaxEntries][kDRuns];          // rank 0: (shift, sum of 2^t under it) of every run, by warp of the cluster
    float4 wpart[kDMaxEntries];                // rank 0: every warp's (largest logit, S, T, flags)
    float wtop[kDMaxEntries];                  // rank 0, greedy drafting: every warp's largest logit,
    int32_t widx[kDMaxEntries];                // its index
    unsigned long long bar[NW][kDMaxRing];
};

// NW warps per CTA: 8, or 16 (grids that do not fill the SMs twice); P * NW <= kDMaxEntries.
// IT: iterations of a chunk, 4 or (long shares: half the reductions) 8.
// ALIGNED: every row starts on a 16-byte boundary.  WARPED: an adjusted distribution is set
// (Sec. 2.1.1); the ordinary instantiation carries none of its code.
template <typename T, bool ALIGNED, int NW, int IT, bool WARPED>
__global__ void __launch_bounds__(NW * 32, NW == kDW ? 2 : 1) draft_step_kernel(DraftParams p) {
    using U = Unit<T>;
    constexpr int N = U::N, NP = N / 2;
    constexpr int kDRing = IT == 8 ? 3 : 6, kDStage = IT * 512 + 16;
    const float floor_v = N == 8 ? ADASD_FLOOR_BF : kFloor;
    extern __shared__ __align__(128) unsigned char dyn_smem[];
    __shared__ DraftShared<NW> sh;
    cg::cluster_group cluster = cg::this_cluster();
    const int P = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();
    const int b = blockIdx.x / P;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        for (int s = 0; s < kDRing; ++s) mbar_init(reinterpret_cast<uint64_t*>(&sh.bar[warp][s]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    if (p.early) pdl_trigger();
    // nothing the kernel ahead in the stream wrote (logits, active mask, window lengths) is touched before this
    pdl_wait();
    if (p.active && p.active[b] == 0) return;  // the same in every CTA of the cluster

    // the row in chunks of IT iterations (32 units of N elements each); this warp's share: whole chunks
    // [ch0, ch1), so that only the row's last chunk is ragged
    const int NU = (p.V + N - 1) / N, NC = (NU + 32 * IT - 1) / (32 * IT);
    const int G = P * NW, g = rank * NW + warp;
    auto share_begin = [&](int w) -> int { return (int)((long long)w * NC / G); };
    const int ch0 = share_begin(g), nch = share_begin(g + 1) - ch0;
    const int cpr = ((NC + G - 1) / G + kDRuns - 1) / kDRuns;                    // chunks per run
    const unsigned long long ra = reinterpret_cast<unsigned long long>(reinterpret_cast<const T*>(p.z) + (long long)b * p.row_stride);
    const unsigned char* const base = reinterpret_cast<const unsigned char*>(ALIGNED ? ra : ra & ~15ull);
    const int shift = ALIGNED ? 0 : (int)((ra & 15ull) / sizeof(T));
    const int g1 = (shift + p.V + N - 1) / N;                                    // granules that hold elements: [0, g1)
    unsigned char* const ring = dyn_smem + (size_t)warp * kDRingB;

    // self-test of the give-up path: the warp with the row's first chunk never asks for its first chunk and waits for it only
    // briefly, so the wait runs out with nothing in flight
    const bool expiring = (b == p.expire_row && ch0 == 0 && nch > 0);
    auto issue = [&](int c, int slot) {
        if (lane == 0 && c < nch && !(expiring && c == 0)) {
            const int u0 = 32 * IT * (ch0 + c), u1 = u0 + 32 * IT;
            const uint32_t bytes = (uint32_t)(min(ALIGNED ? u1 : u1 + 1, g1) - u0) * 16u;
            uint64_t* bar = reinterpret_cast<uint64_t*>(&sh.bar[warp][slot]);
            mbar_expect_tx(bar, bytes);
            bulk_g2s(ring + slot * kDStage, base + (size_t)u0 * 16, bytes, bar);
        }
    };
    for (int c = 0; c < kDRing; ++c) issue(c, c);
    // every CTA of the cluster runs before anyone writes into rank 0
    if (P > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    // what the last step of the row needs from global memory, asked for by the warp that will need it
    float u_row = 0.f, tg_row = 0.f;
    int32_t len_row = 0;
    if (g == 0) {
        if (p.u != nullptr) u_row = __ldcg(p.u + b);
        tg_row = p.st.T_G[b];
        if (p.draft_len) len_row = p.draft_len[b];          // (only this row's CTA ever writes it)
    }
    const float c1 = WARPED ? p.c1 : kLog2e;                // log2 e / temperature
    const typename U::Cut cut = U::make_cut((WARPED && p.cut) ? __ldcg(p.cut + b) : -INFINITY);
    const bool greedy = p.argmax != 0;
    if (P > 1) asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    DraftShared<NW>* const r0 = P > 1 ? cluster.map_shared_rank(&sh, 0) : &sh;

    // v: the largest logit so far (kFloorL while there is none): t = (z - v) log2 e is exactly 0 for it, so
    // that a one-hot row gets S = 1, T = 0 and H = 0 exactly.  Under a temperature T adds up 2^t (z - v), scaled once
    // at the end: z - v is finite, t for small temperatures is not
    float v = kFloorL;
    float top = -INFINITY;                                  // greedy drafting: the largest logit, finite but perhaps without
    int vi = -1;                                            // probability (a mask of the type's lowest value), and its index
    float2 S2 = make_float2(0.f, 0.f), T2 = S2, R2 = S2;    // lane partials under v; R2: S of the current run, not yet in S2
    uint32_t bad = 0u;
    const float2 L2 = pair2(c1);
    int run = 0, in_run = 0, cfail = -1;                    // cfail: chunk whose copy never landed
    int slot = 0;                                           // ring slot and phase of chunk c
    uint32_t ph = 0;
    for (int c = 0; c < nch; ++c) {
        bool ok = mbar_wait_bounded(reinterpret_cast<uint64_t*>(&sh.bar[warp][slot]), ph,
                                    expiring && c == 0 ? 64u : kCWaitSpins);
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (!ok) {
            if (lane == 0) atomicOr(p.st.status, ADASD_STATUS_TIMEOUT);
            bad = 1u;
            cfail = c;
            break;
        }
        const unsigned char* sb = ring + slot * kDStage + lane * 16;
        const int ci = (ch0 + c) * IT;
        auto load = [&](int k) -> uint4 {
            uint4 w = *reinterpret_cast<const uint4*>(sb + k * 512);
            if (!ALIGNED) w = U::realign(w, *reinterpret_cast<const uint4*>(sb + k * 512 + 16), shift);
            return w;
        };
        auto mask = [&](uint4& w, int k) {                  // the row's end
            const int e0 = (32 * (ci + k) + lane) * N;
            if (e0 >= p.V) w = U::none4();
            else if (e0 + N > p.V) U::mask(w, 0, p.V - e0);
        };
        const bool edge = ch0 + c == NC - 1;
        uint4 W[IT];
        typename U::Max mx = U::max0();
#pragma unroll
        for (int k = 0; k < IT; ++k) W[k] = load(k);
        if (edge) {
#pragma unroll
            for (int k = 0; k < IT; ++k) mask(W[k], k);
        }
#pragma unroll
        for (int k = 0; k < IT; ++k) U::max_add(mx, W[k]);
        const float lm = U::max_val(mx, bad);
        const float x = warp_max_f32(lm);
        if (x == INFINITY) bad = 1u;
        if (greedy && x > top) {                            // the lowest index of the chunk that has it
            top = x;
            int first = 0x7FFFFFFF;
            if (lm == x) {
#pragma unroll 1
                for (int k = IT - 1; k >= 0; --k) {
                    uint4 w = load(k);
                    mask(w, k);
                    float2 z[NP];
                    U::unpack_raw(w, z);
#pragma unroll
                    for (int j = NP - 1; j >= 0; --j) {
                        const int e = (32 * (ci + k) + lane) * N + 2 * j;
                        if (z[j].y == x) first = e + 1;
                        if (z[j].x == x) first = e;
                    }
                }
            }
            vi = __reduce_min_sync(0xFFFFFFFFu, first);
        }
        __syncwarp();
        issue(c + kDRing, slot);                              // the chunk has been read, its slot is free
        if (++slot == kDRing) {
            slot = 0;
            ph ^= 1u;
        }
        if (x > v && x > floor_v) {                         // a larger maximum: rescale what is summed
            const float dz = v > kFloorL ? v - x : kFloorL, d = WARPED ? dz : dz * c1, f = ex2(dz * c1);
            T2.x = f * fmaf(d, S2.x + R2.x, T2.x);
            T2.y = f * fmaf(d, S2.y + R2.y, T2.y);
            S2.x *= f;
            S2.y *= f;
            R2.x *= f;
            R2.y *= f;
            v = x;
        }
        const float nv = v > kFloorL ? -v : 0.f;
        const float2 nv2 = pair2(nv);
#pragma unroll
        for (int k = 0; k < IT; ++k) {
            if (WARPED) U::cut(W[k], cut);
            float2 z[NP];
            U::unpack(W[k], z);
#pragma unroll
            for (int j = 0; j < NP; ++j) {
                const float2 d = __fadd2_rn(z[j], nv2), t = __fmul2_rn(d, L2);
                const float2 e = make_float2(ex2(t.x), ex2(t.y));
                R2 = __fadd2_rn(R2, e);
                T2 = __ffma2_rn(e, WARPED ? d : t, T2);
            }
        }
        if (++in_run == cpr || c + 1 == nch) {
            S2 = __fadd2_rn(S2, R2);
            const float rs = warp_sum(R2.x + R2.y);
            if (lane == 0) r0->run[g][run] = make_float2(v, rs);
            R2 = make_float2(0.f, 0.f);
            in_run = 0;
            ++run;
        }
    }
    // a warp that gave up still waits (bounded) for what it had asked for and not taken; nothing may
    // land in this CTA after it has gone
    if (cfail >= 0)
        for (int c = cfail; c < min(cfail + kDRing, nch); ++c)
            if (!(expiring && c == 0))
                mbar_wait_bounded(reinterpret_cast<uint64_t*>(&sh.bar[warp][c % kDRing]), (uint32_t)(c / kDRing) & 1u);
    const float Sw = warp_sum(S2.x + S2.y), Tw = (WARPED ? c1 : 1.f) * warp_sum(T2.x + T2.y);
    bad = __reduce_or_sync(0xFFFFFFFFu, bad);
    if (lane >= run && lane < kDRuns) r0->run[g][lane] = make_float2(kFloorL, 0.f);      // runs this warp does not have
    if (lane == 0) {
        r0->wpart[g] = make_float4(v, Sw, Tw, __uint_as_float(bad));
        if (greedy) {
            r0->wtop[g] = top;
            r0->widx[g] = vi;
        }
    }
    // totals and tables of every CTA are in rank 0's shared memory
    if (P > 1) cluster.sync();
    else __syncthreads();
    if (g != 0) return;
    // (rank 0 only reads its own shared memory from here on; nobody writes to it any more)

    // row totals: lane l holds warp l of the cluster, and l + 32
    const float4 none = make_float4(kFloorL, 0.f, 0.f, 0.f);
    const float4 e0 = lane < G ? sh.wpart[lane] : none, e1 = lane + 32 < G ? sh.wpart[lane + 32] : none;
    const float Mr = warp_max_f32(fmaxf(e0.x, e1.x));
    float d0 = (e0.x - Mr) * c1, d1 = (e1.x - Mr) * c1;
    if (WARPED) {                                           // (finite: 0 times it occurs)
        d0 = fmaxf(d0, kFloor);
        d1 = fmaxf(d1, kFloor);
    }
    const float w0 = ex2(d0) * e0.y, w1 = ex2(d1) * e1.y;
    const float S = warp_sum(w0 + w1);
    const float Tt = warp_sum(ex2(d0) * fmaf(d0, e0.y, e0.z) + ex2(d1) * fmaf(d1, e1.y, e1.z));
    const uint32_t fl = __reduce_or_sync(0xFFFFFFFFu, __float_as_uint(e0.w) | __float_as_uint(e1.w));
    const bool rowbad = (fl & 1u) || !(Mr > kFloorL);
    const float lS = lg2(S);
    float H = kLn2 * (lS - Tt / S), lse = kLn2 * fmaf(Mr, c1, lS);
    if (rowbad) H = lse = NAN;

    int tok = -1;
    const bool sampling = !greedy && p.u != nullptr && p.token_out != nullptr;
    if (greedy && !(fl & 1u)) {
        // shares are in index order: the lowest index of those that have the maximum
        const float t0 = lane < G ? sh.wtop[lane] : -INFINITY, t1 = lane + 32 < G ? sh.wtop[lane + 32] : -INFINITY;
        const float t = warp_max_f32(fmaxf(t0, t1));
        const int i0 = lane < G && t0 == t ? sh.widx[lane] : 0x7FFFFFFF, i1 = lane + 32 < G && t1 == t ? sh.widx[lane + 32] : 0x7FFFFFFF;
        tok = t > -INFINITY ? __reduce_min_sync(0xFFFFFFFFu, min(i0, i1)) : -1;
    } else if (sampling && !rowbad) {
        // x ~ q: the crossing of u S in index order: first the share that holds it, then the run in it
        float target = u_row * S;
        float i0 = w0, i1 = w1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float t0 = __shfl_up_sync(0xFFFFFFFFu, i0, o), t1 = __shfl_up_sync(0xFFFFFFFFu, i1, o);
            if (lane >= o) {
                i0 += t0;
                i1 += t1;
            }
        }
        i1 += __shfl_sync(0xFFFFFFFFu, i0, 31);
        const unsigned h0 = __ballot_sync(0xFFFFFFFFu, w0 > 0.f && i0 > target);
        const unsigned h1 = __ballot_sync(0xFFFFFFFFu, w1 > 0.f && i1 > target);
        const unsigned m0 = __ballot_sync(0xFFFFFFFFu, w0 > 0.f), m1 = __ballot_sync(0xFFFFFFFFu, w1 > 0.f);
        int ent;
        if (h0) ent = __ffs(h0) - 1;
        else if (h1) ent = 32 + __ffs(h1) - 1;
        else {                   // rounding left no crossing: last share with mass, last token with mass
            ent = m1 ? 32 + 31 - __clz(m1) : 31 - __clz(m0);
            target = INFINITY;
        }
        const float ebase = ent < 32 ? __shfl_sync(0xFFFFFFFFu, i0 - w0, ent) : __shfl_sync(0xFFFFFFFFu, i1 - w1, ent - 32);
        const float2 rr = lane < kDRuns ? sh.run[ent][lane] : make_float2(kFloorL, 0.f);
        const float rw = ex2((rr.x - Mr) * c1) * rr.y;
        float incl = rw;
#pragma unroll
        for (int o = 1; o < kDRuns; o <<= 1) {
            const float t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += t;
        }
        const unsigned ch = __ballot_sync(0xFFFFFFFFu, rw > 0.f && ebase + incl > target);
        const unsigned cl = __ballot_sync(0xFFFFFFFFu, rw > 0.f);
        const int r = ch ? __ffs(ch) - 1 : 31 - __clz(cl | 1u);
        if (!ch) target = INFINITY;
        float cc0 = ebase + __shfl_sync(0xFFFFFFFFu, incl - rw, r);
        const int a0 = share_begin(ent) + r * cpr, a1 = min(share_begin(ent + 1), a0 + cpr);      // its chunks
        int last = -1;
        // the run again: a chunk at a time, lane l takes the units IT l .. IT l + IT - 1 of it, so that index order is
        // lane order: one prefix over the lanes' sums places the crossing in a lane, which walks its tokens
        const uint4* row = reinterpret_cast<const uint4*>(base);
        for (int ci = a0; ci < a1 && tok < 0; ++ci) {
            const int ub = 32 * IT * ci + lane * IT;
            uint4 W[IT + 1];
#pragma unroll
            for (int k = 0; k < IT + (ALIGNED ? 0 : 1); ++k)
                W[k] = ub + k < g1 ? __ldcg(row + ub + k) : U::none4();
            float e[IT][N], ls = 0.f;
#pragma unroll
            for (int k = 0; k < IT; ++k) {
                uint4 w = ALIGNED ? W[k] : U::realign(W[k], W[k + 1], shift);
                const int el = (ub + k) * N;
                if (el >= p.V) w = U::none4();
                else if (el + N > p.V) U::mask(w, 0, p.V - el);
                if (WARPED) U::cut(w, cut);
                float2 z[NP];
                U::unpack(w, z);
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    e[k][2 * j] = ex2((z[j].x - Mr) * c1);
                    e[k][2 * j + 1] = ex2((z[j].y - Mr) * c1);
                    ls += e[k][2 * j] + e[k][2 * j + 1];
                }
            }
            float li = ls;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float t = __shfl_up_sync(0xFFFFFFFFu, li, o);
                if (lane >= o) li += t;
            }
            float cc = cc0 + (li - ls);
            int hit = -1;
#pragma unroll
            for (int k = 0; k < IT; ++k) {
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    cc += e[k][j];
                    if (e[k][j] > 0.f) {
                        last = (ub + k) * N + j;
                        if (hit < 0 && cc > target) hit = last;
                    }
                }
            }
            const unsigned mh = __ballot_sync(0xFFFFFFFFu, hit >= 0);
            if (mh) tok = __shfl_sync(0xFFFFFFFFu, hit, __ffs(mh) - 1);
            cc0 += __shfl_sync(0xFFFFFFFFu, li, 31);
        }
        if (tok < 0) tok = __reduce_max_sync(0xFFFFFFFFu, last);
    }
    if (lane == 0) {
        if (rowbad) atomicOr(p.st.status, ADASD_STATUS_NAN);
        p.H_out[b] = H;
        if (p.lse_out) p.lse_out[b] = lse;
        if (sampling || greedy) p.token_out[b] = tok;
        const bool stop = H > tg_row;   // strict; NaN never stops
        if (p.stop_out) p.stop_out[b] = stop ? 1 : 0;
        if (p.draft_len) p.draft_len[b] = len_row + 1;
        if (p.active && stop) p.active[b] = 0;
    }
}

}  // namespace adasd
