// Top-k cutoffs of the adjusted distribution (Sec. 2.1.1) by selection, bf16 or fp32 rows of any length,
// alignment and stride.
//
// With a top-k cut only the k largest logits matter, also for the top-p cut behind it.  One cluster of P
// CTAs per row:
//  1. every thread takes the maxima of two groups of the row's elements; a tau with k or a few more of all
//     group maxima at or above it has at least k elements at or above it;
//  2. the elements above tau (not many more than k: each is one of its group's largest) are collected,
//     those equal to tau counted;
//  3. rank 0 finds the k-th largest of the row among them by counting, and the top-p cut among what is left
//     from masses in 2^-40 fixed point (sums that do not depend on the order of the list).
// A row that leaves more than kSelList candidates (its large logits sit in few groups) is left NaN for
// row_cutoff_kernel (only_flagged).
// What bounds it: latency (two reads of the row, the second from L1, and about twenty block and cluster
// barriers, most of them the bisection's): the cluster size makes a launch fill the chip.  k = 50, p = 0.95, 16
// rows of 128256 logits: it adds 15 us to a draft call of bf16 rows (16.8 us by itself), where the
// histogram of all values (row_cutoff_hist_kernel) adds 34; to one of fp32 rows 19, where the radix descent adds 440.
#pragma once

#include "adasd_async.cuh"
#include "adasd_warp.cuh"

namespace adasd {

constexpr int kSelThreads = 512;
constexpr int kSelMaxP = 8;
constexpr int kSelList = 1024;
constexpr int kSelMinV = 4096;                       // shorter rows: the radix descent
constexpr int kSelMaxK = 512;                        // (the rule that chooses this kernel asks for less on some rows)

// Whether a unit has an element at or above tau.
template <typename T>
struct Reach;
template <>
struct Reach<__nv_bfloat16> {
    uint32_t t2;
    __device__ __forceinline__ explicit Reach(float tau) : t2(cut_pair(tau)) {}
    __device__ __forceinline__ uint32_t ge(uint32_t w) const {
        uint32_t m;
        asm("set.ge.u32.bf16x2 %0, %1, %2;" : "=r"(m) : "r"(w), "r"(t2));
        return m;
    }
    __device__ __forceinline__ bool operator()(const uint4& w) const { return (ge(w.x) | ge(w.y) | ge(w.z) | ge(w.w)) != 0u; }
};
template <>
struct Reach<float> {
    float t;
    __device__ __forceinline__ explicit Reach(float tau) : t(tau) {}
    __device__ __forceinline__ bool operator()(const uint4& w) const {
        return fmaxf(fmaxf(__uint_as_float(w.x), __uint_as_float(w.y)), fmaxf(__uint_as_float(w.z), __uint_as_float(w.w))) >= t;
    }
};

struct SelShared {
    union {                                          // rank 0
        uint32_t gmax[kSelMaxP * kSelThreads * 2];   // keys of all group maxima; done with before the others
        struct {
            unsigned long long w[kSelList];          // everybody's candidates and their masses
            float all[kSelList];
        };
    };
    float list[kSelList];                            // this CTA's candidates
    uint32_t cnt[32];                                // counts of the bisection steps
    uint32_t big, small;
    int32_t n, n_eq;                                 // candidates, elements equal to tau (of this CTA)
    int32_t at, total, eq;                           // where this CTA's go; rank 0: of all CTAs
    uint32_t bad;
    uint32_t tau;                                    // key
    uint32_t key_k, key_p;
    unsigned long long S;
    float m;
};

template <typename T, bool ALIGNED>
__global__ void __launch_bounds__(kSelThreads, 3) row_cutoff_select_kernel(CutParams p, CutParams p2) {
    using U = Unit<T>;
    constexpr int N = U::N;
    using K32 = CutKey<float>;                       // (bf16 values too: the keys' order is what counts)
    __shared__ SelShared sh;
    cg::cluster_group cluster = cg::this_cluster();
    const int P = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31;
    // (a verification round: the target rows, then the draft rows)
    int row = blockIdx.x / P;
    if (row >= p.B * p.R) {
        row -= p.B * p.R;
        p = p2;
    }
    const int b = row / p.R, j = row - b * p.R;
    pdl_wait();
    pdl_trigger();
    // (all of these the same in every CTA of the cluster)
    if (p.active && p.active[b] == 0) return;
    if (p.draft_len) {
        const int kt = max(0, min(p.draft_len[b], p.R - p.extra));
        if (j >= kt + p.extra) return;
    }
    float* const out = p.cut + (size_t)b * p.R + j;
    const unsigned long long ra = reinterpret_cast<unsigned long long>(
        reinterpret_cast<const T*>(p.z) + (long long)b * p.seq_stride + (long long)j * p.row_stride);
    const uint4* const base = reinterpret_cast<const uint4*>(ALIGNED ? ra : ra & ~15ull);
    const int shift = ALIGNED ? 0 : (int)((ra & 15ull) / sizeof(T));
    const int g1 = (shift + p.V + N - 1) / N;        // granules that hold elements: [0, g1)
    const int NU = (p.V + N - 1) / N, step = P * kSelThreads, u0 = rank * kSelThreads + tid;
    auto unit = [&](int u) -> uint4 {                // elements u N ..; those past the end read as -inf
        uint4 w = base[u];
        if (!ALIGNED) w = U::realign(w, u + 1 < g1 ? base[u + 1] : U::none4(), shift);
        if (u == NU - 1 && u * N + N > p.V) U::mask(w, 0, p.V - u * N);
        return w;
    };
    if (tid < 32) sh.cnt[tid] = 0u;
    if (tid == 0) {
        sh.big = 0u;
        sh.small = 0xFFFFFFFFu;
        sh.n = 0;
        sh.n_eq = 0;
        sh.total = 0;
        sh.eq = 0;
        sh.bad = 0u;
        sh.key_k = 0u;
        sh.key_p = 0xFFFFFFFFu;
        sh.S = 0ull;
    }

    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    // 1. group maxima: two of every thread
    float m0, m1;
    uint32_t nan = 0u;
    {
        typename U::Max x = U::max0(), y = U::max0();
        int u = u0;
        for (; u + 3 * step < NU; u += 4 * step) {   // four units asked for before the first is used
            uint4 w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) w[q] = unit(u + q * step);
#pragma unroll
            for (int q = 0; q < 4; ++q) U::max_add(q & 1 ? y : x, w[q]);
        }
        for (; u < NU; u += step) U::max_add(x, unit(u));
        if (N == 8) {                                // the halves of the packed pairs
            const uint32_t h = bmax2(*reinterpret_cast<const uint32_t*>(&x), *reinterpret_cast<const uint32_t*>(&y));
            const float2 v = unpack2(h);
            nan = (v.x != v.x || v.y != v.y) ? 1u : 0u;
            m0 = v.x;
            m1 = v.y;
        } else {
            m0 = U::max_val(x, nan);
            m1 = U::max_val(y, nan);
        }
        if (!(m0 == m0)) m0 = -INFINITY;
        if (!(m1 == m1)) m1 = -INFINITY;
    }
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");     // every CTA runs: rank 0 may be written to
    SelShared* const r0 = cluster.map_shared_rank(&sh, 0);
    {
        uint32_t* g = r0->gmax + rank * (2 * kSelThreads);
        g[tid] = K32::of(m0);
        g[kSelThreads + tid] = K32::of(m1);
        if (nan) atomicOr(&r0->bad, 1u);
    }
    cluster.sync();
    if (rank == 0) {
        // tau: a key with at least k of the 2 P kSelThreads keys at or above it, and not many more, by bisection
        // between the smallest and the largest (a histogram of digits would pile up in a few bins)
        // (the key of a bf16 value ends in 16 equal bits: left out)
        constexpr int kLow = N == 8 ? 16 : 0;
        auto value = [](uint32_t k) -> uint32_t { return N == 8 ? (k << 16) | ((k & 0x8000u) ? 0u : 0xFFFFu) : k; };
        uint32_t key[2 * kSelMaxP];
        uint32_t big = 0u, small = 0xFFFFFFFFu;
#pragma unroll
        for (int q = 0; q < 2 * kSelMaxP; ++q) {
            key[q] = q < 2 * P ? sh.gmax[q * kSelThreads + tid] >> kLow : 0u;
            if (q < 2 * P) {
                big = max(big, key[q]);
                small = min(small, key[q]);
            }
        }
        big = __reduce_max_sync(0xFFFFFFFFu, big);
        small = __reduce_min_sync(0xFFFFFFFFu, small);
        if (lane == 0) {
            atomicMax(&sh.big, big);
            atomicMin(&sh.small, small);
        }
        __syncthreads();
        uint32_t lo = sh.small, hi = sh.big;         // at least k keys at or above lo
        const uint32_t need = (uint32_t)p.top_k, enough = need + max(16u, need / 4u);
        for (int it = 0; lo < hi; ++it) {            // (halves hi - lo: at most 32 times)
            const uint32_t mid = lo + (hi - lo + 1u) / 2u;
            uint32_t c = 0u;
#pragma unroll
            for (int q = 0; q < 2 * kSelMaxP; ++q) c += key[q] >= mid ? 1u : 0u;
            c = __reduce_add_sync(0xFFFFFFFFu, c);
            if (lane == 0 && c) atomicAdd(&sh.cnt[it & 31], c);
            __syncthreads();
            c = sh.cnt[it & 31];
            if (c < need) {
                hi = mid - 1u;
            } else {
                lo = mid;
                if (c <= enough) break;
            }
        }
        if (tid == 0) {
            sh.tau = value(lo);
            sh.m = K32::value(value(sh.big));
        }
    }
    cluster.sync();
    const float tau = K32::value(r0->tau), m = r0->m;
    const bool bad = (r0->bad != 0u) || !(m > -INFINITY) || m == INFINITY;   // an unusable row is not cut; the row pass reports it

    // 2. the elements above tau
    if (!bad) {
        const Reach<T> reach(tau);
        auto collect = [&](int u, const uint4& w) {
            float x[N];
            unpack16(w, x);
#pragma unroll
            for (int q = 0; q < N; ++q) {
                if (u * N + q < p.V && x[q] > tau) {
                    const int at = atomicAdd(&sh.n, 1);
                    if (at < kSelList) sh.list[at] = x[q];
                } else if (u * N + q < p.V && x[q] == tau) {
                    atomicAdd(&sh.n_eq, 1);
                }
            }
        };
        int u = u0;
        for (; u + 3 * step < NU; u += 4 * step) {
            uint4 w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) w[q] = unit(u + q * step);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (reach(w[q])) collect(u + q * step, w[q]);
        }
        for (; u < NU; u += step) {
            const uint4 w = unit(u);
            if (reach(w)) collect(u, w);
        }
    }
    __syncthreads();
    // everybody's candidates into rank 0's list
    const int mine = sh.n;
    if (tid == 0) {
        sh.at = atomicAdd(&r0->total, mine);
        atomicAdd(&r0->eq, sh.n_eq);
    }
    __syncthreads();
    if (mine <= kSelList && sh.at + mine <= kSelList)
        for (int i = tid; i < mine; i += kSelThreads) r0->all[sh.at + i] = sh.list[i];
    cluster.sync();                                  // (nobody writes to rank 0 any more)
    if (rank != 0) return;
    const int n = sh.total, n_eq = sh.eq;
    if (bad || n > kSelList) {
        if (tid == 0) *out = bad ? -INFINITY : __int_as_float(0x7FC00000);
        return;
    }

    // 3. the k-th largest: the value with fewer than k above it and k at or above it (tau itself when the list
    // is shorter than k)
    for (int i = tid; i < n; i += kSelThreads) {
        const float v = sh.all[i];
        int gt = 0, ge = 0;
        for (int q = 0; q < n; ++q) {
            gt += sh.all[q] > v;
            ge += sh.all[q] >= v;
        }
        if (gt < p.top_k && ge >= p.top_k) sh.key_k = K32::of(v);            // (one value, perhaps several threads)
        sh.w[i] = (unsigned long long)__double2ll_rn(exp2((double)(fmaxf(v, kFloor) - m) * p.c1) * kCutFix);
    }
    __syncthreads();
    const uint32_t key_tau = sh.tau, key_k = n < p.top_k ? key_tau : sh.key_k;
    if (!(p.top_p < 1.f)) {
        if (tid == 0) *out = K32::value(key_k);
        return;
    }
    // top-p of what is left: the smallest value with less than top_p of the mass strictly above it
    const bool with_tau = key_k == key_tau && n < p.top_k;
    const unsigned long long w_tau = (unsigned long long)__double2ll_rn(exp2((double)(fmaxf(tau, kFloor) - m) * p.c1) * kCutFix);
    unsigned long long part = 0ull;
    for (int i = tid; i < n; i += kSelThreads)
        if (K32::of(sh.all[i]) >= key_k) part += sh.w[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xFFFFFFFFu, part, o);
    if (lane == 0 && part) atomicAdd(&sh.S, part);
    __syncthreads();
    const unsigned long long list_mass = sh.S, S = list_mass + (with_tau ? (unsigned long long)n_eq * w_tau : 0ull);
    const double thr = (double)p.top_p * (double)S;
    for (int i = tid; i < n; i += kSelThreads) {
        const float v = sh.all[i];
        const uint32_t k = K32::of(v);
        if (k < key_k) continue;
        unsigned long long above = 0ull;
        for (int q = 0; q < n; ++q)
            if (sh.all[q] > v) above += sh.w[q];
        if ((double)above < thr) atomicMin(&sh.key_p, k);
    }
    if (tid == 0 && with_tau && (double)list_mass < thr) atomicMin(&sh.key_p, key_tau);
    __syncthreads();
    if (tid == 0) *out = K32::value(max(key_k, sh.key_p));
}

}  // namespace adasd
