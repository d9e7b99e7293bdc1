// The tail of a verification round as a kernel of its own, behind the one that works out every position's
// scalars: KDE densities and the Bayes posterior P(A|d_i) for every candidate (Sec. 4.4), the
// first-rejection accept scan, the list appends and the T_G update (Algorithm 1, steps 2 and 3).
//
// One cluster of S CTAs per sequence.  The KDE sums over the two lists are the only part that grows
// (Sec. 4.4): entries are dealt to all threads of the cluster, every thread sums them for eight
// candidates at a time, and the sums meet in rank 0; everything else is one warp with lane i on
// candidate i.  S follows the lists' capacity and the number of sequences, so that long lists spread
// over the chip (tail_cluster in adasd_api.cu).  Latency bounds it, a chain of about five dependent
// memory accesses and a few float64 functions: the state, the caller's tokens and uniforms are therefore
// read before the wait for the kernel ahead (they are older than that kernel, which lets this one start
// only after its own wait).
#pragma once

#include "adasd_async.cuh"

namespace adasd {

constexpr int kTailThreads = 256;
constexpr int kTailWarps = kTailThreads / 32;
constexpr int kTailMaxS = 8;

struct TailParams {
    TailConfig cfg;
    State st;
    const float* H_d;          // [B,Kmax] this round's positions
    const float* dist;         // [B,Kmax]
    const int32_t* y;          // [B,Kmax+1]
    const int32_t* x;          // [B,Kmax]
    const float* u_accept;     // [B,Kmax]
    const int32_t* draft_len;  // [B] or null
    float* p_acc;              // nullable from here on: the caller's record
    int32_t* accept_len_rec;
    int32_t* rejected_rec;
    int32_t* draft_len_rec;
    int32_t* accept_len;       // [B]
    int32_t* next_token;       // [B]
};

struct VerifyTailShared {
    float d[ADASD_KMAX_LIMIT];
    float cA[ADASD_KMAX_LIMIT];                      // -log2(e) / (2 h_A,i^2)
    float red[kTailWarps][16];
    float part[kTailMaxS][ADASD_KMAX_LIMIT / 8][16]; // rank 0: every CTA's sums, 8 candidates x (A, R) a group
    int32_t any;
};

// Sums of 16 values over the warp; lane l gets the total of value l / 2.
__device__ __forceinline__ float tail_reduce16(float (&v)[16]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int m = 8, o = 16; m > 0; m >>= 1, o >>= 1) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (k < m) {
                const bool up = lane & o;
                const float give = up ? v[k] : v[k + m], keep = up ? v[k + m] : v[k];
                v[k] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, o);
            }
        }
    }
    return v[0] + __shfl_xor_sync(0xFFFFFFFFu, v[0], 1);
}

__global__ void __launch_bounds__(kTailThreads) verify_tail_kernel(TailParams p) {
    __shared__ VerifyTailShared sh;
    cg::cluster_group cluster = cg::this_cluster();
    const int S = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int b = blockIdx.x / S;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int Kmax = p.cfg.Kmax;
    pdl_trigger();

    int K_t = p.draft_len ? __ldcg(p.draft_len + b) : Kmax;
    K_t = max(0, min(K_t, Kmax));
    const int nA0 = p.st.nA[b], nR0 = p.st.nR[b];
    double sA = 0.0, sA2 = 0.0, sE = 0.0, sR = 0.0, sR2 = 0.0;
    int nE0 = 0, x = 0;
    float u = 0.f;
    if (warp == 0) {
        sA = p.st.sumA[b];
        sA2 = p.st.sumA2[b];
        sR = p.st.sumR[b];
        sR2 = p.st.sumR2[b];
        sE = p.st.sumE[b];
        nE0 = p.st.nE[b];
        if (lane < K_t) {
            x = p.x[(size_t)b * Kmax + lane];
            u = p.u_accept[(size_t)b * Kmax + lane];
        }
    }
    // rejected side: one bandwidth for the round
    const bool longR = nR0 >= p.cfg.min_samples, longA = nA0 + K_t >= p.cfg.min_samples;
    double hR = 0.0;
    if (longR && longA) hR = kde_bandwidth((double)nR0, p.st.sumR[b], p.st.sumR2[b], p.cfg.bw_rule);
    const bool validR = hR > 0.0;
    const float cR = validR ? (float)(-0.5 * 1.4426950408889634 / (hR * hR)) : 0.f;
    if (S > 1) cluster.sync();                       // every CTA of the cluster runs: rank 0 may be written to
    pdl_wait();

    float d = 0.f, H = 0.f, cA = 0.f, ihA = 0.f;
    int y = 0;
    double n = (double)nA0, s = sA, s2 = sA2;
    bool ok = false;
    if (warp == 0) {
        if (lane < K_t) {
            d = __ldcg(p.dist + (size_t)b * Kmax + lane);
            H = __ldcg(p.H_d + (size_t)b * Kmax + lane);
            y = __ldcg(p.y + (size_t)b * (Kmax + 1) + lane);
        }
        // candidate i sees L_D^A plus the distances d_1..d_{i-1} of this round that lie strictly inside
        // (0,1): the list "as it stands" when candidate i is reached at all
        for (int j = 0; j < K_t; ++j) {
            const float dj = __shfl_sync(0xFFFFFFFFu, d, j);
            if (j < lane && dj > 0.f && dj < 1.f) {
                n += 1.0;
                s += (double)dj;
                s2 += (double)dj * (double)dj;
            }
        }
        if (validR) {
            const double hA = kde_bandwidth(n, s, s2, p.cfg.bw_rule);
            ok = lane < K_t && (n >= (double)p.cfg.min_samples) && (hA > 0.0);
            cA = ok ? (float)(-0.5 * 1.4426950408889634 / (hA * hA)) : 0.f;
            ihA = ok ? (float)(1.0 / hA) : 0.f;
        }
        const int any = __any_sync(0xFFFFFFFFu, ok);
        sh.d[lane] = d;
        sh.cA[lane] = cA;
        if (lane == 0) sh.any = any;
    }
    __syncthreads();
    const bool any = sh.any != 0;                    // the same in every CTA of the cluster
    if (any) {
        const float* LA = p.st.LA + (size_t)b * p.st.cap;
        const float* LR = p.st.LR + (size_t)b * p.st.cap;
        const int step = S * kTailThreads, j0 = rank * kTailThreads + tid;
        for (int i0 = 0; i0 < K_t; i0 += 8) {
            float acc[16], di[8], ci[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int i = min(i0 + k, K_t - 1);
                acc[k] = acc[8 + k] = 0.f;
                di[k] = sh.d[i];
                ci[k] = sh.cA[i];
            }
            // four entries a trip, their loads in flight together
            auto sums = [&](const float* list, int len, bool rejected) {
                for (int j = j0; j < len; j += 4 * step) {
                    float xj[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) xj[q] = j + q * step < len ? __ldcg(list + j + q * step) : 0.f;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        if (j + q * step < len) {
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                const float t = di[k] - xj[q];
                                if (rejected) acc[8 + k] += ex2(cR * t * t);
                                else acc[k] += ex2(ci[k] * t * t);
                            }
                        }
                    }
                }
            };
            sums(LA, nA0, false);
            sums(LR, nR0, true);
            const float v = tail_reduce16(acc);
            if (i0) __syncthreads();                 // sh.red free again
            if (!(lane & 1)) sh.red[warp][lane >> 1] = v;
            __syncthreads();
            if (tid < 16) {
                float a = 0.f;
#pragma unroll
                for (int w = 0; w < kTailWarps; ++w) a += sh.red[w][tid];
                (S > 1 ? cluster.map_shared_rank(&sh, 0) : &sh)->part[rank][i0 >> 3][tid] = a;
            }
        }
    }
    if (S > 1) cluster.sync();
    else __syncthreads();
    if (rank != 0 || warp != 0) return;

    float SA = 0.f, SR = 0.f;
    if (any && lane < K_t) {
        for (int r = 0; r < S; ++r) {
            SA += sh.part[r][lane >> 3][lane & 7];
            SR += sh.part[r][lane >> 3][8 + (lane & 7)];
        }
    }
    // kernel terms of this round's earlier distances, then the posterior
    float P = 0.f;
    if (any) {
        for (int j = 0; j < K_t; ++j) {
            const float dj = __shfl_sync(0xFFFFFFFFu, d, j);
            if (j < lane && dj > 0.f && dj < 1.f) {
                const float t = d - dj;
                SA += ex2(cA * t * t);
            }
        }
        if (ok) {
            // n_A f_A = SA / (h_A sqrt(2 pi)),  n_R f_R = SR / (h_R sqrt(2 pi))
            const float a = SA * ihA, r = SR * (float)(1.0 / hR), den = a + r;
            if (den > 0.f && den < INFINITY) P = a / den;
        }
    }
    if (p.p_acc && lane < K_t) p.p_acc[(size_t)b * Kmax + lane] = P;
    const bool rej = p.cfg.reject_rule == 0 ? (u >= P) : (P < 0.5f);
    const unsigned m = __ballot_sync(0xFFFFFFFFu, lane < K_t && x != y && rej);
    const int w = m ? (__ffs(m) - 1) : K_t;
    const bool rejected = (m != 0u);
    if (lane == 0) {
        p.accept_len[b] = w;
        p.next_token[b] = __ldcg(p.y + (size_t)b * (Kmax + 1) + w);
        if (p.accept_len_rec) p.accept_len_rec[b] = w;
        if (p.rejected_rec) p.rejected_rec[b] = rejected ? 1 : 0;
        if (p.draft_len_rec) p.draft_len_rec[b] = K_t;
    }
    if (!p.cfg.update) return;

    // appends (as apply_update): accepted distances strictly inside (0,1), in order, while there is room
    const int cap = p.st.cap;
    const bool in = lane < w && d > 0.f && d < 1.f;
    const unsigned mi = __ballot_sync(0xFFFFFFFFu, in);
    const int at = nA0 + __popc(mi & ((1u << lane) - 1u));
    if (in && at < cap) p.st.LA[(size_t)b * cap + at] = d;
    const int cnt = __popc(mi), room = min(cnt, max(cap - nA0, 0));
    if (room < cnt && lane == 0) atomicOr(p.st.status, ADASD_STATUS_CAPACITY);
    if (room > 0) {
        double a = sA, a2 = sA2;
        int left = room;
        for (int j = 0; j < w; ++j) {
            const float dj = __shfl_sync(0xFFFFFFFFu, d, j);
            if (dj > 0.f && dj < 1.f && left > 0) {
                --left;
                a += (double)dj;
                a2 += (double)dj * (double)dj;
            }
        }
        if (lane == 0) {
            p.st.nA[b] = nA0 + room;
            p.st.sumA[b] = a;
            p.st.sumA2[b] = a2;
        }
    }
    if (rejected) {
        // The entropy of a row with NaN or no finite logit is NaN (the status word says so already):
        // it is not recorded.  A full list skips the append whole, so that T_G stays the mean of the
        // entries the list holds (what a checkpoint restores).
        const float Hw = __shfl_sync(0xFFFFFFFFu, H, w), dw = __shfl_sync(0xFFFFFFFFu, d, w);
        if (lane == 0) {
            bool full = false;
            if (Hw == Hw && fabsf(Hw) < INFINITY) {
                if (nE0 < cap) {
                    p.st.LE[(size_t)b * cap + nE0] = Hw;
                    const double t = sE + (double)Hw;
                    p.st.nE[b] = nE0 + 1;
                    p.st.sumE[b] = t;
                    p.st.T_G[b] = (float)(t / (double)(nE0 + 1));      // T_G <- average(L_E^R)
                } else {
                    full = true;
                }
            }
            if (dw > 0.f && dw < 1.f) {
                if (nR0 < cap) {
                    p.st.LR[(size_t)b * cap + nR0] = dw;
                    p.st.nR[b] = nR0 + 1;
                    p.st.sumR[b] = sR + (double)dw;
                    p.st.sumR2[b] = sR2 + (double)dw * (double)dw;
                } else {
                    full = true;
                }
            }
            if (full) atomicOr(p.st.status, ADASD_STATUS_CAPACITY);
        }
    }
}

}  // namespace adasd
