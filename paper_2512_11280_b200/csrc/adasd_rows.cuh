// Parameters of the row kernels, the kernel of the allocation-free vanilla verification (which has no context,
// hence no tables: one thread-block cluster per candidate position, any V, any stride, bf16 or fp32, rows read
// from global memory once per pass, the later passes from L2), and the small kernels of the state.
#pragma once

#include "adasd_device.cuh"
#include "adasd_tail.cuh"
#include "adasd_warp.cuh"

namespace adasd {

struct Scratch {            // per-round scratch: the context's, or the fixed array of the allocation-free call
    float* H_d;             // [B,Kmax] entropies and distances of a round's candidates, for its tail
    float* dist;
    int32_t* y;             // [B,Kmax+1] target samples
    int32_t* van_flag;      // allocation-free vanilla call: [B,Kmax] 1 accept / 0 reject
    int32_t* van_tok;       // ... [B,Kmax+1] resample (or bonus) candidate
    uint32_t* ticket;       // ... [B] arrival counter of a sequence's positions
};

struct VerifyParams {
    const void* zd;
    const void* zt;
    long long d_seq, d_row, t_seq, t_row;
    const int32_t* x;
    const int32_t* draft_len;
    const float* u_target;
    const float* u_accept;
    const float* u_resample;
    int32_t* accept_len;
    int32_t* next_token;
    float* alpha_out;
    adasd_round_record user;   // caller's record (entries may be null)
    Scratch sc;
    State st;
    int32_t B, V, Kmax;
    // adjusted distribution (Sec. 2.1.1): 1 / temperature and, per row, the logit below which
    // tokens are cut (null: no cut); the staged kernels fold the temperature into c1 = log2 e / T
    float inv_temp, c1;
    const float* cut_t;     // [B,Kmax+1]
    const float* cut_d;     // [B,Kmax]
};

struct DraftParams {
    const void* z;
    long long row_stride;
    const float* u;
    uint8_t* active;
    float* H_out;
    float* lse_out;
    int32_t* token_out;
    uint8_t* stop_out;
    int32_t* draft_len;
    State st;
    int32_t B, V;
    int32_t expire_row;     // self-test of the bounded waits: the row whose first copy is never asked for (-1: none)
    int32_t argmax;         // 1: the token is argmax q (greedy drafting)
    int32_t early;          // 1: the next call's CTAs may be set up while this one runs
    float c1;               // adjusted distribution: log2 e / temperature
    const float* cut;       // [B] logit below which a row's tokens are cut (null: no cut)
};

struct RowShared {
    float warp[kWarps * 4];
    float xA[kMaxCluster * 4];
    float xB[kMaxCluster * 2];
    float xC[kMaxCluster * 4];
    float wtab[kMaxGW];      // per-warp weight totals of the row being sampled
    float wtab2[kMaxGW];     // vanilla: per-warp residual totals
};

// ------------------------------------------------------------------------------------
// Vanilla verification of position (b,i): softmax statistics of q_i and p_i, alpha_i, the residual sample.
// ------------------------------------------------------------------------------------
template <typename T, bool VEC>
__global__ void __launch_bounds__(kThreads) static_vanilla_kernel(VerifyParams p) {
    constexpr int N = Elt<T>::N;
    cg::cluster_group cluster = cg::this_cluster();
    const int CS = (int)cluster.num_blocks();
    const int rank = (int)cluster.block_rank();
    const int pos = blockIdx.x / CS;
    const int Kmax = p.Kmax;
    const int b = pos / (Kmax + 1), i = pos % (Kmax + 1);
    int K_t = p.draft_len ? p.draft_len[b] : Kmax;
    K_t = max(0, min(K_t, Kmax));
    if (i > K_t) return;                       // same decision in every CTA of the cluster
    const bool bonus = (i == K_t);

    __shared__ RowShared sh;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int GW = CS * kWarps, gw = rank * kWarps + warp;
    const int NU = (p.V + N - 1) / N;
    const int u0 = (int)((long long)gw * NU / GW), u1 = (int)((long long)(gw + 1) * NU / GW);
    const T* rt = reinterpret_cast<const T*>(p.zt) + (long long)b * p.t_seq + (long long)i * p.t_row;
    const T* rd = bonus ? rt
                        : reinterpret_cast<const T*>(p.zd) + (long long)b * p.d_seq + (long long)i * p.d_row;

    // pass A: maxima, NaN flag
    float vA[4] = {-INFINITY, -INFINITY, 0.f, 0.f};
    for (int u = u0 + lane; u < u1; u += 32) {
        float xt[N], xd[N];
        load_unit<T, VEC>(rt, u, p.V, xt);
        if (!bonus) load_unit<T, VEC>(rd, u, p.V, xd);
#pragma unroll
        for (int j = 0; j < N; ++j) {
            if (bonus) xd[j] = xt[j];
            vA[2] = (xt[j] != xt[j] || xd[j] != xd[j]) ? 1.f : vA[2];
            vA[0] = fmaxf(vA[0], xt[j]);
            vA[1] = fmaxf(vA[1], xd[j]);
        }
    }
    cluster_allreduce<4, true>(vA, sh.warp, sh.xA, CS, rank, cluster);
    const bool bad = (vA[2] > 0.f) || !(vA[0] > kFloor) || !(vA[1] > kFloor) ||
                     (vA[0] == INFINITY) || (vA[1] == INFINITY);
    const float mt = vA[0], md = vA[1];

    // pass B: S_t, S_d; per-warp S_t for sampling y_i
    float vB[2] = {0.f, 0.f};
    for (int u = u0 + lane; u < u1; u += 32) {
        float xt[N], xd[N];
        load_unit<T, VEC>(rt, u, p.V, xt);
        if (!bonus) load_unit<T, VEC>(rd, u, p.V, xd);
#pragma unroll
        for (int j = 0; j < N; ++j) {
            vB[0] += ex2((fmaxf(xt[j], kFloor) - mt) * kLog2e);
            if (!bonus) vB[1] += ex2((fmaxf(xd[j], kFloor) - md) * kLog2e);
        }
    }
    {
        float ws = warp_sum(vB[0]);
        if (lane == 0)
            for (int r = 0; r < CS; ++r) cluster.map_shared_rank(sh.wtab, r)[gw] = ws;
    }
    cluster_allreduce<2, false>(vB, sh.warp, sh.xB, CS, rank, cluster);
    if (bonus) vB[1] = vB[0];
    // log2 p = (z - m) log2e - log2 S: exactly 0 for the only token of a one-hot row
    const float lSt = lg2(vB[0]), lSd = lg2(vB[1]);

    // vanilla: alpha_i at the draft token, known to every thread
    bool van_accept = true;
    float alpha = 1.f;
    if (!bonus && !bad) {
        const int xi = p.x[(size_t)b * Kmax + i];
        if (xi >= 0 && xi < p.V) {
            float a = fmaf(fmaxf(to_f32(rt[xi]), kFloor) - mt, kLog2e, -lSt);
            float q = fmaf(fmaxf(to_f32(rd[xi]), kFloor) - md, kLog2e, -lSd);
            alpha = fminf(1.f, ex2(a - q));
            if (!(ex2(q) > 0.f)) alpha = 1.f;   // q(x) = 0 cannot have been drafted
        } else {
            alpha = 0.f;
        }
        van_accept = p.u_accept[(size_t)b * Kmax + i] < alpha;
    }

    // pass C, on a rejected row: residual mass max(0, p - q), per warp and in total
    float vC[2] = {0.f, 0.f};
    const bool need_resid = !bonus && !van_accept;
    if (need_resid) {
        for (int u = u0 + lane; u < u1; u += 32) {
            float xt[N], xd[N];
            load_unit<T, VEC>(rt, u, p.V, xt);
            load_unit<T, VEC>(rd, u, p.V, xd);
#pragma unroll
            for (int j = 0; j < N; ++j) {
                const float pp = ex2(fmaf(fmaxf(xt[j], kFloor) - mt, kLog2e, -lSt));
                const float qq = ex2(fmaf(fmaxf(xd[j], kFloor) - md, kLog2e, -lSd));
                vC[0] += fmaxf(pp - qq, 0.f);
            }
        }
        const float ws = warp_sum(vC[0]);
        if (lane == 0)
            for (int r = 0; r < CS; ++r) cluster.map_shared_rank(sh.wtab2, r)[gw] = ws;
    }
    cluster_allreduce<2, false>(vC, sh.warp, sh.xC, CS, rank, cluster);

    // sampling: bonus row, or rejected row (the target row itself where the residual has no mass)
    const size_t it = (size_t)b * (Kmax + 1) + i;
    const size_t id = (size_t)b * Kmax + i;
    if (!bad) {
        const bool from_resid = need_resid && (vC[0] > 0.f);
        if (bonus || need_resid) {
            const float uu = p.u_resample[b];
            float base = 0.f, target = 0.f;
            int chosen = select_warp(from_resid ? sh.wtab2 : sh.wtab, GW, uu, base, target);
            if (chosen == gw) {
                int tok;
                if (from_resid) {
                    tok = warp_scan_select<N>(u0, u1, p.V, base, target, [&](int u, float(&w)[N]) {
                        float xt[N], xd[N];
                        load_unit<T, VEC>(rt, u, p.V, xt);
                        load_unit<T, VEC>(rd, u, p.V, xd);
#pragma unroll
                        for (int j = 0; j < N; ++j) {
                            float pp = ex2(fmaf(fmaxf(xt[j], kFloor) - mt, kLog2e, -lSt));
                            float qq = ex2(fmaf(fmaxf(xd[j], kFloor) - md, kLog2e, -lSd));
                            w[j] = fmaxf(pp - qq, 0.f);
                        }
                    });
                } else {
                    tok = warp_scan_select<N>(u0, u1, p.V, base, target, [&](int u, float(&w)[N]) {
                        float xt[N];
                        load_unit<T, VEC>(rt, u, p.V, xt);
#pragma unroll
                        for (int j = 0; j < N; ++j)
                            w[j] = ex2((fmaxf(xt[j], kFloor) - mt) * kLog2e);
                    });
                }
                if (lane == 0) p.sc.van_tok[it] = tok;
            }
        }
    }

    // publish this position's scalars
    if (rank == 0 && threadIdx.x == 0) {
        if (bad) atomicOr(p.st.status, ADASD_STATUS_NAN);
        if (!bonus) {
            p.sc.van_flag[id] = (van_accept && !bad) ? 1 : 0;
            if (p.alpha_out) p.alpha_out[id] = bad ? NAN : alpha;
        }
        if (bad) p.sc.van_tok[it] = -1;
    }

    // all writes of this cluster are done once every CTA has passed this barrier
    cluster.sync();
    if (rank != 0 || threadIdx.x != 0) return;
    // the cluster that publishes the last position of a sequence finds its longest accepted prefix
    __threadfence();
    if (atomicAdd(p.sc.ticket + b, 1u) != (unsigned)K_t) return;
    p.sc.ticket[b] = 0u;    // ready for the next round
    __threadfence();
    int w = K_t;
    for (int j = 0; j < K_t; ++j) {
        if (__ldcg(p.sc.van_flag + (size_t)b * Kmax + j) == 0) {
            w = j;
            break;
        }
    }
    p.accept_len[b] = w;
    p.next_token[b] = __ldcg(p.sc.van_tok + (size_t)b * (Kmax + 1) + w);
}

// ------------------------------------------------------------------------------------
// Stand-alone update from a record (for callers that do not fuse it into verify)
// ------------------------------------------------------------------------------------
__global__ void update_kernel(State st, adasd_round_record rec, int B, int Kmax) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    int K_t = max(0, min(rec.draft_len[b], Kmax));
    int w = max(0, min(rec.accept_len[b], K_t));
    bool rejected = rec.rejected[b] != 0 && w < K_t;
    apply_update(st, b, w, rejected, rec.dist + (size_t)b * Kmax, rec.H_d + (size_t)b * Kmax);
}

__global__ void reset_kernel(State st, const int32_t* ids, int n, int B) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    int b = ids ? ids[k] : k;
    if (b < 0 || b >= B) return;
    st.T_G[b] = 0.f;
    st.sumE[b] = 0.0;
    st.nE[b] = st.nA[b] = st.nR[b] = 0;
    st.sumA[b] = st.sumA2[b] = st.sumR[b] = st.sumR2[b] = 0.0;
}

__global__ void get_thresholds_kernel(State st, float* T_G, int32_t* nE, int32_t* nA, int32_t* nR,
                                      int B) {
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    if (T_G) T_G[b] = st.T_G[b];
    if (nE) nE[b] = st.nE[b];
    if (nA) nA[b] = st.nA[b];
    if (nR) nR[b] = st.nR[b];
}

}  // namespace adasd
