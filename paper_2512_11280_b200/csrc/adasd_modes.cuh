// The Gen-Only ablation variant (Sec. 5): the feedback of the generation component alone, the entropy of
// the candidate that vanilla verification rejected joins L_E^R, T_G = mean(L_E^R).
#pragma once

#include "adasd_device.cuh"

namespace adasd {

// One thread per sequence: L_E^R += H(q) of the candidate vanilla verification rejected.
__global__ void gen_only_update_kernel(State st, const float* __restrict__ H_d, const int32_t* __restrict__ draft_len,
                                       const int32_t* __restrict__ accept_len, int B, int Kmax) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    int kt = draft_len ? draft_len[b] : Kmax;
    kt = max(0, min(kt, Kmax));
    const int w = accept_len[b];
    if (w < 0 || w >= kt) return;                     // nothing was rejected
    const float Hw = H_d[(size_t)b * Kmax + w];
    if (!(Hw == Hw) || !(fabsf(Hw) < INFINITY)) return;
    const int nE = st.nE[b];
    if (nE >= st.cap) {
        atomicOr(st.status, ADASD_STATUS_CAPACITY);
        return;
    }
    st.LE[(size_t)b * st.cap + nE] = Hw;
    const double sE = st.sumE[b] + (double)Hw;
    st.nE[b] = nE + 1;
    st.sumE[b] = sE;
    st.T_G[b] = (float)(sE / (double)(nE + 1));
}

}  // namespace adasd
