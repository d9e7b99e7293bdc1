// Pieces of the per-sequence tail of a round: the KDE bandwidth (Sec. 4.4) and the list appends with the
// T_G update (Algorithm 1, steps 2 and 3).
#pragma once

#include "adasd_device.cuh"

namespace adasd {

struct TailConfig {
    int32_t Kmax;
    int32_t min_samples;
    int32_t bw_rule;      // 0 Silverman, 1 Scott
    int32_t reject_rule;  // 0 Bernoulli, 1 threshold 1/2
    uint32_t update;      // append to the lists and refresh T_G
};

// Bandwidth from running sums: h = sample_std * factor(n).  Returns 0 when undefined.
__device__ __forceinline__ double kde_bandwidth(double n, double sum, double sum2, int rule) {
    if (n < 2.0) return 0.0;
    double var = (sum2 - sum * sum / n) / (n - 1.0);
    // identical samples leave rounding noise instead of an exact zero
    if (!(var > 1e-13 * (sum2 / n))) return 0.0;
    const double f = exp2(-0.2 * log2(rule == 0 ? 0.75 * n : n));
    return sqrt(var) * f;
}

// Appends and threshold update of one sequence (Algorithm 1: the append lines of the
// verify loop and step 3).  One thread.
__device__ __forceinline__ void apply_update(State& st, int b, int w, bool rejected,
                                             const float* d, const float* H) {
    const int cap = st.cap;
    int nA = st.nA[b];
    double sA = st.sumA[b], sA2 = st.sumA2[b];
    for (int j = 0; j < w; ++j) {
        float dj = d[j];
        if (dj > 0.f && dj < 1.f) {
            if (nA < cap) {
                st.LA[(size_t)b * cap + nA] = dj;
                ++nA;
                sA += (double)dj;
                sA2 += (double)dj * (double)dj;
            } else {
                atomicOr(st.status, ADASD_STATUS_CAPACITY);
            }
        }
    }
    st.nA[b] = nA;
    st.sumA[b] = sA;
    st.sumA2[b] = sA2;
    if (rejected) {
        // The entropy of a row with NaN or no finite logit is NaN (the status word says so
        // already): recording it would leave T_G = NaN and switch the draft-stop check off for
        // good.  A full list skips the append whole, like the other two lists, so that T_G stays
        // the mean of the entries the list holds (what a checkpoint restores).
        const float Hw = H[w];
        int nE = st.nE[b];
        if (Hw == Hw && fabsf(Hw) < INFINITY) {
            if (nE < cap) {
                st.LE[(size_t)b * cap + nE] = Hw;
                double sE = st.sumE[b] + (double)Hw;
                ++nE;
                st.nE[b] = nE;
                st.sumE[b] = sE;
                st.T_G[b] = (float)(sE / (double)nE);  // T_G <- average(L_E^R)
            } else {
                atomicOr(st.status, ADASD_STATUS_CAPACITY);
            }
        }
        float dw = d[w];
        if (dw > 0.f && dw < 1.f) {
            int nR = st.nR[b];
            if (nR < cap) {
                st.LR[(size_t)b * cap + nR] = dw;
                st.nR[b] = nR + 1;
                st.sumR[b] += (double)dw;
                st.sumR2[b] += (double)dw * (double)dw;
            } else {
                atomicOr(st.status, ADASD_STATUS_CAPACITY);
            }
        }
    }
}

}  // namespace adasd
