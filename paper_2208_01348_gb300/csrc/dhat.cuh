// Phases of the D-hat build (k_dhat.cu): one axis of the transform of a
// sequence that is even or odd along it, from its non-negative half.
//
// Along an axis the padded Green's tensor holds g(i) at 0 <= i < n, +-g(L - i)
// at the mirrored indices and zero between.  With h(0) = g(0)/2, h(i) = g(i)
// and H the length-L transform of the half-filled line h, the transform wanted
// on the octant is F(k) = H(k) +- H(L - k), k <= L/2.
#pragma once
#include "dft.cuh"

namespace eels {

// W lines in A[L][es]; place j of set a in row a RE + j.  LANE_J: adjacent
// threads take adjacent j of a line (lines contiguous in memory).
template <int RE, int RO, bool LANE_J, class In>
HD void dhat_1(double2* A, int es, int W, int n, int tid, int nthr, In in) {
    for (int t = tid; t < W * RO; t += nthr) {
        const int j = LANE_J ? t % RO : t / W, w = LANE_J ? t / RO : t % W;
        double2 v[RE];
#pragma unroll
        for (int r = 0; r < RE / 2; ++r) {
            const int i = j + r * RO;
            v[r] = i < n ? in(w, i) : make_double2(0.0, 0.0);
        }
        dft_hin<RE, false>(v);
#pragma unroll
        for (int r = 0; r < RE; ++r) A[(j * RE + r) * es + w] = v[r];
    }
}
// Second step: row k then holds H(k).
template <int RE, int RO>
HD void dhat_2(double2* A, int es, int W, const double2* tw, int tid, int nthr) {
    for (int t = tid; t < W * RE; t += nthr) {
        const int w = t % W, j = t / W;
        double2 v[RO];
#pragma unroll
        for (int r = 0; r < RO; ++r) {
            v[r] = A[(j + r * RE) * es + w];
            if (r) v[r] = v[r] * tw[r * RE + j];
        }
        Dft<RO, false, double2>::run(v);
#pragma unroll
        for (int r = 0; r < RO; ++r) A[(j + r * RE) * es + w] = v[r];
    }
}
HD double2 dhat_fold(const double2* A, int es, int L, int k, int w, bool odd) {
    const double2 a = A[k * es + w], b = A[(k ? L - k : 0) * es + w];
    return odd ? a - b : a + b;
}

}  // namespace eels
