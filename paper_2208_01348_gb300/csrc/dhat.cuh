// Phases of the D-hat build (k_dhat.cu): one axis of the transform of a
// sequence that is even or odd along it, from its non-negative half to the
// frequencies 0 <= k <= L/2.
//
// Along an axis the padded Green's tensor g holds g(i) at 0 <= i < n, +-g(i) at
// L - i and zero between; its transform F has the same symmetry.  Of the two
// register steps of a line of L = RE RO points, only half is worked out:
//   step 1: the set RO - j is the set j reversed, so its length-RE DFT is
//           T_{RO-j}(k) = +- w_RE^-k T_j(RE - k): the sets j <= RO/2 do;
//   step 2: F(k + RE m) and F(RE - k + RE m') mirror each other: the outputs
//           k <= RE/2 of the sets do, each a length-RO DFT of T_j(k) w^(j k) in
//           place j and +- T_j(RE - k) w^-(j k) in place RO - j.
#pragma once
#include "dft.cuh"

namespace eels {

template <int RE, int RO> struct DhatLine {
    static constexpr int L = RE * RO;
    static constexpr int SETS = RO / 2 + 1;    // j = 0 .. RO/2
    static constexpr int ROWS = SETS * RE;     // row j RE + k holds T_j(k)
    static constexpr int OUTS = RE / 2 + 1;
};

// Step 1 of W lines into A[ROWS][es]; in(w, i) for i < n.
template <int RE, int RO, class In>
HD void dhat_1(double2* A, int es, int W, int n, bool odd, int tid, int nthr, In in) {
    using D = DhatLine<RE, RO>;
    for (int t = tid; t < W * D::SETS; t += nthr) {
        const int j = t / W, w = t - j * W;
        double2 v[RE];
#pragma unroll
        for (int r = 0; r < RE; ++r) {
            const int i = j + r * RO, m = D::L - i;
            v[r] = make_double2(0.0, 0.0);
            if (i < n) {
                if (!odd || i > 0) v[r] = in(w, i);
            } else if (m < n) {
                v[r] = in(w, m);
                if (odd) v[r] = -v[r];
            }
        }
        Dft<RE, false, double2>::run(v);
#pragma unroll
        for (int r = 0; r < RE; ++r) A[(j * RE + r) * es + w] = v[r];
    }
}
// Step 2: out(w, k, F(k)) for every k <= L/2.  tw: w^(j k) at [j][k], j <= RO/2.
template <int RE, int RO, class Out>
HD void dhat_2(const double2* A, int es, int W, bool odd, const double2* tw, int tid, int nthr, Out out) {
    using D = DhatLine<RE, RO>;
    for (int t = tid; t < W * D::OUTS; t += nthr) {
        const int k = t / W, w = t - k * W, kr = k ? RE - k : 0;
        double2 v[RO];
        v[0] = A[k * es + w];
#pragma unroll
        for (int j = 1; j < D::SETS; ++j) {
            const double2 f = tw[j * RE + k];
            v[j] = A[(j * RE + k) * es + w] * f;
            if (2 * j < RO) {
                const double2 b = A[(j * RE + kr) * es + w] * conj_(f);
                v[RO - j] = odd ? -b : b;
            }
        }
        Dft<RO, false, double2>::run(v);
        const bool own = k == 0 || 2 * k == RE;          // its mirror images are its own outputs
#pragma unroll
        for (int m = 0; m < RO; ++m) {
            const int q = k + RE * m;
            if (2 * q <= D::L) out(w, q, odd && (q == 0 || 2 * q == D::L) ? make_double2(0.0, 0.0) : v[m]);
            else if (!own) out(w, D::L - q, odd ? -v[m] : v[m]);
        }
    }
}

}  // namespace eels
