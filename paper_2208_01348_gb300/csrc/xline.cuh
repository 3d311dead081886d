// Phases of the shared-memory x pass (k_xline.cuh): forward x transforms of
// the three components of W kz-adjacent lines, the symmetric D-hat product
// and the inverse transforms, for L = RE * RO points.
//
// The 3W lines are interleaved in one buffer A[L][3W]; place (set a, j) of a
// line sits in row a RE + j.  The middle step reads row j + r RE (r < RO) of
// the three components, finishes the forward transform (elements
// kx = j + r RE), multiplies by D-hat and starts the inverse transform on the
// same elements, all in registers (xline_mid), or a lane does so for one
// component and takes the products from its neighbours (xline_mid_in, _out).
#pragma once
#include "dft.cuh"

namespace eels {

// Octant of D-hat: address of (kx, ky, kz) in [6][Hy][Hx][Hz] and the signs
// of the odd components (D(M - k) = +-D(k)).
HD float flip(float v, bool neg) { return neg ? -v : v; }
HD double flip(double v, bool neg) { return neg ? -v : v; }
template <typename C> HD C flip_c(C v, bool neg) { v.x = flip(v.x, neg); v.y = flip(v.y, neg); return v; }

// Step 1 forward: in(c, w, ix) for ix < n.
template <int RE, int RO, typename C, class In>
HD void xline_1(C* A, int lgw, int n, int tid, int nthr, In in) {
    const int W = 1 << lgw, es = 3 * W, total = es * RO;
    for (int t = tid; t < total; t += nthr) {
        const int w = t & (W - 1), q = t >> lgw, c = q % 3, j = q / 3;
        C v[RE];
#pragma unroll
        for (int r = 0; r < RE / 2; ++r) {
            const int ix = j + r * RO;
            v[r] = ix < n ? in(c, w, ix) : mk<C>(0.0, 0.0);
        }
        dft_hin<RE, false>(v);
        C* d = A + (size_t)(j * RE) * es + c * W + w;
#pragma unroll
        for (int r = 0; r < RE; ++r) d[r * es] = v[r];
    }
}
// Middle step; dhat(w, kx, d) fills the six signed components at (kx, this
// block's ky, kz of line w).
template <int RE, int RO, typename C, class Dh>
HD void xline_mid(C* A, int lgw, int nw, const C* tw, int tid, int nthr, Dh dhat) {
    const int W = 1 << lgw, es = 3 * W, total = W * RE;
    for (int t = tid; t < total; t += nthr) {
        const int w = t & (W - 1), j = t >> lgw;
        if (w >= nw) continue;
        C v[3][RO];
        C* d = A + (size_t)j * es + w;
#pragma unroll
        for (int r = 0; r < RO; ++r) {
            const C f = tw[r * RE + j];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                v[c][r] = d[(size_t)r * RE * es + c * W];
                if (r) v[c][r] = v[c][r] * f;
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) Dft<RO, false, C>::run(v[c]);
#pragma unroll
        for (int r = 0; r < RO; ++r) {
            C g[6];
            dhat(w, j + r * RE, g);
            const C X = v[0][r], Y = v[1][r], Z = v[2][r];
            v[0][r] = g[0] * X + g[1] * Y + g[2] * Z;
            v[1][r] = g[1] * X + g[3] * Y + g[4] * Z;
            v[2][r] = g[2] * X + g[4] * Y + g[5] * Z;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) Dft<RO, true, C>::run(v[c]);
#pragma unroll
        for (int r = 0; r < RO; ++r) {
            const C f = conj_(tw[r * RE + j]);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                if (r) v[c][r] = v[c][r] * f;
                d[(size_t)r * RE * es + c * W] = v[c][r];
            }
        }
    }
}
// The middle step of one component of one line, as three lanes share it: up to
// the end of the forward transform, and from the start of the inverse one.  d is
// row j of the component and line, es the row length, tw the twiddle (0, j).
template <int RE, int RO, typename C> HD void xline_mid_in(const C* d, int es, const C* tw, C (&v)[RO]) {
#pragma unroll
    for (int r = 0; r < RO; ++r) {
        v[r] = d[(size_t)r * RE * es];
        if (r) v[r] = v[r] * tw[r * RE];
    }
    Dft<RO, false, C>::run(v);
}
template <int RE, int RO, typename C> HD void xline_mid_out(C* d, int es, const C* tw, C (&v)[RO]) {
    Dft<RO, true, C>::run(v);
#pragma unroll
    for (int r = 0; r < RO; ++r) {
        if (r) v[r] = v[r] * conj_(tw[r * RE]);
        d[(size_t)r * RE * es] = v[r];
    }
}
// Row c of the symmetric tensor xx xy xz yy yz zz, in the order of the
// components c, c + 1, c + 2 (mod 3), and the sign of an off-diagonal entry
// where the frequency lies in the upper half along (x, y, z).
HD int sym_own(int c) { return c == 0 ? 0 : c == 1 ? 3 : 5; }
HD int sym_next(int c) { return c == 0 ? 1 : c == 1 ? 4 : 2; }
HD int sym_prev(int c) { return c == 0 ? 2 : c == 1 ? 1 : 4; }
HD bool sym_flip(int i, bool nx, bool ny, bool nz) { return i == 1 ? nx != ny : i == 2 ? nx != nz : ny != nz; }
// Step 2 inverse: out(c, w, ix, value) for ix < n.
template <int RE, int RO, typename C, class Out>
HD void xline_2(const C* A, int lgw, int n, int tid, int nthr, Out out) {
    const int W = 1 << lgw, es = 3 * W, total = es * RO;
    for (int t = tid; t < total; t += nthr) {
        const int w = t & (W - 1), q = t >> lgw, c = q % 3, j = q / 3;
        const C* d = A + (size_t)(j * RE) * es + c * W + w;
        C v[RE];
#pragma unroll
        for (int r = 0; r < RE; ++r) v[r] = d[r * es];
        dft_hout<RE, true>(v);
#pragma unroll
        for (int r = 0; r < RE / 2; ++r) {
            const int ix = j + r * RO;
            if (ix < n) out(c, w, ix, v[r]);
        }
    }
}

}  // namespace eels
