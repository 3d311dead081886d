// Phases of the fused slab passes (k_slab.cuh): one cluster of CL blocks owns
// the x-slab ix of one (system, component).
//
// Forward:  y1, y2   transform the slab's Nz columns along y in place in
//                    shared memory: block r of the cluster holds the columns
//                    iz in [r cpc, (r+1) cpc), S[ky][column];
//           z1, z2   transform the rows ky in [r rpc, (r+1) rpc) along z: step
//                    1 reads a row from the shared memory of all the
//                    cluster's blocks, step 2 writes it to U.
// Inverse:  z1, z2   rows of U, first Nz outputs into the owners' S;
//           y1, y2   the block's columns, first Ny outputs combined with x and
//                    scattered.
// A warp takes G rows at a time through a private exchange tile
// T[G][Ro][Re + 1] (the odd stride keeps both steps' accesses off each
// other's banks), so the z phase needs no block barrier; with the wide form
// (large FP64 slabs, SlabRows in k_slab.cuh) the block's warps share G rows each
// and their tiles, and two block barriers follow a turn.
//
// What bounds it: instruction issue and the latency of the gather and of U in
// FP32 (the rod's 48 x 144 slabs, 256 systems: 0.47 ms forward and 0.54 ms
// back against 0.17 ms for their DRAM traffic), the FP64 pipe in FP64.  Two
// radices per line (one exchange) with the lengths compiled in, in place of
// one thread per butterfly of three or four run-time Stockham stages with a
// block barrier each: 1.50 and 1.40 ms before.  Half of every line is zero on
// the way in and unwanted on the way out, and is neither computed nor moved.
#pragma once
#include "dft.cuh"
#include "kernels.h"

namespace eels {

// One phase's geometry as the threads see it.
template <typename Rl> struct SlabCtx {
    using C = cx<Rl>;
    const C* twy;                 // w_My^(r j) at [r][j], r < Ro, j < Re (step-2 twiddles)
    const C* twz;
    C* S;                         // this block's columns, [My][sls]
    int sls;
    int c0, ncol;                 // this block's columns iz = c0 + c
    int r0, nrow;                 // this block's rows ky
};

// The radices of an axis: at run time, or compiled in (every stride is then
// an immediate offset).
struct RtPlan {
    const Plan2& p;
    HD int Re() const { return p.Re; }
    HD int Ro() const { return p.Ro; }
    HD int div_re(int t) const { return (int)p.dRe.div(t); }
    HD int div_ro(int t) const { return (int)p.dRo.div(t); }
};
template <int RE, int RO> struct CtPlan {
    HD static constexpr int Re() { return RE; }
    HD static constexpr int Ro() { return RO; }
    HD static int div_re(int t) { return t / RE; }
    HD static int div_ro(int t) { return t / RO; }
};

// ---------------------------------------------------------------- y phase
// Step 1 of the forward y transforms (R = Re); in(c, y) is the gathered input.
template <int R, typename Rl, class P, class In>
HD void slab_y1(const SlabCtx<Rl>& s, P p, FastDiv dcol, int n, int tid, int nthr, In in) {
    using C = cx<Rl>;
    const int total = s.ncol * p.Ro();
    for (int t = tid; t < total; t += nthr) {
        const int j = (int)dcol.div(t), c = t - j * s.ncol;
        C v[R];
#pragma unroll
        for (int r = 0; r < R / 2; ++r) {
            const int y = j + r * p.Ro();
            v[r] = y < n ? in(c, y) : mk<C>(0.0, 0.0);
        }
        dft_hin<R, false>(v);
        C* d = s.S + (j * R) * s.sls + c;
#pragma unroll
        for (int r = 0; r < R; ++r) d[r * s.sls] = v[r];
    }
}
// The middle step (R = Ro), in place: forward step 2 (twiddles before) or
// inverse step 1 (conjugate twiddles after).
template <int R, bool INV, typename Rl, class P>
HD void slab_ymid(const SlabCtx<Rl>& s, P p, FastDiv dcol, int tid, int nthr) {
    using C = cx<Rl>;
    const int total = s.ncol * p.Re(), st = p.Re() * s.sls;
    for (int t = tid; t < total; t += nthr) {
        const int j = (int)dcol.div(t), c = t - j * s.ncol;
        C* d = s.S + j * s.sls + c;
        const C* w = s.twy + j;
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            v[r] = d[r * st];
            if (!INV && r) v[r] = v[r] * w[r * p.Re()];
        }
        Dft<R, INV, C>::run(v);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (INV && r) v[r] = v[r] * conj_(w[r * p.Re()]);
            d[r * st] = v[r];
        }
    }
}
// Step 2 of the inverse y transforms (R = Re); out(c, y, value) for y < n.
template <int R, typename Rl, class P, class Out>
HD void slab_y2i(const SlabCtx<Rl>& s, P p, FastDiv dcol, int n, int tid, int nthr, Out out) {
    using C = cx<Rl>;
    const int total = s.ncol * p.Ro();
    for (int t = tid; t < total; t += nthr) {
        const int j = (int)dcol.div(t), c = t - j * s.ncol;
        const C* d = s.S + (j * R) * s.sls + c;
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = d[r * s.sls];
        dft_hout<R, true>(v);
#pragma unroll
        for (int r = 0; r < R / 2; ++r) {
            const int y = j + r * p.Ro();
            if (y < n) out(c, y, v[r]);
        }
    }
}

// ---------------------------------------------------------------- z phase
// g rows; nl lanes (a warp, or a whole block) share their butterflies.  in and
// out return the address of element z (or kz) of row q.
template <int R, typename C, class P, class In>
HD void slab_z1(P p, int n, int g, C* T, int lane, In in, int nl = 32) {
    const int total = g * p.Ro(), lp = p.Ro() * (R + 1);
    for (int t = lane; t < total; t += nl) {
        const int q = p.div_ro(t), j = t - q * p.Ro();
        C v[R];
#pragma unroll
        for (int r = 0; r < R / 2; ++r) {
            const int z = j + r * p.Ro();
            v[r] = z < n ? *in(q, j, r * p.Ro()) : mk<C>(0.0, 0.0);
        }
        dft_hin<R, false>(v);
        C* d = T + q * lp + j * (R + 1);
#pragma unroll
        for (int r = 0; r < R; ++r) d[r] = v[r];
    }
}
template <int R, typename C, class P, class Out>
HD void slab_z2(P p, int g, const C* T, const C* tw, int lane, Out out, int nl = 32) {
    const int total = g * p.Re(), lp = R * (p.Re() + 1);
    for (int t = lane; t < total; t += nl) {
        const int q = p.div_re(t), j = t - q * p.Re();
        const C* d = T + q * lp + j;
        const C* w = tw + j;
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            v[r] = d[r * (p.Re() + 1)];
            if (r) v[r] = v[r] * w[r * p.Re()];
        }
        Dft<R, false, C>::run(v);
        C* o = out(q, j);
#pragma unroll
        for (int r = 0; r < R; ++r) o[r * p.Re()] = v[r];
    }
}
template <int R, typename C, class P, class In>
HD void slab_z1i(P p, int g, C* T, const C* tw, int lane, In in, int nl = 32) {
    const int total = g * p.Re(), lp = R * (p.Re() + 1);
    for (int t = lane; t < total; t += nl) {
        const int q = p.div_re(t), j = t - q * p.Re();
        const C* i = in(q, j);
        const C* w = tw + j;
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = i[r * p.Re()];
        Dft<R, true, C>::run(v);
        C* d = T + q * lp + j;
#pragma unroll
        for (int r = 0; r < R; ++r) d[r * (p.Re() + 1)] = r ? v[r] * conj_(w[r * p.Re()]) : v[r];
    }
}
template <int R, typename C, class P, class Out>
HD void slab_z2i(P p, int n, int g, const C* T, int lane, Out out, int nl = 32) {
    const int total = g * p.Ro(), lp = p.Ro() * (R + 1);
    for (int t = lane; t < total; t += nl) {
        const int q = p.div_ro(t), j = t - q * p.Ro();
        const C* d = T + q * lp + j * (R + 1);
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = d[r];
        dft_hout<R, true>(v);
#pragma unroll
        for (int r = 0; r < R / 2; ++r) {
            const int z = j + r * p.Ro();
            if (z < n) *out(q, j, r * p.Ro()) = v[r];
        }
    }
}

#define EELS_SWITCH_RE(re, CALL) \
    switch (re) { EELS_RE_LIST(CALL) default: break; }
#define EELS_SWITCH_RO(ro, CALL) \
    switch (ro) { EELS_RO_LIST(CALL) default: break; }

}  // namespace eels
