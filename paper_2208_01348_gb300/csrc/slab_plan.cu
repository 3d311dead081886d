// Plans of the transforms: the two radices of an axis and the split of a slab
// over blocks, threads and warps.
#include <algorithm>

#include "kernels.h"

namespace eels {

// Shared memory of a slab block (SlabSmem in k_slab.cuh).
size_t slab_smem(const LatticeDev& L, const SlabPlan& p, size_t el) {
    const size_t lp = (size_t)L.qz.Ro * (L.qz.Re + 1);
    return (size_t)L.Ny * sizeof(int4) +
           ((size_t)L.My + L.Mz + 2 * EELS_MAX_MAT + (size_t)L.My * p.sls + (size_t)(p.nthr / 32) * p.G * lp) * el;
}

Plan2 make_plan2(int L) {
#define PLAN(RE, RO) \
    if (RE * RO == L) return Plan2{L, RE, RO, fast_div(RE), fast_div(RO)};
    EELS_PLANS(PLAN)
#undef PLAN
    return Plan2{};
}

// Threads per block, rows per warp and blocks per slab.  A warp instruction
// costs the same however many of its lanes work, so the split is the one that
// takes the fewest of them per slab (a z step of a warp keeps G Ro and then
// G Re lanes busy, a y step the block's columns times Ro and Re), weighed by
// the warps that the shared memory leaves on an SM: the exchange tiles of more
// rows in flight are paid for with resident blocks.  Registers allow 24 warps
// per SM in FP32 (80 a thread) and 16 in FP64 (128).  A block alone on its SM
// waits at its barriers with nothing beside it (the rod's 48 x 144 slabs: 0.80
// ms with one block of 24 warps, 0.47 ms with three of 8).
//
// FP32, and FP64 slabs of up to 8192 points (4096 with 128 and more along z): more
// than one block per slab pays cluster barriers and remote shared-memory accesses
// (+70 % in FP32, +30 % in FP64): only where one does not fit, or too few of its
// warps do.  In a sweep over lattices of 11 to 96 cells the splits chosen here came
// within 6 % of the fastest of 100 per lattice.
//
// Larger FP64 slabs are bound by the FP64 pipe, where idle lanes cost as much as busy
// ones: the z transforms may run over the rows of a whole block (wide), warps without
// a column issue nothing, and two or four blocks per slab cost next to nothing (eight
// 30 %).  Slabs that leave some of the 152 SMs idle take more blocks: one and a half
// systems are reckoned with, since the lattice alone decides.  (By this rule smaller
// slabs of short z lines gain with one or two systems and lose up to 14 % with more.)
// Fitted to 91 sets of lattice and batch, up to 400 splits each: 0.9 % above the
// fastest matvec on average, 10 % at worst.  us a matvec with the rule of the small
// slabs, as chosen here, and with the five passes of run-time stages that such
// lattices had before:
//   12 x  96 x 125 cells, 3 systems  2991, 1889, 1867
//   12 x 120 x 120                   2832, 2074, 2204
//   12 x  48 x 108                    855,  760,  784
//   30 x  80 x 125        2 systems  4313, 2914, 2800
//    1 x 128 x 128        1 system    207,  207,  125
// Lattices of a few cells along x, whose slabs do not fill the chip, and of 250 points
// along z (radices 10 and 25) are what stays behind those.
SlabPlan make_slab_plan(const LatticeDev& L, size_t el) {
    const Plan2 &y = L.qy, &z = L.qz;
    const bool fp64 = el == sizeof(double2), large = fp64 && (L.My * L.Mz > 8192 || (L.My * L.Mz >= 4096 && L.Mz >= 128));
    const int most = fp64 ? 512 : 768, enough = large ? 12 : most / 32;
    const double slowest = large ? 6 : 4;
    auto remote = [&](int cl) { return cl == 1 ? 1.0 : !fp64 ? 1.7 : !large || cl == 8 ? 1.3 : cl == 2 ? 1.03 : 1.0; };
    auto idle = [&](int cl) { return large ? std::max(1.0, 152 / (4.5 * std::max(1, L.Nx) * cl)) : 1.0; };
    auto iters = [](int items, int lanes) { return (items + lanes - 1) / lanes; };
    SlabPlan best{};
    double best_cost = 0;
    for (int cl : {1, 2, 4, 8}) {
        SlabPlan p{};
        p.CL = cl;
        p.cpc = (L.Nz + cl - 1) / cl;
        p.rpc = (L.My + cl - 1) / cl;
        p.sls = p.cpc | 1;
        p.dcpc = fast_div(p.cpc);
        for (int nthr : {64, 96, 128, 192, 256, 384, 512, 768}) {
            if (nthr > most) break;
            for (int g = 1; g <= 16; ++g) {
                p.nthr = nthr;
                p.G = g;
                const size_t sm = slab_smem(L, p, el);
                if (sm > 224 * 1024) break;
                const int blocks = std::min((int)(227 * 1024 / (sm + 1024)), most / nthr), nw = nthr / 32;
                if (blocks < 1) continue;
                // instructions of all warps, and of the slowest one, which a small batch waits for
                const double ychain = iters(p.cpc * y.Ro, nthr) * y.Re + iters(p.cpc * y.Re, nthr) * y.Ro;
                const double ywork = large ? iters(p.cpc * y.Ro, 32) * y.Re + iters(p.cpc * y.Re, 32) * y.Ro : nw * ychain;
                for (p.wide = 0; p.wide <= large; ++p.wide) {
                    // one turn of n rows, and how many: full ones and the rest
                    const int turn = p.wide ? g * nw : g, full = p.rpc / turn, rest = p.rpc % turn;
                    auto zt = [&](int n, int lanes) { return iters(n * z.Ro, lanes) * z.Re + iters(n * z.Re, lanes) * z.Ro; };
                    const double zwork = p.wide ? full * zt(turn, 32) + zt(rest, 32) : iters(p.rpc, g) * zt(g, 32);
                    const double zchain = p.wide ? full * zt(turn, nthr) + zt(rest, nthr) : iters(p.rpc, g * nw) * zt(g, 32);
                    const double cost = cl * remote(cl) * idle(cl) *
                                        (ywork + zwork + slowest * (ychain + zchain)) * (1.0 + 0.7 / (blocks * blocks)) *
                                        std::max(1.0, (double)enough / (blocks * nw));
                    if (!best.nthr || cost < best_cost * 0.999) { best = p; best_cost = cost; }
                }
            }
        }
    }
    return best;
}

}  // namespace eels
