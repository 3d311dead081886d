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
// ms with one block of 24 warps, 0.47 ms with three of 8).  More than one
// block per slab pays cluster barriers and remote shared-memory accesses
// (+70 % in FP32, +30 % in FP64): only where one does not fit, or too few of
// its warps do.  In a sweep over lattices of 11 to 96 cells the splits chosen
// here came within 6 % of the fastest of 100 per lattice.
SlabPlan make_slab_plan(const LatticeDev& L, size_t el) {
    const Plan2 &y = L.qy, &z = L.qz;
    const int most = el == 8 ? 768 : 512, enough = most / 32;
    const double remote = el == 8 ? 1.7 : 1.3;
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
                const double zc = iters(g * z.Ro, 32) * z.Re + iters(g * z.Re, 32) * z.Ro;
                const double yc = iters(p.cpc * y.Ro, nthr) * y.Re + iters(p.cpc * y.Re, nthr) * y.Ro;
                const double work = nw * yc + iters(p.rpc, g) * zc;
                // the slowest warp of the block (a small batch waits for it)
                const double chain = yc + iters(p.rpc, g * nw) * zc;
                const double cost = cl * (cl > 1 ? remote : 1.0) * (work + 4 * chain) * (1.0 + 0.7 / (blocks * blocks)) *
                                    std::max(1.0, (double)enough / (blocks * nw));
                if (!best.nthr || cost < best_cost * 0.999) { best = p; best_cost = cost; }
            }
        }
    }
    return best;
}

}  // namespace eels
