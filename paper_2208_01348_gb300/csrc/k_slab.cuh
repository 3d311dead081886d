// Fused slab passes of the matvec for any padded y and z length: gather, y and
// z transforms (forward), and inverse z and y transforms, combination with x
// and scatter (inverse), one cluster of blocks per x-slab of a (system,
// component).  FP32 slabs of 64 x 64 and 128 x 128 points run the
// register-resident kernels of k_fft.cu instead.
#pragma once
#include <cooperative_groups.h>
#include <cuda_pipeline.h>

#include <algorithm>

#include "slab.cuh"

namespace eels {

namespace cg = cooperative_groups;

template <typename Rl> __device__ __forceinline__ const cx<Rl>* slab_tw(const LatticeDev& L, int axis);
template <> __device__ __forceinline__ const double2* slab_tw<double>(const LatticeDev& L, int axis) {
    return axis == 1 ? L.tw64y : L.tw64z;
}
template <> __device__ __forceinline__ const float2* slab_tw<float>(const LatticeDev& L, int axis) {
    return axis == 1 ? L.tw32y : L.tw32z;
}
template <typename Rl> __host__ __device__ __forceinline__ const SlabPlan& plan_of(const LatticeDev& L) {
    return sizeof(Rl) == 4 ? L.s32 : L.s64;
}

// Shared memory of a block: step-2 twiddles of both axes, coefficients, the
// slab's column table, the columns S and the warps' exchange tiles.
template <typename Rl> struct SlabSmem {
    using C = cx<Rl>;
    C *twy, *twz, *cf, *dg, *S, *T;
    int4* ci;
    __device__ SlabSmem(unsigned char* raw, const LatticeDev& L, const SlabPlan& p) {
        ci = reinterpret_cast<int4*>(raw);
        twy = reinterpret_cast<C*>(ci + L.Ny);
        twz = twy + L.My;
        cf = twz + L.Mz;
        dg = cf + EELS_MAX_MAT;
        S = dg + EELS_MAX_MAT;
        T = S + (size_t)L.My * p.sls;
    }
};
// Tables of a block, copied asynchronously in two groups: the column table, then
// the twiddles.
template <typename Rl>
__device__ __forceinline__ void slab_tables(const LatticeDev& L, const MatvecArgs<Rl>& a, const SlabSmem<Rl>& m, int s,
                                            int ix) {
    using C = cx<Rl>;
    if (L.contig)
        for (int t = threadIdx.x; t < L.Ny; t += blockDim.x)
            __pipeline_memcpy_async(m.ci + t, L.colinfo + (size_t)ix * L.Ny + t, sizeof(int4));
    __pipeline_commit();
    const C* gy = slab_tw<Rl>(L, 1);
    const C* gz = slab_tw<Rl>(L, 2);
    for (int t = threadIdx.x; t < L.My; t += blockDim.x) {
        const int r = (int)L.qy.dRe.div(t), j = t - r * L.qy.Re;
        __pipeline_memcpy_async(m.twy + t, gy + r * j, sizeof(C));
    }
    for (int t = threadIdx.x; t < L.Mz; t += blockDim.x) {
        const int r = (int)L.qz.dRe.div(t), j = t - r * L.qz.Re;
        __pipeline_memcpy_async(m.twz + t, gz + r * j, sizeof(C));
    }
    __pipeline_commit();
    if (threadIdx.x < EELS_MAX_MAT) {
        m.cf[threadIdx.x] = cvt<C>(a.coef[(size_t)s * EELS_MAX_MAT + threadIdx.x]);
        m.dg[threadIdx.x] = cvt<C>(a.diag[(size_t)s * EELS_MAX_MAT + threadIdx.x]);
    }
}

// The rows of a thread's z transforms: those of its warp (G at a time), or, with
// the wide form, of its block (G per warp), whose threads then take the butterflies
// of all of them, one row after another.  The FP64 pipe takes a warp's instruction in
// the same time however many of its lanes work, and a warp's own rows leave lanes idle
// wherever G Ro or G Re are not near multiples of 32: with 250 points (radices 10 and
// 25) and G = 1 the slab passes of three systems of 12 x 96 x 125 cells issued 14.4 M and
// 15.2 M FP64 instructions and took 1.07 and 1.05 ms; shared by blocks of twelve warps
// with G = 2 they issue 6.8 M and 7.6 M and take 0.48 and 0.54 ms.  The bits are the
// same.  Two block barriers a turn are what it costs, so slabs whose rows fill their
// warps keep the private form (make_slab_plan).
template <typename Rl> struct SlabRows {
    int lane, nl;                 // place among the threads that share rows
    int first, step, g;           // rows of a turn, and of the next one
    size_t tile;                  // exchange tile
    bool wide;
    __device__ SlabRows(const SlabPlan& p, const Plan2& qz) {
        const int warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
        wide = sizeof(Rl) == 8 && p.wide;
        lane = wide ? threadIdx.x : threadIdx.x & 31;
        nl = wide ? blockDim.x : 32;
        step = nwarp * p.G;
        first = wide ? 0 : warp * p.G;
        g = wide ? step : p.G;
        tile = (size_t)first * qz.Ro * (qz.Re + 1);
    }
    __device__ void sync() const {
        if (wide) __syncthreads();
        else __syncwarp();
    }
};

template <typename Rl, bool CLUSTER>
__global__ void __launch_bounds__(sizeof(Rl) == 4 ? 768 : 512, 1) k_slab_fwd(LatticeDev L, MatvecArgs<Rl> a) {
    using C = cx<Rl>;
    dep_wait(a.dep);
    const SlabPlan& sp = plan_of<Rl>(L);
    const int CL = CLUSTER ? sp.CL : 1, rank = CLUSTER ? blockIdx.x % CL : 0, ix = CLUSTER ? blockIdx.x / CL : blockIdx.x;
    const int b = blockIdx.y, s = b / 3, c = b % 3;
    if (a.active && !a.active[s]) return;             // the whole cluster leaves: one system per cluster
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const SlabSmem<Rl> m(smem_raw, L, sp);
    slab_tables<Rl>(L, a, m, s, ix);
    __pipeline_wait_prior(1);
    __syncthreads();
    const int Ny = L.Ny, Nz = L.Nz;
    SlabCtx<Rl> sc;
    sc.twy = m.twy; sc.twz = m.twz; sc.S = m.S; sc.sls = sp.sls;
    sc.c0 = rank * sp.cpc; sc.ncol = max(0, min(sp.cpc, Nz - sc.c0));
    sc.r0 = rank * sp.rpc; sc.nrow = max(0, min(sp.rpc, L.My - sc.r0));
    const FastDiv dcol = fast_div(sc.ncol);
    const C* xs = a.x + ((size_t)s * 3 + c) * L.N;
    const int* cm = L.cellmap + (size_t)ix * Ny * Nz;
    const bool contig = L.contig, one_mat = L.nmat == 1;
    const C zero = mk<C>(0.0, 0.0);
    auto gather = [&](int col, int y) -> C {
        const int iz = sc.c0 + col;
        const int dip = contig ? col_dip(m.ci[y], iz) : cm[y * Nz + iz];
        if (dip < 0) return zero;
        return xs[dip] * m.cf[one_mat ? 0 : L.mat[dip]];
    };
    // y transforms of this block's columns
    const RtPlan ry{L.qy}, rz{L.qz};
    if (CLUSTER) {
#define Y1(R) case R: slab_y1<R, Rl>(sc, ry, dcol, Ny, threadIdx.x, blockDim.x, gather); break;
        EELS_SWITCH_RE(L.qy.Re, Y1)
#undef Y1
        __pipeline_wait_prior(0);
        __syncthreads();
#define YM(R) case R: slab_ymid<R, false, Rl>(sc, ry, dcol, threadIdx.x, blockDim.x); break;
        EELS_SWITCH_RO(L.qy.Ro, YM)
#undef YM
    } else {
#define Y(RE, RO)                                                                                     \
    case RE * RO:                                                                                     \
        slab_y1<RE, Rl>(sc, CtPlan<RE, RO>{}, dcol, Ny, threadIdx.x, blockDim.x, gather);             \
        __pipeline_wait_prior(0);                                                                     \
        __syncthreads();                                                                              \
        slab_ymid<RO, false, Rl>(sc, CtPlan<RE, RO>{}, dcol, threadIdx.x, blockDim.x);                \
        break;
        switch (L.My) { EELS_PLANS(Y) default: break; }
#undef Y
    }
    if (CLUSTER) cg::this_cluster().sync();
    else __syncthreads();
    // z transforms of this block's rows
    const SlabRows<Rl> rows(sp, L.qz);
    C* T = m.T + rows.tile;
    C* U = a.U + (((size_t)s * 3 + c) * L.My * L.Nx + ix) * (size_t)L.Mz;
    const size_t urow = (size_t)L.Nx * L.Mz;
    for (int row = sc.r0 + rows.first; row < sc.r0 + sc.nrow; row += rows.step) {
        const int g = min(rows.g, sc.r0 + sc.nrow - row);
        auto out = [&](int q, int kz) -> C* { return U + (size_t)(row + q) * urow + kz; };
        if (CLUSTER) {
            auto in = [&](int q, int j, int dz) -> const C* {
                const int z = j + dz, o = (int)sp.dcpc.div(z);
                return cg::this_cluster().map_shared_rank(m.S, o) + (row + q) * sp.sls + z - o * sp.cpc;
            };
#define Z1(R) case R: slab_z1<R, C>(rz, Nz, g, T, rows.lane, in, rows.nl); break;
            EELS_SWITCH_RE(L.qz.Re, Z1)
#undef Z1
            rows.sync();
#define Z2(R) case R: slab_z2<R, C>(rz, g, T, m.twz, rows.lane, out, rows.nl); break;
            EELS_SWITCH_RO(L.qz.Ro, Z2)
#undef Z2
        } else {
            const C* Sr = m.S + row * sp.sls;
            auto in = [&](int q, int j, int dz) -> const C* { return Sr + q * sp.sls + j + dz; };
#define Z(RE, RO)                                                                     \
    case RE * RO:                                                                     \
        slab_z1<RE, C>(CtPlan<RE, RO>{}, Nz, g, T, rows.lane, in, rows.nl);       \
        rows.sync();                                                                  \
        slab_z2<RO, C>(CtPlan<RE, RO>{}, g, T, m.twz, rows.lane, out, rows.nl);   \
        break;
            switch (L.Mz) { EELS_PLANS(Z) default: break; }
#undef Z
        }
        rows.sync();
    }
    if (CLUSTER) cg::this_cluster().sync();           // other blocks may still read this block's S
}

template <typename Rl, bool CLUSTER>
__global__ void __launch_bounds__(sizeof(Rl) == 4 ? 768 : 512, 1) k_slab_inv(LatticeDev L, MatvecArgs<Rl> a, Rl invM) {
    using C = cx<Rl>;
    dep_wait(a.dep);
    const SlabPlan& sp = plan_of<Rl>(L);
    const int CL = CLUSTER ? sp.CL : 1, rank = CLUSTER ? blockIdx.x % CL : 0, ix = CLUSTER ? blockIdx.x / CL : blockIdx.x;
    const int b = blockIdx.y, s = b / 3, c = b % 3;
    if (a.active && !a.active[s]) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Rl red[2 * 24];
    const SlabSmem<Rl> m(smem_raw, L, sp);
    slab_tables<Rl>(L, a, m, s, ix);
    __pipeline_wait_prior(0);
    if (CLUSTER) cg::this_cluster().sync();           // every block of the cluster runs before the remote stores
    else __syncthreads();
    const int Ny = L.Ny, Nz = L.Nz;
    SlabCtx<Rl> sc;
    sc.twy = m.twy; sc.twz = m.twz; sc.S = m.S; sc.sls = sp.sls;
    sc.c0 = rank * sp.cpc; sc.ncol = max(0, min(sp.cpc, Nz - sc.c0));
    sc.r0 = rank * sp.rpc; sc.nrow = max(0, min(sp.rpc, L.My - sc.r0));
    const FastDiv dcol = fast_div(sc.ncol);
    // inverse z transforms of this block's rows of U, first Nz outputs into the columns' owners
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    const SlabRows<Rl> rows(sp, L.qz);
    C* T = m.T + rows.tile;
    const C* U = a.U + (((size_t)s * 3 + c) * L.My * L.Nx + ix) * (size_t)L.Mz;
    const size_t urow = (size_t)L.Nx * L.Mz;
    for (int row = sc.r0 + rows.first; row < sc.r0 + sc.nrow; row += rows.step) {
        const int g = min(rows.g, sc.r0 + sc.nrow - row);
        auto in = [&](int q, int kz) -> const C* { return U + (size_t)(row + q) * urow + kz; };
        if (CLUSTER) {
            const RtPlan rz{L.qz};
            auto out = [&](int q, int j, int dz) -> C* {
                const int z = j + dz, o = (int)sp.dcpc.div(z);
                return cg::this_cluster().map_shared_rank(m.S, o) + (row + q) * sp.sls + z - o * sp.cpc;
            };
#define Z1(R) case R: slab_z1i<R, C>(rz, g, T, m.twz, rows.lane, in, rows.nl); break;
            EELS_SWITCH_RO(L.qz.Ro, Z1)
#undef Z1
            rows.sync();
#define Z2(R) case R: slab_z2i<R, C>(rz, Nz, g, T, rows.lane, out, rows.nl); break;
            EELS_SWITCH_RE(L.qz.Re, Z2)
#undef Z2
        } else {
            C* Sr = m.S + row * sp.sls;
            auto out = [&](int q, int j, int dz) -> C* { return Sr + q * sp.sls + j + dz; };
#define Z(RE, RO)                                                                     \
    case RE * RO:                                                                     \
        slab_z1i<RO, C>(CtPlan<RE, RO>{}, g, T, m.twz, rows.lane, in, rows.nl);                     \
        rows.sync();                                                                  \
        slab_z2i<RE, C>(CtPlan<RE, RO>{}, Nz, g, T, rows.lane, out, rows.nl);     \
        break;
            switch (L.Mz) { EELS_PLANS(Z) default: break; }
#undef Z
        }
        rows.sync();
    }
    if (CLUSTER) cg::this_cluster().sync();
    else __syncthreads();
    // inverse y transforms of this block's columns, first Ny outputs combined with x and scattered
    const C* xs = a.x + ((size_t)s * 3 + c) * L.N;
    C* ys = a.y + ((size_t)s * 3 + c) * L.N;
    const int* cm = L.cellmap + (size_t)ix * Ny * Nz;
    const bool contig = L.contig, one_mat = L.nmat == 1;
    Rl dot0 = 0, dot1 = 0;
    auto scatter = [&](int col, int y, C v) {
        const int iz = sc.c0 + col;
        const int dip = contig ? col_dip(m.ci[y], iz) : cm[y * Nz + iz];
        if (dip < 0) return;
        const int mt = one_mat ? 0 : L.mat[dip];
        const C xv = xs[dip];
        const C yv = m.dg[mt] * xv - m.cf[mt] * (invM * v);
        ys[dip] = yv;
        dot0 += xv.x * yv.x - xv.y * yv.y;
        dot1 += xv.x * yv.y + xv.y * yv.x;
    };
    if (CLUSTER) {
        const RtPlan ry{L.qy};
#define YM(R) case R: slab_ymid<R, true, Rl>(sc, ry, dcol, threadIdx.x, blockDim.x); break;
        EELS_SWITCH_RO(L.qy.Ro, YM)
#undef YM
        __syncthreads();
#define Y2(R) case R: slab_y2i<R, Rl>(sc, ry, dcol, Ny, threadIdx.x, blockDim.x, scatter); break;
        EELS_SWITCH_RE(L.qy.Re, Y2)
#undef Y2
    } else {
#define Y(RE, RO)                                                                                     \
    case RE * RO:                                                                                     \
        slab_ymid<RO, true, Rl>(sc, CtPlan<RE, RO>{}, dcol, threadIdx.x, blockDim.x);                 \
        __syncthreads();                                                                              \
        slab_y2i<RE, Rl>(sc, CtPlan<RE, RO>{}, dcol, Ny, threadIdx.x, blockDim.x, scatter);           \
        break;
        switch (L.My) { EELS_PLANS(Y) default: break; }
#undef Y
    }
    if (a.dot_part) {
        // block sum in a fixed order (warp shuffles, then thread 0 over the warps)
        for (int o = 16; o > 0; o >>= 1) {
            dot0 += __shfl_xor_sync(0xffffffffu, dot0, o);
            dot1 += __shfl_xor_sync(0xffffffffu, dot1, o);
        }
        if (lane == 0) { red[2 * warp] = dot0; red[2 * warp + 1] = dot1; }
        __syncthreads();
        if (threadIdx.x == 0) {
            double s0 = 0, s1 = 0;
            for (int i = 0; i < nwarp; ++i) { s0 += red[2 * i]; s1 += red[2 * i + 1]; }
            double* p = a.dot_part + ((((size_t)s * 3 + c) * L.Nx + ix) * CL + rank) * 4;
            p[0] = s0; p[1] = s1; p[2] = 0.0; p[3] = 0.0;
        }
    }
}

template <typename Rl>
void launch_slab(const LatticeDev& L, const MatvecArgs<Rl>& a, bool inv, cudaStream_t st) {
    const SlabPlan& p = plan_of<Rl>(L);
    const size_t sm = slab_smem(L, p, sizeof(cx<Rl>));
    const Rl invM = (Rl)(1.0 / ((double)L.Mx * L.My * L.Mz));
    count_launch();
    if (p.CL == 1) {
        const dim3 grid(L.Nx, a.S * 3);
        if (!inv) launch_dep(a.dep, k_slab_fwd<Rl, false>, grid, p.nthr, sm, 1, st, L, a);
        else launch_dep(a.dep, k_slab_inv<Rl, false>, grid, p.nthr, sm, 1, st, L, a, invM);
        return;
    }
    const dim3 grid(L.Nx * p.CL, a.S * 3);
    if (!inv) launch_dep(a.dep, k_slab_fwd<Rl, true>, grid, p.nthr, sm, p.CL, st, L, a);
    else launch_dep(a.dep, k_slab_inv<Rl, true>, grid, p.nthr, sm, p.CL, st, L, a, invM);
}
template <typename K> static void allow(K k) {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024);
    // these kernels keep their working tiles in shared memory: give it the whole carveout
    cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
}
template <typename Rl> void prepare_slab_kernels() {
    allow(k_slab_fwd<Rl, false>); allow(k_slab_fwd<Rl, true>);
    allow(k_slab_inv<Rl, false>); allow(k_slab_inv<Rl, true>);
}

}  // namespace eels
