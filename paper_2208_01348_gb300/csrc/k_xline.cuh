// Shared-memory x pass (see xline.cuh), one kernel per padded length.
//
// Block: W z-adjacent lines of the three components at fixed ky, for up to
// spb consecutive systems.  In FP32 the D-hat rows of those lines (octant
// kx', six components) are copied into shared memory while step 1 runs, once
// per D-hat slot (the beams of an energy share it); FP64 is bound by its
// arithmetic and reads D-hat where it needs it, leaving the shared memory to
// more blocks.  Two block barriers per system:
// step 1 reads U, the middle step runs in registers (end of the forward
// transform, D-hat product, start of the inverse transform), step 2 writes U;
// step 2 reads the places that the same thread's next step 1 writes.
//
// FP32 is bound by latency (12 warps per SM at 160 points: shared memory), FP64
// by its pipe.  160-point lines, 4 systems of 79^3 cells: 0.27 ms, against
// 0.37 ms for one thread per butterfly of three run-time stages with D-hat
// read from L2 in the product (0.31 ms with the middle in registers but D-hat
// still read there).
#pragma once
#include <cuda_pipeline.h>

#include <algorithm>

#include "kernels.h"
#include "xline.cuh"

namespace eels {

template <typename Rl> __device__ __forceinline__ const cx<Rl>* xline_tw(const LatticeDev& L);
template <> __device__ __forceinline__ const double2* xline_tw<double>(const LatticeDev& L) { return L.tw64x; }
template <> __device__ __forceinline__ const float2* xline_tw<float>(const LatticeDev& L) { return L.tw32x; }

template <typename C> __device__ __forceinline__ C shfl_c(C v, int l) {
    v.x = __shfl_sync(0xffffffffu, v.x, l);
    v.y = __shfl_sync(0xffffffffu, v.y, l);
    return v;
}

// SPLIT (FP64, lattices of at most 32768 padded points): the middle step of a
// line and butterfly is shared by three lanes, one a component.  Such a grid gives
// a scheduler one warp or none, and a warp's FP64 instruction takes 64 cycles of
// its scheduler even when it is alone there (76 with all four of an SM busy), so
// the step's 312 instructions in a row are the kernel.  Where there are warps enough
// it costs more than it gives (idle lanes, shuffles).  The lattice alone decides: the
// compiler fuses the two forms' products differently, and a system's bits must not
// depend on the batch.  So the line lies where few systems stop gaining, although
// many systems of the smaller lattices lose.  us a matvec, one lane and three:
//   12^3 cells   1 system 42.5, 36.7    2: 52.1, 44.6    4: 62.3, 66.4   256: 1713, 1839
//   14^3         1: 71.9, 54.8          2: 74.6, 61.0    4: 86.2, 90.3
//   16^3         1: 56.9, 48.7          2: 57.6, 58.2    4: 83.2, 87.6    64: 778, 880
//   11 x 11 x 31 1: 61.7, 57.6          2: 69.9, 73.9   16: 266, 286
//   18^3         1: 90.3, 96.5          2: 109, 121     16: 576, 626
//   20^3         1: 96.5, 103           4: 206, 227    128: 5032, 5668
template <typename Rl, int RE, int RO, bool SPLIT>
__global__ void __launch_bounds__(SPLIT ? 512 : 256, sizeof(Rl) == 4 && RO <= 10 ? (RO <= 6 ? 3 : 2) : 1)
k_xline(LatticeDev L, MatvecArgs<Rl> a, int lgw) {
    using C = cx<Rl>;
    dep_wait(a.dep);
    constexpr int LEN = RE * RO, HX = LEN / 2 + 1;
    const int s0 = blockIdx.z * a.spb, s1 = min(a.S, s0 + a.spb);
    const int W = 1 << lgw, ky = blockIdx.y, kz0 = blockIdx.x << lgw;
    const int Mz = L.Mz, Nx = L.Nx;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* tw = reinterpret_cast<C*>(smem_raw);             // w^(r j) at [r][j]
    C* A = tw + LEN;                                    // [LEN][3][W]
    C* D = A + 3 * LEN * W;                             // [6][HX][W] (FP32)
    constexpr bool STAGE = sizeof(Rl) == 4;
    const C* twg = xline_tw<Rl>(L);
    for (int t = threadIdx.x; t < LEN; t += blockDim.x) tw[t] = twg[(t / RE) * (t % RE)];
    const size_t plane = (size_t)Nx * Mz, cstride = (size_t)L.My * plane;
    const int nw = min(W, Mz - kz0), hz = Mz / 2;
    const bool ny = ky > L.My / 2;
    const size_t cs = (size_t)L.Hy * L.Hx * L.Hz;
    const int lane = threadIdx.x & 31, gl = lane / 3, c = lane - 3 * gl;
    const int l1 = min(31, 3 * gl + (c + 1) % 3), l2 = min(31, 3 * gl + (c + 2) % 3);
    int cur = -1;
    for (int s = s0; s < s1; ++s) {
        if (a.active && !a.active[s]) continue;
        const int slot = a.sys_slot[s];
        const C* Ds = a.Dr + (size_t)slot * 6 * cs + (size_t)(ny ? L.My - ky : ky) * L.Hx * L.Hz;
        if (STAGE && slot != cur) {                     // every thread is past the middle step that read D
            for (int t = threadIdx.x; t < 6 * HX * W; t += blockDim.x) {
                const int w = t & (W - 1), q = t >> lgw, c = q / HX, kx = q - c * HX, kz = kz0 + w;
                if (w < nw)
                    __pipeline_memcpy_async(D + t, Ds + c * cs + (size_t)kx * L.Hz + (kz > hz ? Mz - kz : kz), sizeof(C));
            }
            cur = slot;
        }
        C* U0 = a.U + ((size_t)s * 3 * L.My + ky) * plane + kz0;
        xline_1<RE, RO>(A, lgw, Nx, threadIdx.x, blockDim.x, [&](int c, int w, int ix) -> C {
            return w < nw ? U0[c * cstride + (size_t)ix * Mz + w] : mk<C>(0.0, 0.0);
        });
        if (STAGE) {
            __pipeline_commit();
            __pipeline_wait_prior(0);
        }
        __syncthreads();
        if constexpr (SPLIT) {
            // ten triples of lanes a warp, one triple a line and butterfly
            for (int g0 = (threadIdx.x >> 5) * 10; g0 < RE << lgw; g0 += (blockDim.x >> 5) * 10) {
                const int g = g0 + gl, w = g & (W - 1), j = g >> lgw, kz = kz0 + w;
                const bool ok = lane < 30 && j < RE && w < nw, nz = kz > hz;
                C v[RO];
                C* d = A + (ok ? j * 3 * W + c * W + w : 0);
                const C* tj = tw + (ok ? j : 0);
                xline_mid_in<RE, RO>(d, 3 * W, tj, v);
#pragma unroll
                for (int r = 0; r < RO; ++r) {
                    const int kx = j + r * RE, kxr = kx > LEN / 2 ? LEN - kx : kx;
                    const bool nx = kx > LEN / 2;
                    const C next = shfl_c(v[r], l1), prev = shfl_c(v[r], l2);
                    if (!ok) continue;
                    const C* q = Ds + (size_t)kxr * L.Hz + (nz ? Mz - kz : kz);
                    v[r] = q[sym_own(c) * cs] * v[r] +
                           flip_c(q[sym_next(c) * cs], sym_flip(sym_next(c), nx, ny, nz)) * next +
                           flip_c(q[sym_prev(c) * cs], sym_flip(sym_prev(c), nx, ny, nz)) * prev;
                }
                if (ok) xline_mid_out<RE, RO>(d, 3 * W, tj, v);
            }
        } else {
            xline_mid<RE, RO>(A, lgw, nw, tw, threadIdx.x, blockDim.x, [&](int w, int kx, C (&g)[6]) {
                const int kz = kz0 + w, kxr = kx > LEN / 2 ? LEN - kx : kx;
                const bool nx = kx > LEN / 2, nz = kz > hz;
                const C* d = STAGE ? D + (kxr << lgw) + w : Ds + (size_t)kxr * L.Hz + (nz ? Mz - kz : kz);
                const size_t st = STAGE ? (size_t)(HX << lgw) : cs;
                g[0] = d[0];
                g[1] = flip_c(d[st], nx != ny);
                g[2] = flip_c(d[2 * st], nx != nz);
                g[3] = d[3 * st];
                g[4] = flip_c(d[4 * st], ny != nz);
                g[5] = d[5 * st];
            });
        }
        __syncthreads();
        xline_2<RE, RO>(A, lgw, Nx, threadIdx.x, blockDim.x, [&](int c, int w, int ix, C v) {
            if (w < nw) U0[c * cstride + (size_t)ix * Mz + w] = v;
        });
    }
}

template <typename Rl> size_t xline_smem(const LatticeDev& L, int w) {
    return (size_t)(L.Mx + 3 * w * L.Mx + (sizeof(Rl) == 4 ? 6 * w * (L.Mx / 2 + 1) : 0)) * sizeof(cx<Rl>);
}
template <typename Rl> bool xline_fits(const LatticeDev& L, int w) { return xline_smem<Rl>(L, w) <= 224 * 1024; }

template <typename Rl> static bool xline_split(const LatticeDev& L) {
    return sizeof(Rl) == 8 && (long long)L.Mx * L.My * L.Mz <= 32768;
}

template <typename Rl> void launch_xline(const LatticeDev& L, const MatvecArgs<Rl>& a, int w, cudaStream_t st) {
    int lgw = 0;
    while ((2 << lgw) <= w) ++lgw;
    // a grid that leaves SMs idle takes narrower tiles (the lines do not depend on the tile they are in):
    // 144 blocks of 4 lines instead of 72 of 8 for one 12^3 system
    while (lgw > 1 && (long long)((L.Mz + (1 << lgw) - 1) >> lgw) * L.My * a.S < 100) --lgw;
    // systems per block: several when they can share D-hat and the grid stays large
    const int tiles = ((L.Mz + (1 << lgw) - 1) >> lgw) * L.My;
    MatvecArgs<Rl> b = a;
    b.spb = std::max(1, std::min(a.spb, a.S));
    while (b.spb > 1 && (long long)tiles * ((a.S + b.spb - 1) / b.spb) < 1216) b.spb /= 2;
    const dim3 grid((L.Mz + (1 << lgw) - 1) >> lgw, L.My, (a.S + b.spb - 1) / b.spb);
    const bool split = xline_split<Rl>(L);
    const int items = L.qx.Re << lgw;
    const int nthr = split ? std::min(512, std::max(64, (items + 9) / 10 * 32))
                           : std::min(256, std::max(64, (items + 31) / 32 * 32));
    const size_t sm = xline_smem<Rl>(L, 1 << lgw);
    count_launch();
    switch (L.Mx) {
#define XL(RE, RO)                                                                            \
    case RE * RO:                                                                             \
        if (split) launch_dep(b.dep, k_xline<Rl, RE, RO, sizeof(Rl) == 8>, grid, nthr, sm, 1, st, L, b, lgw); \
        else launch_dep(b.dep, k_xline<Rl, RE, RO, false>, grid, nthr, sm, 1, st, L, b, lgw);             \
        break;
        EELS_PLANS(XL)
#undef XL
        default: break;
    }
}

template <typename K> static void prepare_xline(K k) {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024);
    cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
}
template <typename Rl> void prepare_xline_kernels() {
#define XL(RE, RO) prepare_xline(k_xline<Rl, RE, RO, false>); prepare_xline(k_xline<Rl, RE, RO, sizeof(Rl) == 8>);
    EELS_PLANS(XL)
#undef XL
}

}  // namespace eels
