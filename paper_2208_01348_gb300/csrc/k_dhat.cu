// D-hat build: the transform of the six components of the Green's tensor
// (Eq. 5, or the cell-integrated tensor for near offsets) on the padded
// lattice, for n_slot wavenumbers kappa = k d, FP64.
//
//   G~' = exp(i kappa R)/R [kappa^2 (I - RR) - (1 - i kappa R)/R^2 (I - 3 RR)]   (Eq. 5)
//
// The diagonal components are even in each of x, y, z and xy, xz, yz are odd in
// the two axes they name, so only the octant of non-negative offsets is
// evaluated, and each axis is transformed from its non-negative half
// (dhat.cuh) to the frequencies 0 <= k <= M/2 that are kept: 3 N^2 lines per
// component in place of 12 N^2, half of each line's butterflies, and N^3
// exponentials in place of 8 N^3.  The FP64 pipe bounds it (the arrays of one
// energy of 64^3 cells are 25 MB): 0.33 ms per energy of 64^3 cells, against 0.46
// ms with half-filled lines transformed whole and 2.2 ms for the padded
// lattice.  The last axis writes D-hat in the layouts that the x passes read.
#include <algorithm>

#include "dhat.cuh"
#include "kernels.h"

namespace eels {

// G[slot][comp][z][y][x] over the octant, x fastest.
__global__ void k_green(LatticeDev L, const double2* kappa, double2* G) {
    const int n = L.Nx * L.Ny * L.Nz;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n) return;
    const int slot = blockIdx.y;
    const int x = idx % L.Nx, y = idx / L.Nx % L.Ny, z = idx / (L.Nx * L.Ny);
    const double2 kap = kappa[slot];
    double2 g[6];
    for (int c = 0; c < 6; ++c) g[c] = make_double2(0.0, 0.0);
    const double rn2 = (double)(x * x + y * y + z * z);
    if (rn2 > 0.0) {
        const double rn = sqrt(rn2);
        double sn, cs;
        sincos(kap.x * rn, &sn, &cs);
        const double ex = kap.y == 0.0 ? 1.0 : exp(-kap.y * rn);
        const double2 k2 = kap * kap;
        if (L.igt && x <= IGT_NEAR && y <= IGT_NEAR && z <= IGT_NEAR) {
            // cell-averaged tensor to second order in kappa: exp(i kappa R)(-T0 + i kappa T1 + kappa^2 T2)
            const int side = 2 * IGT_NEAR + 1;
            const double* t = L.igt + ((size_t)((z + IGT_NEAR) * side + (y + IGT_NEAR)) * side + (x + IGT_NEAR)) * 18;
            const double2 ph = make_double2(ex * cs, ex * sn);
            const double2 ik = make_double2(-kap.y, kap.x);
            for (int c = 0; c < 6; ++c) g[c] = ph * (make_double2(-t[c], 0.0) + t[6 + c] * ik + t[12 + c] * k2);
        } else {
            const double inv = 1.0 / rn;
            const double h[3] = {x * inv, y * inv, z * inv};
            const double2 ph = make_double2(ex * inv * cs, ex * inv * sn);                       // exp(i kappa R) / R
            const double2 t = (1.0 / rn2) * make_double2(1.0 + kap.y * rn, -kap.x * rn);         // (1 - i kappa R) / R^2
            const int pa[6] = {0, 0, 0, 1, 1, 2}, pb[6] = {0, 1, 2, 1, 2, 2};
            for (int c = 0; c < 6; ++c) {
                const double hh = h[pa[c]] * h[pb[c]], dd = pa[c] == pb[c] ? 1.0 : 0.0;
                g[c] = ph * ((dd - hh) * k2 - (dd - 3.0 * hh) * t);
            }
        }
    }
    double2* out = G + (size_t)slot * 6 * n + idx;
    for (int c = 0; c < 6; ++c) out[(size_t)c * n] = g[c];
}

// A block takes W adjacent lines of one component, a lane each; a warp then
// works on one set or output (a whole number of them: 32 lines) of 32 lines.
template <int RE, int RO> struct DhatBlock : DhatLine<RE, RO> {
    static constexpr int W = RE * RO <= 128 ? 32 : 16;
    static constexpr int THREADS = (W * DhatLine<RE, RO>::SETS + 31) / 32 * 32 < 64 ? 64 : (W * DhatLine<RE, RO>::SETS + 31) / 32 * 32;
    static constexpr int LINE_SMEM = (DhatLine<RE, RO>::ROWS * (W + 1)) * 16;      // twiddles and A
    static_assert(THREADS <= 512, "threads");
};
template <int RE, int RO> __device__ __forceinline__ void dhat_twiddles(double2* tw, const double2* g) {
    for (int t = threadIdx.x; t < DhatLine<RE, RO>::ROWS; t += blockDim.x) tw[t] = g[(t / RE) * (t % RE)];
}

// One axis: line l of n_line has its entries at (l / in_row) * in_fix + l %
// in_row + i * in_line; its frequencies k <= L/2 go to l + k * n_line.
template <int RE, int RO>
__global__ void __launch_bounds__((DhatBlock<RE, RO>::THREADS), 1)
k_dhat_axis(const double2* in, size_t in_comp, int in_line, int in_row, int in_fix, double2* out, size_t out_comp,
            int n_line, int n, unsigned odd_mask, const double2* twg) {
    using B = DhatBlock<RE, RO>;
    constexpr int W = B::W;
    extern __shared__ __align__(16) double2 dsm[];
    double2 *tw = dsm, *A = dsm + B::ROWS;
    dhat_twiddles<RE, RO>(tw, twg);
    const int l0 = blockIdx.x * W;
    const bool odd = odd_mask >> (blockIdx.z % 6) & 1;
    const double2* src = in + blockIdx.z * in_comp;
    dhat_1<RE, RO>(A, W, W, n, odd, threadIdx.x, blockDim.x, [&](int w, int i) {
        const int l = l0 + w;
        return l < n_line ? src[(size_t)(l / in_row) * in_fix + l % in_row + (size_t)i * in_line] : make_double2(0.0, 0.0);
    });
    __syncthreads();
    double2* dst = out + blockIdx.z * out_comp + l0;
    dhat_2<RE, RO>(A, W, W, odd, tw, threadIdx.x, blockDim.x, [&](int w, int k, double2 v) {
        if (l0 + w < n_line) dst[(size_t)k * n_line + w] = v;
    });
}

// The x axis: lines contiguous in in[slot * 6 + comp][ky][kz][x], staged through
// shared memory; outputs D-hat [slot][comp][ky][kx][kz] in FP64 and FP32 and, for
// the register x pass, [slot][ky][kz][comp][kx] in FP32.
template <int RE, int RO>
__global__ void __launch_bounds__((DhatBlock<RE, RO>::THREADS), 1)
k_dhat_x(LatticeDev L, const double2* in, double2* Dr64, float2* Dr32, float2* Dx) {
    using B = DhatBlock<RE, RO>;
    constexpr int W = B::W, Hx = RE * RO / 2 + 1;
    extern __shared__ __align__(16) double2 dsm[];
    double2 *tw = dsm, *A = dsm + B::ROWS, *X = A + B::ROWS * W;       // X[W][Nx + 1], then the FP32 rows R[Hx][W + 1]
    float2* R = reinterpret_cast<float2*>(X);
    dhat_twiddles<RE, RO>(tw, L.tw64x);
    const int n_line = L.Hy * L.Hz, l0 = blockIdx.x * W, nw = min(W, n_line - l0), Nx = L.Nx;
    const int sc = blockIdx.z, slot = sc / 6, c = sc % 6;
    const bool odd = c == 1 || c == 2;
    const double2* src = in + ((size_t)sc * n_line + l0) * Nx;
    for (int t = threadIdx.x; t < nw * Nx; t += blockDim.x) {
        const int w = t / Nx;
        X[t + w] = src[t];
    }
    __syncthreads();
    dhat_1<RE, RO>(A, W, W, Nx, odd, threadIdx.x, blockDim.x, [&](int w, int i) {
        return w < nw ? X[w * (Nx + 1) + i] : make_double2(0.0, 0.0);
    });
    __syncthreads();
    dhat_2<RE, RO>(A, W, W, odd, tw, threadIdx.x, blockDim.x, [&](int w, int k, double2 v) {
        if (w >= nw) return;
        const int l = l0 + w, ky = l / L.Hz;
        const size_t o = ((size_t)sc * L.Hy + ky) * Hx * L.Hz + (size_t)k * L.Hz + (l - ky * L.Hz);
        const float2 f = to_f(v);
        Dr64[o] = v;
        Dr32[o] = f;
        R[k * (W + 1) + w] = f;
    });
    if (!Dx) return;
    __syncthreads();
    for (int t = threadIdx.x; t < nw * Hx; t += blockDim.x) {
        const int w = t / Hx, k = t - w * Hx;
        Dx[(((size_t)slot * n_line + l0 + w) * 6 + c) * Hx + k] = R[k * (W + 1) + w];
    }
}
template <int RE, int RO> static size_t dhat_x_smem(int Nx) {
    using B = DhatBlock<RE, RO>;
    return B::LINE_SMEM + std::max((size_t)B::W * (Nx + 1) * 16, (size_t)(RE * RO / 2 + 1) * (B::W + 1) * 8);
}

// Two scratch arrays per slot: the octant (then the y pass's output) and the z
// pass's output.
static size_t dhat_a(const LatticeDev& L) { return (size_t)6 * L.Nx * std::max(L.Ny * L.Nz, L.Hy * L.Hz); }
static size_t dhat_b(const LatticeDev& L) { return (size_t)6 * L.Nx * L.Ny * L.Hz; }
size_t dhat_scratch_bytes(const LatticeDev& L) { return (dhat_a(L) + dhat_b(L)) * sizeof(double2); }

static void axis(const Plan2& p, int slots, cudaStream_t st, const double2* in, size_t in_comp, int in_line, int in_row,
                 int in_fix, double2* out, size_t out_comp, int n_line, int n, unsigned odd_mask, const double2* tw) {
    count_launch();
    switch (p.L) {
#define AX(RE, RO)                                                                                                    \
    case RE * RO: {                                                                                                   \
        using B = DhatBlock<RE, RO>;                                                                                  \
        k_dhat_axis<RE, RO><<<dim3((n_line + B::W - 1) / B::W, 1, slots * 6), B::THREADS, B::LINE_SMEM, st>>>(        \
            in, in_comp, in_line, in_row, in_fix, out, out_comp, n_line, n, odd_mask, tw);                            \
        break;                                                                                                        \
    }
        EELS_PLANS(AX)
#undef AX
        default: break;
    }
}

void prepare_dhat_kernels() {
#define AX(RE, RO)                                                                                                    \
    cudaFuncSetAttribute(k_dhat_axis<RE, RO>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);              \
    cudaFuncSetAttribute(k_dhat_x<RE, RO>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    EELS_PLANS(AX)
#undef AX
}

void launch_dhat_build(const LatticeDev& L, int n_slot, const double2* kappa, double2* G, double2* Dr64, float2* Dr32,
                       cudaStream_t st, float2* Dx32) {
    double2 *A = G, *B = G + (size_t)n_slot * dhat_a(L);
    const int n = L.Nx * L.Ny * L.Nz, plane = L.Nx * L.Ny, rows = L.Hz * L.Nx, lines = L.Hy * L.Hz;
    count_launch();
    k_green<<<dim3((n + 127) / 128, n_slot), 128, 0, st>>>(L, kappa, A);
    // z: [z][y x] -> [kz][y x]
    axis(L.qz, n_slot, st, A, (size_t)n, plane, plane, 0, B, (size_t)L.Hz * plane, plane, L.Nz, 1u << 2 | 1u << 4, L.tw64z);
    // y: [kz][y][x] -> [ky][kz x]
    axis(L.qy, n_slot, st, B, (size_t)L.Hz * plane, L.Nx, L.Nx, plane, A, (size_t)L.Hy * rows, rows, L.Ny,
         1u << 1 | 1u << 4, L.tw64y);
    count_launch();
    switch (L.Mx) {
#define AX(RE, RO)                                                                                                    \
    case RE * RO: {                                                                                                   \
        using P = DhatBlock<RE, RO>;                                                                                  \
        k_dhat_x<RE, RO><<<dim3((lines + P::W - 1) / P::W, 1, n_slot * 6), P::THREADS, dhat_x_smem<RE, RO>(L.Nx), st>>>( \
            L, A, Dr64, Dr32, Dx32);                                                                                  \
        break;                                                                                                        \
    }
        EELS_PLANS(AX)
#undef AX
        default: break;
    }
}

}  // namespace eels
