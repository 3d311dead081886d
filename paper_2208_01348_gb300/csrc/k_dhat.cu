// D-hat build: the transform of the six components of the Green's tensor
// (Eq. 5, or the cell-integrated tensor for near offsets) on the padded
// lattice, for n_slot wavenumbers kappa = k d, FP64.
//
//   G~' = exp(i kappa R)/R [kappa^2 (I - RR) - (1 - i kappa R)/R^2 (I - 3 RR)]   (Eq. 5)
//
// The diagonal components are even in each of x, y, z and xy, xz, yz are odd in
// the two axes they name, so only the octant of non-negative offsets is
// evaluated, and each axis is transformed from its non-negative half
// (dhat.cuh) to the frequencies 0 <= k <= M/2 that are kept: 3 N^2 half-filled
// lines per component in place of 12 N^2 full ones, N^3 exponentials in place
// of 8 N^3.  The FP64 pipe bounds it (the axis passes run at its measured rate;
// the arrays of one energy of 64^3 cells are 25 MB): 0.46 ms per energy of 64^3
// cells, against 2.2 ms for the padded lattice.  The last axis writes D-hat in
// the layouts that the x passes read.
#include <algorithm>

#include "dhat.cuh"
#include "kernels.h"

namespace eels {

// G[slot][comp][z][y][x] over the octant, x fastest, the samples at offset 0
// of an even axis halved.
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
    // halve offset 0 of every axis (odd components vanish there)
    const double f = (x ? 1.0 : 0.5) * (y ? 1.0 : 0.5) * (z ? 1.0 : 0.5);
    double2* out = G + (size_t)slot * 6 * n + idx;
    for (int c = 0; c < 6; ++c) out[(size_t)c * n] = f * g[c];
}

constexpr int DHAT_W = 8;        // lines per block
constexpr int DHAT_THREADS = 64;

// One axis: lines of n entries (stride in_line) at (fixed index blockIdx.y,
// lane x), to the entries k <= L/2 of their transforms.
template <int RE, int RO>
__global__ void __launch_bounds__(DHAT_THREADS)
k_dhat_axis(const double2* in, size_t in_comp, int in_line, int in_fix, double2* out, size_t out_comp, int out_line,
            int out_fix, int n, int n_lane, unsigned odd_mask, const double2* twg) {
    constexpr int LEN = RE * RO, W = DHAT_W;
    __shared__ double2 tw[LEN], A[LEN * W];
    for (int t = threadIdx.x; t < LEN; t += DHAT_THREADS) tw[t] = twg[(t / RE) * (t % RE)];
    const int x0 = blockIdx.x * W;
    const bool odd = odd_mask >> (blockIdx.z % 6) & 1;
    const double2* src = in + blockIdx.z * in_comp + (size_t)blockIdx.y * in_fix + x0;
    dhat_1<RE, RO, false>(A, W, W, n, threadIdx.x, DHAT_THREADS, [&](int w, int i) {
        return x0 + w < n_lane ? src[(size_t)i * in_line + w] : make_double2(0.0, 0.0);
    });
    __syncthreads();
    dhat_2<RE, RO>(A, W, W, tw, threadIdx.x, DHAT_THREADS);
    __syncthreads();
    double2* dst = out + blockIdx.z * out_comp + (size_t)blockIdx.y * out_fix + x0;
    for (int t = threadIdx.x; t < (LEN / 2 + 1) * W; t += DHAT_THREADS) {
        const int w = t % W, k = t / W;
        if (x0 + w < n_lane) dst[(size_t)k * out_line + w] = dhat_fold(A, W, LEN, k, w, odd);
    }
}

// The x axis: lines contiguous in in[slot * 6 + comp][ky][kz][x]; outputs D-hat
// [slot][comp][ky][kx][kz] in FP64 and FP32 and, for the register x pass,
// [slot][ky][kz][comp][kx] in FP32.
template <int RE, int RO>
__global__ void __launch_bounds__(DHAT_THREADS)
k_dhat_x(LatticeDev L, const double2* in, double2* Dr64, float2* Dr32, float2* Dx) {
    constexpr int LEN = RE * RO, W = DHAT_W, ES = W + 1;
    __shared__ double2 tw[LEN], A[LEN * ES];
    for (int t = threadIdx.x; t < LEN; t += DHAT_THREADS) tw[t] = L.tw64x[(t / RE) * (t % RE)];
    const int kz0 = blockIdx.x * W, ky = blockIdx.y, sc = blockIdx.z, slot = sc / 6, c = sc % 6;
    const int nw = min(W, L.Hz - kz0), Hx = LEN / 2 + 1;
    const bool odd = c == 1 || c == 2;
    const double2* src = in + (((size_t)sc * L.Hy + ky) * L.Hz + kz0) * L.Nx;
    dhat_1<RE, RO, true>(A, ES, W, L.Nx, threadIdx.x, DHAT_THREADS, [&](int w, int i) {
        return w < nw ? src[(size_t)w * L.Nx + i] : make_double2(0.0, 0.0);
    });
    __syncthreads();
    dhat_2<RE, RO>(A, ES, W, tw, threadIdx.x, DHAT_THREADS);
    __syncthreads();
    const size_t base = (((size_t)sc * L.Hy + ky) * Hx) * L.Hz + kz0;
    for (int t = threadIdx.x; t < Hx * W; t += DHAT_THREADS) {
        const int w = t % W, k = t / W;
        if (w >= nw) continue;
        const double2 v = dhat_fold(A, ES, LEN, k, w, odd);
        const float2 f = to_f(v);
        Dr64[base + (size_t)k * L.Hz + w] = v;
        Dr32[base + (size_t)k * L.Hz + w] = f;
        // rows k and LEN - k are read for this frequency alone: row k keeps the rounded value
        reinterpret_cast<float2*>(A + k * ES + w)[0] = f;
    }
    if (!Dx) return;
    __syncthreads();
    for (int t = threadIdx.x; t < nw * Hx; t += DHAT_THREADS) {
        const int k = t % Hx, w = t / Hx;
        Dx[((((size_t)slot * L.Hy + ky) * L.Hz + kz0 + w) * 6 + c) * Hx + k] = *reinterpret_cast<const float2*>(A + k * ES + w);
    }
}

// Two scratch arrays per slot: the octant (then the y pass's output) and the z
// pass's output.
static size_t dhat_a(const LatticeDev& L) { return (size_t)6 * L.Nx * std::max(L.Ny * L.Nz, L.Hy * L.Hz); }
static size_t dhat_b(const LatticeDev& L) { return (size_t)6 * L.Nx * L.Ny * L.Hz; }
size_t dhat_scratch_bytes(const LatticeDev& L) { return (dhat_a(L) + dhat_b(L)) * sizeof(double2); }

static void axis(const Plan2& p, dim3 grid, cudaStream_t st, const double2* in, size_t in_comp, int in_line, int in_fix,
                 double2* out, size_t out_comp, int out_line, int out_fix, int n, int n_lane, unsigned odd_mask,
                 const double2* tw) {
    count_launch();
    switch (p.L) {
#define AX(RE, RO)                                                                                                 \
    case RE * RO:                                                                                                  \
        k_dhat_axis<RE, RO><<<grid, DHAT_THREADS, 0, st>>>(in, in_comp, in_line, in_fix, out, out_comp, out_line,  \
                                                           out_fix, n, n_lane, odd_mask, tw);                      \
        break;
        EELS_PLANS(AX)
#undef AX
        default: break;
    }
}

void launch_dhat_build(const LatticeDev& L, int n_slot, const double2* kappa, double2* G, double2* Dr64, float2* Dr32,
                       cudaStream_t st, float2* Dx32) {
    double2 *A = G, *B = G + (size_t)n_slot * dhat_a(L);
    const int n = L.Nx * L.Ny * L.Nz, tiles = (L.Nx + DHAT_W - 1) / DHAT_W, plane = L.Nx * L.Ny;
    count_launch();
    k_green<<<dim3((n + 127) / 128, n_slot), 128, 0, st>>>(L, kappa, A);
    // z: [z][y][x] -> [kz][y][x]
    axis(L.qz, dim3(tiles, L.Ny, n_slot * 6), st, A, (size_t)n, plane, L.Nx, B, (size_t)L.Hz * plane, plane, L.Nx, L.Nz,
         L.Nx, 1u << 2 | 1u << 4, L.tw64z);
    // y: [kz][y][x] -> [ky][kz][x]
    axis(L.qy, dim3(tiles, L.Hz, n_slot * 6), st, B, (size_t)L.Hz * plane, L.Nx, plane, A, (size_t)L.Hy * L.Hz * L.Nx,
         L.Hz * L.Nx, L.Nx, L.Ny, L.Nx, 1u << 1 | 1u << 4, L.tw64y);
    const dim3 grid((L.Hz + DHAT_W - 1) / DHAT_W, L.Hy, n_slot * 6);
    count_launch();
    switch (L.Mx) {
#define AX(RE, RO) case RE * RO: k_dhat_x<RE, RO><<<grid, DHAT_THREADS, 0, st>>>(L, A, Dr64, Dr32, Dx32); break;
        EELS_PLANS(AX)
#undef AX
        default: break;
    }
}

}  // namespace eels
