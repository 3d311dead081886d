// FFT kernels of the DDA matrix-vector product.
//
// The interaction sum conv(u)_i = sum_{j != i} G~'(r_i - r_j) u_j over a
// cubic lattice is a 3-D convolution; embedding it in a circulant of
// extents M >= 2N - 1 per axis turns it into  IFFT( D-hat . FFT(u) ), where
// D-hat is the FFT of the six symmetric components of G~' on the padded
// lattice (separation (i - M) for the upper indices, zero at R = 0 and at
// indices no separation reaches).  The input u is non-zero only on the
// first Nx x Ny x Nz corner and only that corner of the output is needed, so
// a matvec is three passes over one scratch array U[s][c][y][x][z] (z
// fastest): a slab pass (gather, y and z transforms of one x-slab), the x pass
// (My*Mz lines: x transform, D-hat product, inverse x transform) and a slab
// pass back (inverse z and y transforms, combination with x, scatter).  This
// file holds the slab passes of 64 x 64 and 128 x 128 points in FP32 and the
// launch of a matvec; k_dhat.cu the D-hat build, k_slab.cuh and k_xline.cuh the passes of
// any length, k_xreg.cu the x pass of 64 and 128 points in FP32.
//
// D-hat is stored on the octant 0 <= k <= M/2 only (6 (M/2+1)^3 values):
// the diagonal components are even in each k and xy, xz, yz are odd in the
// two axes they name, so D(M - k) = +-D(k).
#include <algorithm>
#include <cstdio>

#include "fft_warp.cuh"
#include "kernels.h"

namespace eels {

template <typename Rl> __device__ __forceinline__ const cx<Rl>* tw_of(const LatticeDev& L, int axis);
template <> __device__ __forceinline__ const double2* tw_of<double>(const LatticeDev& L, int axis) {
    return axis == 0 ? L.tw64x : (axis == 1 ? L.tw64y : L.tw64z);
}
template <> __device__ __forceinline__ const float2* tw_of<float>(const LatticeDev& L, int axis) {
    return axis == 0 ? L.tw32x : (axis == 1 ? L.tw32y : L.tw32z);
}

// ---------------------------------------------------------------------------
// Fused slab passes for My = Mz = L = 64 or 128 in FP32, register resident.
//
// A warp transforms 4 lines at once (fft_warp.cuh): lane = q + 4p holds, for
// its line q, the elements p + 8r (r < R = L/8) of the line, and the
// transform leaves element j + 8m in register m of lane j.  Between the y and
// the z transforms the slab S[L][Nz] sits in shared memory (row stride
// 4 mod 16: the 4 x 4 (line, lane) patterns of every access hit distinct
// banks); the block synchronises once per pass.  Every loop over line quads
// loads the next quad's inputs before transforming the current one, so the
// global loads of one quad overlap the arithmetic of the previous one.
// HALF: Ny = Nz = L/2 (the lattice fills exactly half of every line): the
// zero padding and the discarded outputs are known at compile time.  FAST:
// every column's occupied cells are contiguous in z, so a dipole's index is
// the column's base plus iz (no cell-map load).
// ---------------------------------------------------------------------------
// 64 points: blocks of 4 warps, seven on an SM, so that the block barriers of
// one slab are filled by more others (four blocks of 8 warps: 773 -> 733 us a
// matvec of 200 systems of 32^3 cells, although 28 warps are resident in place
// of 32); the larger slab of 128 points leaves room for two blocks of 8 warps.
template <int R> struct SlabR {
    static constexpr int L = 8 * R;
    static constexpr int SLS = R == 8 ? 36 : 68;           // slab row stride
    static constexpr int TILE = R == 8 ? R64_TILE : R128_TILE;
    static constexpr int THREADS = R == 8 ? 128 : 256, BLOCKS = R == 8 ? 7 : 2;     // per SM
};

template <int R> struct SlabRSmem {
    float2 tw2[(R - 1) * 8];                     // exp(-2 pi i p k / L) at [k - 1][p]: conflict-free per k
    float2 cf[EELS_MAX_MAT], dg[EELS_MAX_MAT];   // this system's per-material coefficients
    float2 S[SlabR<R>::L * SlabR<R>::SLS];
    alignas(16) float2 tile[SlabR<R>::THREADS / 32][SlabR<R>::TILE];
    int4 ci[SlabR<R>::L / 2];                    // this slab's column table (contiguous columns)
};

// Persistent forward slab pass: the grid holds as many blocks as fit on the
// GPU at once, and each block walks the (system, component, slab) items with
// a stride of the grid size.  For single-material lattices with contiguous
// columns, a block loads the first column quad of its next item while it runs
// the z transforms of the current one, so the gather's latency is hidden
// behind arithmetic instead of opening every item.
template <int R, bool HALF, bool FAST>
__global__ void __launch_bounds__(SlabR<R>::THREADS, SlabR<R>::BLOCKS) k_slab_fwd_r(LatticeDev L, MatvecArgs<float> a) {
    using C = float2;
    using P = SlabR<R>;
    constexpr int LEN = P::L, SLS = P::SLS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SlabRSmem<R>& sm = *reinterpret_cast<SlabRSmem<R>*>(smem_raw);
    const int Ny = L.Ny, Nz = L.Nz, Nx = L.Nx, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = lane & 3,
              p = lane >> 2;
    const int nwarp = blockDim.x >> 5;
    const int n_items = a.S * 3 * Nx;
    const bool one_mat = L.nmat == 1;
    const bool prefetch = FAST && one_mat;
    const float2* twg = tw_of<float>(L, 1);          // My = Mz: the y and z tables coincide
    for (int t = threadIdx.x; t < (R - 1) * 8; t += blockDim.x) sm.tw2[t] = twg[(t & 7) * ((t >> 3) + 1)];
    float2* tile = sm.tile[warp];
    auto tw = [&](int k) { return sm.tw2[(k - 1) * 8 + p]; };
    const C zero = make_float2(0.f, 0.f);
    const int stride = nwarp * 4;
    auto active = [&](int item) { return !a.active || a.active[item / (3 * Nx)]; };
    auto next_item = [&](int item) {
        for (item += gridDim.x; item < n_items && !active(item); item += gridDim.x) {}
        return item;
    };
    // raw x values of the first column quad (iz0 = 4 warp) of an item, dipoles
    // addressed through the column table in global memory
    auto gather_raw = [&](int item, C (&v)[R]) {
        const int s = item / (3 * Nx), c = (item / Nx) % 3, ix = item % Nx, iz = warp * 4 + q;
        const C* xs = a.x + ((size_t)s * 3 + c) * L.N;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int y = p + 8 * r;
            v[r] = zero;
            if ((HALF ? r < R / 2 : y < Ny) && iz < Nz) {
                const int dip = col_dip(L.colinfo[(size_t)ix * Ny + y], iz);
                if (dip >= 0) v[r] = xs[dip];
            }
        }
    };
    C pf[R];
    int item = blockIdx.x;
    if (item < n_items && !active(item)) item = next_item(item);
    if (prefetch && item < n_items && warp * 4 < Nz) gather_raw(item, pf);
    for (; item < n_items;) {
        const int s = item / (3 * Nx), c = (item / Nx) % 3, ix = item % Nx;
        if (threadIdx.x < EELS_MAX_MAT) sm.cf[threadIdx.x] = to_f(a.coef[(size_t)s * EELS_MAX_MAT + threadIdx.x]);
        if (FAST)
            for (int t = threadIdx.x; t < Ny; t += blockDim.x) sm.ci[t] = L.colinfo[(size_t)ix * Ny + t];
        __syncthreads();
        const C* xs = a.x + ((size_t)s * 3 + c) * L.N;
        const int* cm = L.cellmap + (size_t)ix * Ny * Nz;
        // y transforms of the Nz columns, 4 per warp: gathered from x, into S
        auto gather = [&](int iz0, C (&v)[R]) {
            const int iz = iz0 + q;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int y = p + 8 * r;
                v[r] = zero;
                if ((HALF ? r < R / 2 : y < Ny) && iz < Nz) {
                    const int dip = FAST ? col_dip(sm.ci[y], iz) : cm[y * Nz + iz];
                    if (dip >= 0) v[r] = xs[dip] * (one_mat ? sm.cf[0] : sm.cf[L.mat[dip]]);
                }
            }
        };
        C vn[R];
        if (warp * 4 < Nz) {
            if (prefetch) {
#pragma unroll
                for (int r = 0; r < R; ++r) vn[r] = pf[r] * sm.cf[0];
            } else {
                gather(warp * 4, vn);
            }
        }
        for (int iz0 = warp * 4; iz0 < Nz; iz0 += stride) {
            C v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = vn[r];
            if (iz0 + stride < Nz) gather(iz0 + stride, vn);
            fft_warp_t<R, false, HALF>(v, tile, q, p, tw);
            const int iz = iz0 + q;
            if (iz < Nz) {
#pragma unroll
                for (int m = 0; m < R; ++m) sm.S[(p + 8 * m) * SLS + iz] = v[m];
            }
        }
        __syncthreads();
        const int nxt = next_item(item);
        if (prefetch && nxt < n_items && warp * 4 < Nz) gather_raw(nxt, pf);
        // z transforms of the LEN rows, 4 per warp: from S, written to U
        C* U = a.U + (((size_t)s * 3 + c) * LEN * L.Nx + ix) * LEN;
        const size_t row = (size_t)L.Nx * LEN;
        for (int ky0 = warp * 4; ky0 < LEN; ky0 += stride) {
            const int ky = ky0 + q;
            C v[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int z = p + 8 * r;
                v[r] = (HALF ? r < R / 2 : z < Nz) ? sm.S[ky * SLS + z] : zero;
            }
            fft_warp_t<R, false, HALF>(v, tile, q, p, tw);
#pragma unroll
            for (int m = 0; m < R; ++m) U[(size_t)ky * row + p + 8 * m] = v[m];
        }
        item = nxt;
        __syncthreads();                              // S, ci and cf are refilled for the next item
    }
}

template <int R, bool HALF, bool FAST>
__global__ void __launch_bounds__(SlabR<R>::THREADS, SlabR<R>::BLOCKS) k_slab_inv_r(LatticeDev L, MatvecArgs<float> a, float invM) {
    using C = float2;
    using P = SlabR<R>;
    constexpr int LEN = P::L, SLS = P::SLS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SlabRSmem<R>& sm = *reinterpret_cast<SlabRSmem<R>*>(smem_raw);
    __shared__ float red[2 * SlabR<R>::THREADS / 32];
    const int ix = blockIdx.x, b = blockIdx.y, s = b / 3, c = b % 3;
    if (a.active && !a.active[s]) return;
    const int Ny = L.Ny, Nz = L.Nz, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, q = lane & 3, p = lane >> 2;
    const int nwarp = blockDim.x >> 5;
    const float2* twg = tw_of<float>(L, 2);
    for (int t = threadIdx.x; t < (R - 1) * 8; t += blockDim.x) sm.tw2[t] = twg[(t & 7) * ((t >> 3) + 1)];
    if (threadIdx.x < EELS_MAX_MAT) {
        sm.cf[threadIdx.x] = to_f(a.coef[(size_t)s * EELS_MAX_MAT + threadIdx.x]);
        sm.dg[threadIdx.x] = to_f(a.diag[(size_t)s * EELS_MAX_MAT + threadIdx.x]);
    }
    if (FAST)
        for (int t = threadIdx.x; t < Ny; t += blockDim.x) sm.ci[t] = L.colinfo[(size_t)ix * Ny + t];
    const bool one_mat = L.nmat == 1;
    __syncthreads();
    float2* tile = sm.tile[warp];
    auto tw = [&](int k) { return sm.tw2[(k - 1) * 8 + p]; };
    const int stride = nwarp * 4;
    // inverse z transforms of the LEN rows of U, first Nz outputs into S
    const C* U = a.U + (((size_t)s * 3 + c) * LEN * L.Nx + ix) * LEN;
    const size_t row = (size_t)L.Nx * LEN;
    C vn[R];
#pragma unroll
    for (int r = 0; r < R; ++r) vn[r] = U[(size_t)(warp * 4 + q) * row + p + 8 * r];
    for (int ky0 = warp * 4; ky0 < LEN; ky0 += stride) {
        const int ky = ky0 + q;
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = vn[r];
        if (ky0 + stride < LEN) {
#pragma unroll
            for (int r = 0; r < R; ++r) vn[r] = U[(size_t)(ky + stride) * row + p + 8 * r];
        }
        fft_warp_t<R, true, false>(v, tile, q, p, tw);
#pragma unroll
        for (int m = 0; m < R; ++m) {
            const int z = p + 8 * m;
            if (HALF ? m < R / 2 : z < Nz) sm.S[ky * SLS + z] = v[m];
        }
    }
    __syncthreads();
    // inverse y transforms of the Nz columns, first Ny outputs combined with x
    // and scattered; each lane loads its x values before its transform
    const C* xs = a.x + ((size_t)s * 3 + c) * L.N;
    C* ys = a.y + ((size_t)s * 3 + c) * L.N;
    const int* cm = L.cellmap + (size_t)ix * Ny * Nz;
    constexpr int RO = HALF ? R / 2 : R;             // registers that can hold lattice rows
    float dot0 = 0.f, dot1 = 0.f;
    for (int iz0 = warp * 4; iz0 < Nz; iz0 += stride) {
        const int iz = iz0 + q;
        int dip[RO];
        C xv[RO];
#pragma unroll
        for (int m = 0; m < RO; ++m) {
            const int y = p + 8 * m;
            dip[m] = -1;
            if (iz < Nz && (HALF || y < Ny)) dip[m] = FAST ? col_dip(sm.ci[y], iz) : cm[y * Nz + iz];
            xv[m] = dip[m] >= 0 ? xs[dip[m]] : make_float2(0.f, 0.f);
        }
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = iz < Nz ? sm.S[(p + 8 * r) * SLS + iz] : make_float2(0.f, 0.f);
        fft_warp_t<R, true, false>(v, tile, q, p, tw);
#pragma unroll
        for (int m = 0; m < RO; ++m) {
            if (dip[m] < 0) continue;
            const int mt = one_mat ? 0 : L.mat[dip[m]];
            const C yv = sm.dg[mt] * xv[m] - sm.cf[mt] * (invM * v[m]);
            ys[dip[m]] = yv;
            dot0 += xv[m].x * yv.x - xv[m].y * yv.y;
            dot1 += xv[m].x * yv.y + xv[m].y * yv.x;
        }
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
            double* pp = a.dot_part + (((size_t)s * 3 + c) * L.Nx + ix) * 4;
            pp[0] = s0; pp[1] = s1; pp[2] = 0.0; pp[3] = 0.0;
        }
    }
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
template <typename K> static void allow_smem(K kernel) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
    // these kernels keep their working tiles in shared memory: give it the whole carveout
    cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
}

// Register-resident slab kernels: FP32 with 64- or 128-point y and z transforms.
int sm_count() {
    static int cache[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return 132; }
    if (!cache[dev]) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
            cudaGetLastError();
            n = 132;
        }
        cache[dev] = n;
    }
    return cache[dev];
}

template <int R, bool HALF, bool FAST>
static void slab_r_launch(const LatticeDev& L, const MatvecArgs<float>& a, bool inv, cudaStream_t st) {
    const size_t sm = sizeof(SlabRSmem<R>);
    const float invM = (float)(1.0 / ((double)L.Mx * L.My * L.Mz));
    if (!inv) {
        // persistent: the blocks resident at once
        const int items = a.S * 3 * L.Nx;
        const int blocks = std::min(items, sm_count() * SlabR<R>::BLOCKS);
        k_slab_fwd_r<R, HALF, FAST><<<blocks, SlabR<R>::THREADS, sm, st>>>(L, a);
    } else {
        k_slab_inv_r<R, HALF, FAST><<<dim3(L.Nx, a.S * 3), SlabR<R>::THREADS, sm, st>>>(L, a, invM);
    }
}

template <int R>
static void slab_r_any(const LatticeDev& L, const MatvecArgs<float>& a, bool inv, cudaStream_t st) {
    const bool half = 2 * L.Ny == 8 * R && 2 * L.Nz == 8 * R;
    count_launch();
    if (half && L.contig) slab_r_launch<R, true, true>(L, a, inv, st);
    else if (half) slab_r_launch<R, true, false>(L, a, inv, st);
    else if (L.contig) slab_r_launch<R, false, true>(L, a, inv, st);
    else slab_r_launch<R, false, false>(L, a, inv, st);
}

template <typename Rl> static bool slab_reg_launch(const LatticeDev& L, const MatvecArgs<Rl>& a, bool inv, cudaStream_t st);
template <> bool slab_reg_launch<double>(const LatticeDev&, const MatvecArgs<double>&, bool, cudaStream_t) { return false; }
template <> bool slab_reg_launch<float>(const LatticeDev& L, const MatvecArgs<float>& a, bool inv, cudaStream_t st) {
    if (L.My == 64 && L.Mz == 64) { slab_r_any<8>(L, a, inv, st); return true; }
    if (L.My == 128 && L.Mz == 128) { slab_r_any<16>(L, a, inv, st); return true; }
    return false;
}

template <typename Rl> static void slab_launch_any(const LatticeDev& L, const MatvecArgs<Rl>& a, bool inv,
                                                   cudaStream_t st) {
    if (slab_reg_launch<Rl>(L, a, inv, st)) return;
    launch_slab<Rl>(L, a, inv, st);
}

// Tile width of the x pass before the autotuner has timed it (eels_matvec_dev and
// eels_krylov_solve_dev without an earlier eels_solve): the widest of 32, 16 and 8
// lines whose block keeps to 56 KB of shared memory in FP32 and 28 KB in FP64.  Most
// widths time alike (8 systems of 32^3 cells in FP64 969, 969 and 974 us with 8, 16 and
// 32 lines), but the wide ones lose where few blocks of them fit: 16 of 24^3 in FP64
// 982, 981 and 1240, 2 of 64^3 2117, 2180 and 2167, and 4 of 79^3 in FP32 515 us with 8
// lines and 608 with 16.
template <typename Rl> static int pick_xpass_w(const LatticeDev& L) {
    for (int W : {32, 16})
        if (xline_smem<Rl>(L, W) <= (sizeof(Rl) == 4 ? 56 : 28) * 1024) return W;
    return 8;
}

template <typename Rl> static int tuned_w(const LatticeDev& L) { return sizeof(Rl) == 4 ? L.xw32 : L.xw64; }

template <typename Rl>
int autotune_xpass(const LatticeDev& L, const MatvecArgs<Rl>& a, cudaStream_t st) {
    int best = pick_xpass_w<Rl>(L);
    float best_ms = 0.f;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return best;
    if (cudaEventCreate(&e1) != cudaSuccess) { cudaEventDestroy(e0); return best; }
    bool first = true;
    for (int w : {8, 16, 32}) {
        if (!xline_fits<Rl>(L, w)) continue;
        launch_xline<Rl>(L, a, w, st);              // warm-up
        cudaEventRecord(e0, st);
        for (int r = 0; r < 3; ++r) launch_xline<Rl>(L, a, w, st);
        cudaEventRecord(e1, st);
        float ms = 0.f;
        if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) break;
        if (first || ms < best_ms) { best = w; best_ms = ms; first = false; }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return best;
}
template int autotune_xpass<float>(const LatticeDev&, const MatvecArgs<float>&, cudaStream_t);
template int autotune_xpass<double>(const LatticeDev&, const MatvecArgs<double>&, cudaStream_t);

template <typename Rl> static void xpass_any(const LatticeDev& L, const MatvecArgs<Rl>& a, cudaStream_t st) {
    if constexpr (sizeof(Rl) == 4) {
        if (launch_xpass_reg(L, a, st)) return;
    }
    launch_xline<Rl>(L, a, tuned_w<Rl>(L) ? tuned_w<Rl>(L) : pick_xpass_w<Rl>(L), st);
}

template <typename Rl>
void launch_matvec(const LatticeDev& L, const MatvecArgs<Rl>& a, cudaStream_t st) {
    // slab (gather, y, z) -> x * D-hat * x -> slab (z, y, scatter)
    MatvecArgs<Rl> b = a;
    b.dep = !a.no_dep && matvec_dep(L, a.S, sizeof(Rl) == 8);
    slab_launch_any<Rl>(L, b, false, st);
    xpass_any<Rl>(L, b, st);
    slab_launch_any<Rl>(L, b, true, st);
}

void prepare_dhat_kernels();
void prepare_far_kernels();
void prepare_xreg_kernels();

void prepare_kernels() {
    allow_smem(k_slab_fwd_r<8, true, true>);
    allow_smem(k_slab_fwd_r<8, true, false>);
    allow_smem(k_slab_fwd_r<8, false, true>);
    allow_smem(k_slab_fwd_r<8, false, false>);
    allow_smem(k_slab_inv_r<8, true, true>);
    allow_smem(k_slab_inv_r<8, true, false>);
    allow_smem(k_slab_inv_r<8, false, true>);
    allow_smem(k_slab_inv_r<8, false, false>);
    allow_smem(k_slab_fwd_r<16, true, true>);
    allow_smem(k_slab_fwd_r<16, true, false>);
    allow_smem(k_slab_fwd_r<16, false, true>);
    allow_smem(k_slab_fwd_r<16, false, false>);
    allow_smem(k_slab_inv_r<16, true, true>);
    allow_smem(k_slab_inv_r<16, true, false>);
    allow_smem(k_slab_inv_r<16, false, true>);
    allow_smem(k_slab_inv_r<16, false, false>);
    prepare_dhat_kernels();
    prepare_far_kernels();
    prepare_slab_kernels<float>();
    prepare_slab_kernels<double>();
    prepare_xline_kernels<float>();
    prepare_xline_kernels<double>();
    prepare_xreg_kernels();
}

template void launch_matvec<float>(const LatticeDev&, const MatvecArgs<float>&, cudaStream_t);
template void launch_matvec<double>(const LatticeDev&, const MatvecArgs<double>&, cudaStream_t);

static bool slab_reg(const LatticeDev& L) { return (L.My == 64 && L.Mz == 64) || (L.My == 128 && L.Mz == 128); }
bool matvec_dep(const LatticeDev& L, int S, bool fp64) {
    if (!fp64 && (slab_reg(L) || xpass_reg_supported(L))) return false;
    const long long slabs = 3LL * L.Nx * S * (fp64 ? L.s64.CL : L.s32.CL), lines = (L.Mz + 3) / 4 * (long long)L.My * S;
    return std::max(slabs, lines) <= sm_count();
}
int matvec_dot_parts(const LatticeDev& L, bool fp64) {
    return 3 * L.Nx * (fp64 ? L.s64.CL : slab_reg(L) ? 1 : L.s32.CL);
}

}  // namespace eels
