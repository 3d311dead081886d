// Internal launch interface between the host engine and the CUDA kernels.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <array>
#include <utility>
#include <vector>

#include "common.cuh"
#include "dft.cuh"

namespace eels {

// Process-wide count of kernels this library has launched (graph replays
// add their kernel nodes; launches recorded during a stream capture are not
// counted until the graph runs).
extern std::atomic<long long> g_kernel_launches;
extern thread_local bool g_capturing;
inline void count_launch(int n = 1) {
    if (!g_capturing) g_kernel_launches += n;
}

// Multiprocessors of the current device (queried once per device).
int sm_count();

// Launch of a kernel in clusters of cl blocks along x; dep: it begins with
// dep_wait(1) and may start while the kernel before it drains.
template <typename... P, typename... A>
void launch_dep(int dep, void (*kernel)(P...), dim3 grid, int threads, size_t smem, int cl, cudaStream_t st, A&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2]{};
    if (cl > 1) {
        at[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        at[cfg.numAttrs].val.clusterDim.x = cl;
        at[cfg.numAttrs].val.clusterDim.y = at[cfg.numAttrs].val.clusterDim.z = 1;
        ++cfg.numAttrs;
    }
    if (dep) {
        at[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
        ++cfg.numAttrs;
    }
    cfg.attrs = at;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// Split of a slab pass (k_slab.cuh) over the blocks of a cluster: chosen from
// the lattice alone, so that a system's sums do not depend on the batch.
struct SlabPlan {
    int CL;                       // blocks per slab
    int cpc, rpc;                 // columns iz and rows ky per block
    int sls;                      // row stride of a block's columns S[My][sls]
    int G;                        // rows a warp transforms at a time
    int nthr;
    int wide;                     // FP64: the block's warps share the rows of all of them
    FastDiv dcpc;                 // division by cpc
};

// Lattice description shared by every kernel (device pointers).
struct LatticeDev {
    int Nx, Ny, Nz, N;            // box extents, occupied cells
    int Mx, My, Mz;               // padded FFT extents (even)
    int Hx, Hy, Hz;               // reduced D-hat extents: M/2 + 1
    const int* cellmap;           // [Nx][Ny][Nz] (slab-major) -> internal dipole index or -1
    const uint8_t* mat;           // [N] 0-based material
    const int* dip_cell;          // [N] internal dipole -> cell index ix + Nx (iy + Ny iz)
    const int2* col_range;        // [Ny][Nx] occupied iz range [first, last+1) (first = last = 0 if empty)
    const int4* colinfo;          // [Nx][Ny] (index of the column's first dipole - first, first, last+1, 0)
    int contig;                   // 1 if every column's occupied cells are contiguous in z (colinfo is exact)
    int nmat;                     // materials used by the lattice (1: one coefficient per system)
    const double* igt;            // D-hat build only: cell tables of the igt_so interaction (igt.cu), or
                                  // nullptr for point dipoles
    Plan2 qx, qy, qz;
    SlabPlan s32, s64;            // slab passes in FP32 and FP64
    int xw32, xw64;               // x-pass tile width chosen by the autotuner (0: size heuristic)
    int xmode;                    // register x pass: 0 choose by availability, 1 direct loads, 2 tensor copies
    const double2* tw64x; const double2* tw64y; const double2* tw64z;   // exp(-2 pi i t / M)
    const float2* tw32x; const float2* tw32y; const float2* tw32z;
};

// Dipole at depth iz of a column whose occupied cells are contiguous:
// ci = (index of the column's first dipole - its first iz, first iz, last iz + 1).
__host__ __device__ __forceinline__ int col_dip(int4 ci, int iz) { return (iz >= ci.y && iz < ci.z) ? ci.x + iz : -1; }

// y = diag[m] x - coef[m] * conv(coef[m'] x) / M for a batch of systems.
// conv(u)_i = sum_{j != i} G~'(r_i - r_j) u_j evaluated by zero-padded FFT.
// Per-system per-material coefficients are FP64 [S][EELS_MAX_MAT].
template <typename Rl>
struct MatvecArgs {
    const cx<Rl>* x;              // [S][3][N]
    cx<Rl>* y;                    // [S][3][N]
    cx<Rl>* U;                    // scratch [S][3][My][Nx][Mz]
    const cx<Rl>* Dr;             // reduced D-hat [slot][6][Hy][Hx][Hz]
    const int* sys_slot;          // [S] D-hat slot of each system
    const double2* coef;          // [S][EELS_MAX_MAT]
    const double2* diag;          // [S][EELS_MAX_MAT]
    const int* active;            // [S] or nullptr
    double* dot_part;             // optional [S][matvec_dot_parts][4]: per-block sum x.y (unconjugated), written by
                                  // the last kernel
    const float2* Dx;             // FP32 D-hat [slot][Hy][Hz][6][Hx] (register x pass), or nullptr
    int S;
    int dep;                      // generic passes start while the kernel before them drains (set by launch_matvec)
    int no_dep;                   // the caller's kernels may not (see inner_solve)
    int spb;                      // systems per x-pass block (consecutive systems that usually share a
                                  // D-hat slot: the beams of one energy); 0 or 1: one
};

// Cell-integrated Green's tensor (igt_so): lattice offsets of max-norm <=
// IGT_NEAR take exp(i kappa R) (-T0 + i kappa T1 + kappa^2 T2); the host
// table holds, per offset (x fastest over [-IGT_NEAR, IGT_NEAR]^3), T0, T1,
// T2 in the component order xx xy xz yy yz zz (18 doubles), lattice units.
constexpr int IGT_NEAR = 3;
constexpr double IGT_C1 = 2.3800773639795505;   // integral of 1/|u| over the unit cube: 3 ln(2 + sqrt 3) - pi/2
const std::vector<double>& igt_tables();

Plan2 make_plan2(int L);
SlabPlan make_slab_plan(const LatticeDev& L, size_t el);   // el: bytes of a complex element
size_t slab_smem(const LatticeDev& L, const SlabPlan& p, size_t el);
template <typename Rl> void prepare_slab_kernels();
// Slab pass of any y and z length (forward: gather to U; inverse: U to y).
template <typename Rl>
void launch_slab(const LatticeDev& L, const MatvecArgs<Rl>& a, bool inv, cudaStream_t st);
// Whether the kernels of a matvec of S systems overlap their starts with the
// ends of the ones before them: where no pass has more blocks than there are
// SMs: the FP64 matvec of one system of 12^3 cells takes 33.9 us in place of 39.1.
// Larger grids do not: with it on every kernel the inner solve of 16 FP64 systems
// of 11 x 11 x 31 cells took 43.1 ms in place of 38.8.
bool matvec_dep(const LatticeDev& L, int S, bool fp64);
// Partial sums of x^T (A x) per system that launch_matvec writes to dot_part.
int matvec_dot_parts(const LatticeDev& L, bool fp64);

template <typename Rl>
void launch_matvec(const LatticeDev& L, const MatvecArgs<Rl>& a, cudaStream_t st);

// D-hat build for n_slot energies: kappa[slot] = k d (complex).  Scratch of
// n_slot * dhat_scratch_bytes; outputs the octant D-hat [slot][comp][ky][kx][kz]
// in FP64 and FP32 and, with Dx32, [slot][ky][kz][comp][kx] (read by the
// register-resident x pass).
size_t dhat_scratch_bytes(const LatticeDev& L);
void launch_dhat_build(const LatticeDev& L, int n_slot, const double2* kappa, double2* scratch,
                       double2* Dr64, float2* Dr32, cudaStream_t st, float2* Dx32 = nullptr);
// Register-resident x pass (Mx = 64 or 128, FP32): false when the lattice or
// the arguments do not suit it (the caller then launches the shared-memory one).
bool xpass_reg_supported(const LatticeDev& L);
bool launch_xpass_reg(const LatticeDev& L, const MatvecArgs<float>& a, cudaStream_t st);
// Times the register x pass on the systems of a (CUDA events on st; not
// during a stream capture) for each way of moving U (direct loads, tensor
// copies when available) and each number of systems per block in
// {1, 2, 4, 8, 16} up to max_spb, and returns the fastest in *mode, *spb.
// The x pass transforms a.U in place: its contents are lost.  *log
// receives every timed candidate as (mode, spb, ms of three launches).
void autotune_xreg(const LatticeDev& L, const MatvecArgs<float>& a, int max_spb, cudaStream_t st, int* mode, int* spb,
                   std::vector<std::array<float, 3>>* log);

// Bounded device-side waits that gave up since the library was loaded (each
// one left its kernel's results incomplete).  Reading it synchronises the device.
unsigned int wait_timeouts();

// Shared-memory x pass of any length, w kz-adjacent lines per block (a power
// of two; narrower when the grid would leave SMs idle).
template <typename Rl> size_t xline_smem(const LatticeDev& L, int w);   // shared memory of such a block
template <typename Rl> bool xline_fits(const LatticeDev& L, int w);
template <typename Rl> void launch_xline(const LatticeDev& L, const MatvecArgs<Rl>& a, int w, cudaStream_t st);
template <typename Rl> void prepare_xline_kernels();
// Times the x pass with every tile width whose shared memory fits, on the
// systems of a (CUDA events on st; not during a stream capture), and returns
// the fastest width.  The x pass transforms a.U in place: its contents are
// lost.
template <typename Rl>
int autotune_xpass(const LatticeDev& L, const MatvecArgs<Rl>& a, cudaStream_t st);

// Raise the dynamic shared-memory limit of every kernel instance (call once
// per device before any launch or stream capture).
void prepare_kernels();

// Incident field for S systems (per-system params in SysField), FP64 out [S][3][N].
struct SysField {
    double2 kt;         // omega d / (gamma_h v): Bessel argument per unit b/d
    double2 inv_gamma;  // 1 / gamma_h
    double2 pref_unit;  // phase of the Eq. 25 prefactor
    double wdv;         // omega d / v
    double x0, y0;      // beam, lattice units relative to the lattice centre (electron along +z)
    // electron along an arbitrary direction n: the trajectory passes through p
    // (lattice units relative to the lattice centre); along_z selects the +z
    // kernels, for which p = (x0, y0, 0) and n = z
    double px, py, pz, nx, ny, nz;
    int along_z;
};
// along_z: every system's electron moves along +z (the per-column kernel)
void launch_incident_field(const LatticeDev& L, int S, const SysField* sys, bool along_z, double2* e,
                           cudaStream_t st);
void launch_aux_field(const LatticeDev& L, int S, const SysField* sys, const double2* e, double2* ea, cudaStream_t st);
void launch_bessel(const double2* z, double2* k0, double2* k1, int n, cudaStream_t st);

}  // namespace eels
