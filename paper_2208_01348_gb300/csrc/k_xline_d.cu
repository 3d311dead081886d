// Shared-memory x pass, FP64 kernels.
#include "k_xline.cuh"

namespace eels {
template size_t xline_smem<double>(const LatticeDev&, int);
template bool xline_fits<double>(const LatticeDev&, int);
template void launch_xline<double>(const LatticeDev&, const MatvecArgs<double>&, int, cudaStream_t);
template void prepare_xline_kernels<double>();
}  // namespace eels
