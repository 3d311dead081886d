// Shared-memory x pass, FP32 kernels.
#include "k_xline.cuh"

namespace eels {
template size_t xline_smem<float>(const LatticeDev&, int);
template bool xline_fits<float>(const LatticeDev&, int);
template void launch_xline<float>(const LatticeDev&, const MatvecArgs<float>&, int, cudaStream_t);
template void prepare_xline_kernels<float>();
}  // namespace eels
