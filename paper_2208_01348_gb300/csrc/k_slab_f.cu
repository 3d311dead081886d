// Slab passes, FP32 kernels.
#include "k_slab.cuh"

namespace eels {
template void launch_slab<float>(const LatticeDev&, const MatvecArgs<float>&, bool, cudaStream_t);
template void prepare_slab_kernels<float>();
}  // namespace eels
