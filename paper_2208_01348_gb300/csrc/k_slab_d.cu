// Slab passes, FP64 kernels.
#include "k_slab.cuh"

namespace eels {
template void launch_slab<double>(const LatticeDev&, const MatvecArgs<double>&, bool, cudaStream_t);
template void prepare_slab_kernels<double>();
}  // namespace eels
