// Tensor-core convolution kernels for 2-bit activations.
#include "mma_kernel.cuh"

namespace bs {
MmaKernel mma_kernel_a2(int wb, bool half, bool split) { return mma_pick<2>(wb, half, split); }
}  // namespace bs
