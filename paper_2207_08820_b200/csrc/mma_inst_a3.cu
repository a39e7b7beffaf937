// Tensor-core convolution kernels for 3-bit activations.
#include "mma_kernel.cuh"

namespace bs {
MmaKernel mma_kernel_a3(int wb, bool half, bool split) { return mma_pick<3>(wb, half, split); }
}  // namespace bs
