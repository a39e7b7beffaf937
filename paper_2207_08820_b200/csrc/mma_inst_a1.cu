// Tensor-core convolution kernels for 1-bit activations.
#include "mma_kernel.cuh"

namespace bs {
MmaKernel mma_kernel_a1(int wb, bool half, bool split) { return mma_pick<1>(wb, half, split); }
}  // namespace bs
