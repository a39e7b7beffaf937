// Tensor-core convolution kernels for 4-bit activations.
#include "mma_kernel.cuh"

namespace bs {
MmaKernel mma_kernel_a4(int wb, bool half, bool split) { return mma_pick<4>(wb, half, split); }
}  // namespace bs
