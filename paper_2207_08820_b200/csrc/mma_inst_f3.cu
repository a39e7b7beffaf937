// Tensor-core convolution kernels on nibbles for 3-bit activations.
#include "mma_kernel.cuh"

namespace bs {
MmaKernel mma_kernel_f3(int wb, bool half, bool split) { return mma_pick_nibbles<3>(wb, half, split); }
}  // namespace bs
