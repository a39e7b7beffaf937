// Tensor-core convolution kernels on nibbles for 2-bit activations.
#include "mma_kernel.cuh"

namespace bs {
MmaKernel mma_kernel_f2(int wb, bool half, bool split) { return mma_pick_nibbles<2>(wb, half, split); }
}  // namespace bs
