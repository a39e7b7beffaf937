// Tensor-core convolution kernels on nibbles for 1-bit activations.
#include "mma_kernel.cuh"

namespace bs {
MmaKernel mma_kernel_f1(int wb, bool half, bool split) { return mma_pick_nibbles<1>(wb, half, split); }
}  // namespace bs
