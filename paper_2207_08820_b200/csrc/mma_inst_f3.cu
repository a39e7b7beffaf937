// Tensor-core convolution kernels on nibbles for 3-bit activations.
#include "mma_kernel.cuh"

namespace bs {
MmaKernel mma_kernel_f3(int wb, bool half, bool split, bool offset)
{
    if (offset) return wb == 1 ? mma_pick_offset<1>(half) : wb == 2 ? mma_pick_offset<2>(half) : mma_pick_offset<3>(half);
    return mma_pick_nibbles<3>(wb, half, split);
}
}  // namespace bs
