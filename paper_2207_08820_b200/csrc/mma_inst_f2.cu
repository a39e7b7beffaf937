// Tensor-core convolution kernels on nibbles for 2-bit activations.
#include "mma_kernel.cuh"

namespace bs {
MmaKernel mma_kernel_f2(int wb, bool half, bool split) { return mma_pick_nibbles<2>(wb, half, split); }
}  // namespace bs

#ifdef BS_TRACE
// Trace builds: copies the timeline table of the last launches with 2-bit activations and filters of at most two bits to `out` (HOST, 148 x 12 x 48 cycle counts).
extern "C" int bs_tc_trace_read(long long* out, int clear)
{
    if (cudaDeviceSynchronize() != cudaSuccess) return BS_ERR_CUDA;
    if (cudaMemcpyFromSymbol(out, bs::g_mm_trace, sizeof(bs::g_mm_trace)) != cudaSuccess) return BS_ERR_CUDA;
    if (clear) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, bs::g_mm_trace) != cudaSuccess || cudaMemset(p, 0, sizeof(bs::g_mm_trace)) != cudaSuccess) return BS_ERR_CUDA;
    }
    return BS_OK;
}
#endif
