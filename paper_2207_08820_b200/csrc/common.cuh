// Shared host/device helpers of the bit-serial library (CUDA side only).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "bitserial.h"

namespace bs {

// Device status word: kernels OR error bits into it when a bounded wait runs out.
enum : int { STATUS_TIMEOUT = 1 };
int* status_device_ptr();   // device address of the status word of the current device (host call)
int device_sm_count();      // multiprocessors of the CURRENT device (looked up once per device ordinal; 0 on error)

inline int ceil_div(int a, int b) { return (a + b - 1) / b; }
inline long long ceil_div_ll(long long a, long long b) { return (a + b - 1) / b; }

inline bool bits_ok(int bits, int sign)
{
    if (bits < 1 || bits > 4) return false;
    if (sign != BS_UNSIGNED && sign != BS_SIGNED && sign != BS_BIPOLAR) return false;
    if (sign == BS_BIPOLAR && bits != 1) return false;
    return true;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Stored pattern of a code: low `bits` bits, or (code > 0) for bipolar.
__device__ __forceinline__ unsigned stored_pattern(int code, int bits, int sign)
{
    return sign == BS_BIPOLAR ? (code > 0 ? 1u : 0u) : (static_cast<unsigned>(code) & ((1u << bits) - 1u));
}

// Value of a stored pattern.
__device__ __forceinline__ int pattern_value(unsigned pat, int bits, int sign)
{
    if (sign == BS_BIPOLAR) return pat ? 1 : -1;
    int v = static_cast<int>(pat);
    if (sign == BS_SIGNED && (pat >> (bits - 1))) v -= (1 << bits);
    return v;
}

__host__ __device__ __forceinline__ void code_limits(int bits, int sign, int& qmin, int& qmax)
{
    if (sign == BS_SIGNED) { qmin = -(1 << (bits - 1)); qmax = (1 << (bits - 1)) - 1; }
    else if (sign == BS_BIPOLAR) { qmin = -1; qmax = 1; }
    else { qmin = 0; qmax = (1 << bits) - 1; }
}

// Launch that may begin while the kernel before it drains (about 1.5 us of launch latency hidden); the kernel calls dependent_begin first.
template <typename... P, typename... A>
inline int launch_dependent(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...) != cudaSuccess) {
        cudaGetLastError();
        return BS_ERR_CUDA;
    }
    return BS_OK;
}
// First statement of every thread of such a kernel: lets the next launch begin, waits for the kernel before.  Read-only loads may move
// above the wait unless their address comes out of it: `p` is returned through it.
template <typename T>
__device__ __forceinline__ T* dependent_begin(T* p)
{
    asm volatile("griddepcontrol.launch_dependents;\n\tgriddepcontrol.wait;" : "+l"(p) : : "memory");
    return p;
}

}  // namespace bs
