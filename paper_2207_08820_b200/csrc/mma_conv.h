// Tensor-core convolution on packed bitplanes (mma_conv.cu): host interface shared by the entry points.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace bs {

// Column c of a 32-filter group of the accumulator tile holds filter mma_filter_of_column(c) of the group, and byte b of a
// 32-channel block of either operand holds channel mma_channel_of_byte(b): the orders in which the epilogue can pair its
// outputs and the expansion can cut bytes out of the plane words without moving single bits (see mma_kernel.cuh).
__host__ __device__ constexpr int mma_filter_of_column(int c) { return 16 * (c & 1) + 2 * ((c >> 1) & 7) + (c >> 4); }
__host__ __device__ constexpr int mma_column_of_filter(int f) { return 16 * (f & 1) + 2 * ((f & 15) >> 1) + (f >> 4); }
__host__ __device__ constexpr int mma_channel_of_byte(int b) { return 8 * (b & 3) + (b >> 2); }

// Whether a layer runs on nibbles (kind::mxf4, see mma_kernel.cuh): codes of at most two bits on both sides whose sums stay below 2^22 whatever
// the signs.  Also the form of its prepared filters, so it depends only on what their preparation knows.  Signed filters of three bits say by their
// sign what they were prepared as: a tensor in the other form is converted in each launch, 2 to 20 times the time (4096 x 4096 x 4608, two by three
// bits: 94 us on int8, 64 on nibbles, 1496 on int8 filters converted), so those of callers who don't say are int8 for activations of every width.
constexpr bool mma_nibbles(int C, int RS, int a_bits, int w_bits, int w_sign)
{
    return a_bits <= 2 && (w_sign == BS_SIGNED_NIBBLES ? w_bits == 3 && static_cast<long long>(C) * RS * 28 < 4000000
                                                       : w_bits <= 2 && static_cast<long long>(C) * RS * 9 < 4000000);
}
// Packed filters run on nibbles with three bits a side as well (unsigned filters of three bits have no exact form).
constexpr bool mma_nibbles_packed(int C, int RS, int a_bits, int w_bits, int w_sign)
{
    return mma_nibbles(C, RS, a_bits, w_bits, w_sign) ||
           (a_bits <= 3 && (w_bits <= 2 ? a_bits == 3 : w_bits == 3 && w_sign == BS_SIGNED) && static_cast<long long>(C) * RS * 28 < 4000000);
}
// Prepared nibbles end with this word, four pairs of negative zeros, in room that holds no code; int8 codes (-8 .. 15) never contain its bytes.
// A layer tells the form of its filters by it and converts them where it needs the other one.
constexpr unsigned MM_NIBBLE_MARK = 0x88888888u;

#ifdef __CUDACC__
// What vector idx of prepared filters holds, [step][groups of eight filters][taps][2][8 filters][16 bytes]: nibbles of channel word 2 step + half, or 16 int8
// codes of channel word `step`.
struct FilterVector { int o, tap, half, step; };
template <class I>
__device__ __forceinline__ FilterVector filter_vector(I idx, int groups, int RS)
{
    FilterVector f;
    I t = idx / 16;
    f.half = static_cast<int>(idx / 8 % 2);
    f.tap = static_cast<int>(t % RS);       t /= RS;
    const int col = static_cast<int>(t % groups) * 8 + static_cast<int>(idx % 8);
    f.step = static_cast<int>(t / groups);
    f.o = (col & ~31) + mma_filter_of_column(col & 31);
    return f;
}
// Vector idx of n vectors of nibbles; the mark ends the tensor, in vector `last`: this one (of channels that do not exist) or one that no layer reads.
template <class I>
__device__ __forceinline__ void put_nibbles(uint4* out, I idx, I n, long long last, uint4 v)
{
    if (idx == n - 1) {
        if (last == idx) v.w = MM_NIBBLE_MARK;
        else out[last] = make_uint4(0, 0, 0, MM_NIBBLE_MARK);
    }
    out[idx] = v;
}
#endif

// Runs one layer.  `wgt` are filters prepared by bs_tc_prepare_weights; when it is null the packed filters `wgt_packed` are
// expanded inside the kernel.  chained: the caller promises that filters, scale and bias were final before the preceding
// kernel of the stream was launched.  plan_only: validate and plan, launch nothing.
int mma_conv_run(const uint32_t* act, const int8_t* wgt, const uint32_t* wgt_packed, const bs_conv_params* p, int32_t* out_i32,
                 uint32_t* out_packed, cudaStream_t st, bool chained, bool plan_only);

// A sequence of layers bound to its tensors (bs_sequence_*); the layers have been validated.
// workspace: null, or zeroed device memory of oper_workspace_bytes (oper_conv.h) bytes for layers that run on operand tensors.
struct Sequence;
int mma_sequence_create(const bs_sequence_layer* layers, int n, cudaStream_t side, void* workspace, size_t bytes, Sequence** out);
int mma_sequence_launches(const Sequence* q);
// ready: one of its input tensors whose operand forms are up to date, or null.
struct OperTensor;
const OperTensor* mma_sequence_input(const Sequence* q, const uint32_t* packed);
int mma_sequence_run(Sequence* q, const OperTensor* ready, cudaStream_t st);
void mma_sequence_destroy(Sequence* q);

}  // namespace bs
