// Operand tensors: activations as nibbles in the order in which the tensor cores read them (oper_kernel.cuh), and how a kernel writes them.
#pragma once
#include "common.cuh"

namespace bs {

struct FastDiv { unsigned mul, shift; int d; };      // quotient of 0 <= n < 2^31 by d as umulhi(n, mul) >> shift
inline FastDiv make_div(int d)
{
    FastDiv f{0, 0, d};
    if (d > 1) {
        int l = 0;
        while ((1LL << l) < d) ++l;                       // ceil(log2 d)
        const unsigned long long p = 31 + l;
        f.mul = static_cast<unsigned>(((1ULL << p) + d - 1) / d);
        f.shift = static_cast<unsigned>(p - 32);
    }
    return f;
}
__device__ __forceinline__ int fdiv(int n, const FastDiv& f) { return f.d == 1 ? n : static_cast<int>(__umulhi(static_cast<unsigned>(n), f.mul) >> f.shift); }

// One form of a tensor as a kernel writes it: byte address of position 0 of the first channel group written, or null.  For readers of stride 1
// position y * pitch + x of an image; for readers of stride 2 position (y / 2) * pitch + x / 2 of plane 2 (y & 1) + (x & 1).
struct OperDst {
    unsigned char* base;
    long long group;                // bytes between channel groups
    int plane, pitch, img;          // positions of a parity plane, a row, an image
};

// A tensor of packed codes [N][H][W][Cw][bits] and its forms.
struct OperTensor {
    const uint32_t* packed;
    OperDst dst1, dst2;
    int N, H, W, Cw, bits;
    FastDiv d_img, d_row;           // pixels of an image, of a row
};

__device__ __forceinline__ int oper_at1(const OperDst& d, int n, int y, int x) { return n * d.img + y * d.pitch + x; }
__device__ __forceinline__ int oper_at2(const OperDst& d, int n, int y, int x) { return n * d.img + (y >> 1) * d.pitch + (x >> 1) + (2 * (y & 1) + (x & 1)) * d.plane; }
__device__ __forceinline__ uint32_t* oper_words(const OperDst& d, int word, int at) { return reinterpret_cast<uint32_t*>(d.base + word * d.group + static_cast<long long>(at) * 16); }

// 32 codes of a position: e, d = those of the even and the odd channels, two bits each.  Nibble j of word m is channel 4 j + m.
__device__ __forceinline__ void oper_put(const OperDst& d1, const OperDst& d2, int word, int at1, int at2, uint32_t e, uint32_t d)
{
    const uint4 v = make_uint4(e & 0x33333333u, d & 0x33333333u, (e >> 2) & 0x33333333u, (d >> 2) & 0x33333333u);
    if (d1.base) *reinterpret_cast<uint4*>(oper_words(d1, word, at1)) = v;
    if (d2.base) *reinterpret_cast<uint4*>(oper_words(d2, word, at2)) = v;
}
// Plane words of two bits (of one: p1 = 0) -> codes of the even and of the odd channels.
__device__ __forceinline__ void oper_pairs(uint32_t p0, uint32_t p1, uint32_t& e, uint32_t& d)
{
    e = (p0 & 0x55555555u) | ((p1 << 1) & 0xAAAAAAAAu);
    d = ((p0 >> 1) & 0x55555555u) | (p1 & 0xAAAAAAAAu);
}

}  // namespace bs
