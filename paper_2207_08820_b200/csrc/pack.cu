// Quantise + bitplane split of activations (Section IV quantiser, Section V plane split), the inverse
// unpack, and the offline plane split of weights / matrix rows.
#include <cmath>
#include <cstring>
#include <type_traits>

#include "common.cuh"
#include "oper_tensor.cuh"

namespace bs {

// Quantiser of Section IV prepared for the device.  The decision
//     code = round_half_even(clip(x / s, qmin, qmax))
// is monotone in x, so it equals qmin + #{k : x >= bound[k]} where bound[k] is the smallest binary32 value whose
// code is >= qmin + k + 1.  The host finds those bounds by bisection over the ordered float bit patterns using the very
// same IEEE division, clip and rint, so the comparison form takes exactly the decision of the formula while costing
// a few subtractions instead of a division (a binary search over the bounds for 3 and 4 bits).
struct QuantParams {
    float below[16];    // largest binary32 value below bound[k] (never -0): x >= bound[k]  <=>  sign bit of (below[k] - x) is set
    int bits, sign;
    float inv, offset;  // estimate of the level, see LevelPlanes: x * inv + offset
    int estimate;       // the scale is one for which the estimate holds
};

// Stores the BITS plane words of one (pixel, channel word) with the widest aligned store.
template <int BITS>
__device__ __forceinline__ void store_planes(uint32_t* dst, const uint32_t (&w)[BITS])
{
    if constexpr (BITS == 4) *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
    else if constexpr (BITS == 2) *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
    else {
#pragma unroll
        for (int j = 0; j < BITS; ++j) dst[j] = w[j];
    }
}

// Sign-bit form of the comparison quantiser for fp32 input.
//   With p the largest binary32 value below the bound b:  x >= b  <=>  x > p  <=>  the sign bit of p - x is set.
//   An IEEE subtraction never rounds across zero and x == p gives +0; p is stored as +0 when it is a zero, so neither
//   signed zero of x yields -0.  A NaN input gives the canonical NaN (sign clear): no level reached, the lowest
//   code, which is what clip() makes of a NaN in the formula.  +-inf behave like the comparison.
//   2-bit codes: plane 1 = (x >= b1); plane 0 = parity of the three comparisons = sign((p0-x) ^ (p1-x) ^ (p2-x)).
//   3- and 4-bit codes: LevelPlanes below; for scales it does not take, the 7 or 15 bounds are searched binarily: one subtraction,
//   one sign test and one funnel shift per bit plus the selects that pick the next bound.
// One funnel shift moves a sign bit into a plane word (w = 2 w + bit); the inputs of a word are walked from position 31
// down to 0 so that input i ends at bit i.  Per element of a 2-bit tensor: one load, three subtractions, one three-input
// xor and two funnel shifts, which leaves the kernels waiting on HBM rather than on the issue slots.
// Shifts the BITS plane bits of one input into the plane words w (w = 2 w + bit), in the sign-bit comparison form.
template <int BITS>
__device__ __forceinline__ void quant_push(const QuantParams& q, float v, uint32_t (&w)[BITS])
{
    if constexpr (BITS == 1) {
        w[0] = __funnelshift_l(__float_as_uint(q.below[0] - v), w[0], 1);
    } else if constexpr (BITS == 2) {
        const uint32_t d0 = __float_as_uint(q.below[0] - v), d1 = __float_as_uint(q.below[1] - v),
                       d2 = __float_as_uint(q.below[2] - v);
        w[1] = __funnelshift_l(d1, w[1], 1);
        w[0] = __funnelshift_l(d0 ^ d1 ^ d2, w[0], 1);
    } else {
        // binary search for the count of bounds reached, top bit first: with the higher bits m decided, bit L is
        // "bound number m * 2^(L+1) + 2^L reached"; the candidates are folded with selects on the decided bits
        bool c[BITS];
#pragma unroll
        for (int L = BITS - 1; L >= 0; --L) {
            constexpr int MAXC = 1 << (BITS - 1);
            float sel[MAXC];
            const int nd = BITS - 1 - L;
#pragma unroll
            for (int m = 0; m < MAXC; ++m)
                if (m < (1 << nd)) sel[m] = q.below[m * (2 << L) + (1 << L) - 1];
#pragma unroll
            for (int d = 0; d < BITS - 1; ++d)
                if (d < nd) {
#pragma unroll
                    for (int m = 0; m < MAXC / 2; ++m)
                        if (m < (1 << (nd - d - 1))) sel[m] = c[L + 1 + d] ? sel[2 * m + 1] : sel[2 * m];
                }
            const uint32_t e = __float_as_uint(sel[0] - v);
            c[L] = static_cast<int>(e) < 0;
            w[L] = __funnelshift_l(e, w[L], 1);
        }
    }
}

// Plane words of 32 inputs, pushed from input 31 down to input 0, in the sign-bit comparison form.
template <int BITS>
struct SignPlanes {
    uint32_t w[BITS];
    const QuantParams& q;
    __device__ __forceinline__ SignPlanes(const QuantParams& q_, const float*) : q(q_)
    {
#pragma unroll
        for (int j = 0; j < BITS; ++j) w[j] = 0u;
    }
    __device__ __forceinline__ void push(int, float v) { quant_push<BITS>(q, v, w); }
    __device__ __forceinline__ void finish() {}
};

// The same for 3 and 4 bits by estimate and check: k = round(x * inv + offset) with offset = -qmin - 2^-10 is the level (code - qmin) or
// one less (x * inv is within 2^-19 of x / s for every x whose level is not clipped), and which of the two it is, the exact bound of
// level k + 1 decides: level = k + (x >= bound[k]), one look-up in a table of 16 floats in shared memory (different entries lie in
// different banks).  A NaN ends at level 0 (the clamp drops it, the comparison fails), infinities at the ends.
// Adding 1.5 * 2^23 leaves k in the low mantissa bits.  The levels of inputs 4 i + g are gathered as the nibbles i of word g, so that
// plane j is the or over g of ((word g >> j) & 0x11111111) << g: two instructions per word and plane.  About 10 instructions an
// element against 27 of the search, which bound the kernel (64x64x56x56, 4 bits, NCHW: 17.2 -> 12.5 us).
template <int BITS>
struct LevelPlanes {
    uint32_t w[BITS], r[4];
    uint32_t table;
    float inv, offset;
    __device__ __forceinline__ LevelPlanes(const QuantParams& q, const float* s_below)
        : table(static_cast<uint32_t>(__cvta_generic_to_shared(s_below)) - (0x4B400000u << 2)), inv(q.inv), offset(q.offset)
    {
#pragma unroll
        for (int g = 0; g < 4; ++g) r[g] = 0u;
    }
    __device__ __forceinline__ void push(int u, float v)
    {
        constexpr float top = static_cast<float>((1 << BITS) - 1);
        const uint32_t k = __float_as_uint(fminf(fmaxf(fmaf(v, inv, offset), 0.0f), top) + 12582912.0f);
        float below;
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(below) : "r"(table + (k << 2)));
        const uint32_t over = __float_as_uint(below - v) >> 31;
        r[u & 3] = r[u & 3] * 16u + k + over;
    }
    __device__ __forceinline__ void finish()
    {
        // the bit pattern of 1.5 * 2^23 rode along in every level
        constexpr uint32_t carried = 0x4B400000u * 0x11111111u;
#pragma unroll
        for (int g = 0; g < 4; ++g) r[g] -= carried;
#pragma unroll
        for (int j = 0; j < BITS; ++j) {
            w[j] = 0u;
#pragma unroll
            for (int g = 0; g < 4; ++g) w[j] |= (g >= j ? r[g] << (g - j) : r[g] >> (j - g)) & (0x11111111u << g);
        }
    }
};

template <int BITS, bool LEVELS> struct PlanesOf { typedef SignPlanes<BITS> type; };
template <int BITS> struct PlanesOf<BITS, true> { typedef LevelPlanes<BITS> type; };

// The table of LevelPlanes; every thread of the block calls this first.
template <bool LEVELS>
__device__ __forceinline__ void load_levels(float* s_below, const QuantParams& q)
{
    if constexpr (LEVELS) {
        if (threadIdx.x < 16) s_below[threadIdx.x] = q.below[threadIdx.x];
        __syncthreads();
    }
}

// Transpose of the 32 x 32 bit matrix whose row r is the word held by lane r: afterwards lane r holds column r.  Five
// butterfly stages; stage k swaps the off-diagonal k x k blocks between lanes r and r ^ k.
__device__ __forceinline__ uint32_t warp_transpose32(uint32_t x, int lane)
{
#pragma unroll
    for (int k = 16; k >= 1; k >>= 1) {
        const uint32_t mask = k == 16 ? 0x0000FFFFu : k == 8 ? 0x00FF00FFu : k == 4 ? 0x0F0F0F0Fu : k == 2 ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, k);
        x = (lane & k) ? ((x & ~mask) | ((y & ~mask) >> k)) : ((x & mask) | ((y & mask) << k));
    }
    return x;
}

// fp32 NCHW.  Work unit of a warp = 32 consecutive pixels of one image x one 32-channel word (lane = pixel): all 32
// channel rows are in flight at once (32 coalesced 128-byte requests per warp), walked from channel 31 down, and each lane
// stores the BITS plane words of its pixel straight to the packed record (8-byte stores for 2-bit codes; the words of
// the other channel groups of the record come from the neighbouring warps of the block, so the sectors fill up in L2).
// Units are small and numerous, which keeps the tail of the grid short; no shared memory, no barrier.
constexpr int FAST_THREADS = 128;
constexpr int FAST_WARPS = FAST_THREADS / 32;

// OPER: the codes also go to the operand tensors of the layers that read them (o), 16 bytes a lane in runs of 512, where a pass over the packed codes
// would follow.
struct NoOper {};
template <int BITS, bool LEVELS, typename Oper = NoOper>
__global__ void __launch_bounds__(FAST_THREADS, 8)
bitpack_nchw_f32_kernel(const float* __restrict__ x_in, uint32_t* __restrict__ out, int C, int HW, int Cw, long long nunits,
                        int units_per_img, const __grid_constant__ QuantParams q, const __grid_constant__ Oper o)
{
    __shared__ float s_below[16];
    load_levels<LEVELS>(s_below, q);
    const float* x = dependent_begin(x_in);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long unit = static_cast<long long>(blockIdx.x) * FAST_WARPS + warp;
    if (unit >= nunits) return;
    const long long n = unit / units_per_img;
    const int rem = static_cast<int>(unit % units_per_img);
    const int cw = rem % Cw;
    const int hw0 = (rem / Cw) * 32;
    const bool pvalid = lane < HW - hw0;
    // lanes beyond the image re-read the first pixel of the tile (always in bounds) and store nothing
    const float* xin = x + (static_cast<size_t>(n) * C + cw * 32) * HW + hw0 + (pvalid ? lane : 0);
    typename PlanesOf<BITS, LEVELS>::type planes(q, s_below);
    const int nvalid = min(32, C - cw * 32);
    const ptrdiff_t row = HW;
    float v[32];
    if (nvalid == 32) {
        // a full channel word: unconditional loads, walking the channel rows downward from channel 31
        const float* pc = xin + 31 * row;
#pragma unroll
        for (int u = 0; u < 32; ++u) {
            v[31 - u] = __ldcs(pc);
            pc -= row;
        }
    } else {
        // the ragged last word: channels past C count as "no level reached"
#pragma unroll
        for (int u = 0; u < 32; ++u) v[u] = u < nvalid ? __ldcs(xin + u * row) : -INFINITY;
    }
#pragma unroll
    for (int u = 31; u >= 0; --u) planes.push(u, v[u]);
    planes.finish();
    if (!pvalid) return;
    const unsigned fl = nvalid == 32 ? 0xffffffffu : ((1u << nvalid) - 1u);
    // pattern = (qmin + count) mod 2^BITS: two's-complement codes (qmin = -2^(BITS-1)) flip the top plane only
    if (q.sign == BS_SIGNED) planes.w[BITS - 1] ^= fl;
    store_planes<BITS>(out + ((static_cast<size_t>(n) * HW + hw0 + lane) * Cw + cw) * BITS, planes.w);
    if constexpr (!std::is_same<Oper, NoOper>::value) {
        const int y = fdiv(hw0 + lane, o.d_row), x = hw0 + lane - y * o.W;
        uint32_t even, odd;
        oper_pairs(planes.w[0], BITS > 1 ? planes.w[BITS - 1] : 0u, even, odd);
        oper_put(o.dst1, o.dst2, cw, oper_at1(o.dst1, static_cast<int>(n), y, x), oper_at2(o.dst2, static_cast<int>(n), y, x), even, odd);
    }
}

// fp32 NHWC input, comparison form at any width.  Work unit of a warp = 32 consecutive pixels x one 32-channel word, lane
// = channel: the 32 channels of a pixel are one coalesced 128-byte request and all 32 pixels of the unit are in flight
// at once.  A lane shifts the plane bits of its channel into words indexed by PIXEL (pixels walked from 31 down), a
// 32 x 32 bit transpose across the warp (five shuffles per plane) turns them into words indexed by channel held by lane
// = pixel, and the records leave as one store per lane like in the NCHW kernel.  No votes, no shared memory.
template <int BITS, bool LEVELS>
__global__ void __launch_bounds__(FAST_THREADS, 8)
bitpack_nhwc_f32_kernel(const float* __restrict__ x_in, uint32_t* __restrict__ out, int C, int HW, int Cw, long long nunits,
                        int units_per_img, const __grid_constant__ QuantParams q)
{
    __shared__ float s_below[16];
    load_levels<LEVELS>(s_below, q);
    const float* x = dependent_begin(x_in);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long unit = static_cast<long long>(blockIdx.x) * FAST_WARPS + warp;
    if (unit >= nunits) return;
    const long long n = unit / units_per_img;
    const int rem = static_cast<int>(unit % units_per_img);
    const int cw = rem % Cw;
    const int hw0 = (rem / Cw) * 32;
    const int npix = min(32, HW - hw0);
    const bool cvalid = cw * 32 + lane < C;
    const unsigned valid_word = __ballot_sync(0xffffffffu, cvalid);
    // lanes past the last channel re-read the first channel of the word (always in bounds); their words are cleared
    const float* xin = x + (static_cast<size_t>(n) * HW + hw0) * C + cw * 32 + (cvalid ? lane : 0);
    typename PlanesOf<BITS, LEVELS>::type planes(q, s_below);
    const ptrdiff_t row = C;
    float v[32];
    if (npix == 32) {
        const float* pc = xin + 31 * row;
#pragma unroll
        for (int u = 0; u < 32; ++u) {
            v[31 - u] = __ldcs(pc);
            pc -= row;
        }
    } else {
        // the ragged last tile of an image: pixels past the end count as "no level reached" and are not stored
#pragma unroll
        for (int u = 0; u < 32; ++u) v[u] = u < npix ? __ldcs(xin + u * row) : -INFINITY;
    }
#pragma unroll
    for (int u = 31; u >= 0; --u) planes.push(u, v[u]);
    planes.finish();
#pragma unroll
    for (int j = 0; j < BITS; ++j) planes.w[j] = warp_transpose32(cvalid ? planes.w[j] : 0u, lane);
    if (lane >= npix) return;
    if (q.sign == BS_SIGNED) planes.w[BITS - 1] ^= valid_word;
    store_planes<BITS>(out + ((static_cast<size_t>(n) * HW + hw0 + lane) * Cw + cw) * BITS, planes.w);
}

// Four int8 codes as plane bits: bit j of byte k is plane j of code k (the two's-complement low bits; bipolar: code > 0).
template <int BITS>
__device__ __forceinline__ uint32_t codes4(uint32_t r, bool bipolar)
{
    return BITS == 1 && bipolar ? __vcmpgts4(r, 0u) : r;
}

// int8 codes, NCHW.  At one byte per element the HBM roofline leaves about five thread instructions per element, so the plane
// split works on four pixels at a time: a lane owns four consecutive pixels of a channel row, one 32-bit word (a warp = 128
// pixels, 128-byte requests); (r >> j) & 0x01010101 is bit j of the four codes, and a = 2 a + that, over eight channel rows from
// the highest down, leaves in byte k of a the eight channel bits of pixel k.  A byte permute drops each finished byte into the
// plane word of its pixel.  About 1.8 instructions per element for 2-bit codes.  Work unit of a warp = 128 pixels x one 32-channel
// word.  ALIGNED: H*W is a multiple of four, every row starts on a word.  Otherwise the four pixels of a lane straddle two words
// (the second one is the next lane's first and comes from L1), joined by a funnel shift; byte loads of one pixel per lane, 32 bytes
// a request, took 2 to 3 times as long.
// Stores: with CW = 0 every lane writes the plane words of its pixels straight to the records (8-byte pieces of 32-byte
// sectors, four partial writes per sector).  When the channel words of a record number CW = 1, 2 or 4, the four warps of
// a block hold complete records of 4 / CW tiles: they park their words in shared memory as [warp][plane][pixel] (128-bit
// stores, no bank conflicts), and after one barrier the block writes the records as whole 128-bit pieces.
template <int BITS, int CW, bool ALIGNED>
__global__ void __launch_bounds__(FAST_THREADS, 8)
bitpack_nchw_i8_kernel(const int8_t* __restrict__ x_in, uint32_t* __restrict__ out, int C, int HW, int Cw, long long nunits,
                       int units_per_img, long long bytes, int bipolar)
{
    const int8_t* x = ALIGNED ? dependent_begin(x_in) : x_in;
    constexpr bool STAGED = CW != 0;
    __shared__ __align__(16) uint32_t stage[STAGED ? FAST_WARPS * BITS * 128 : 4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long unit = static_cast<long long>(blockIdx.x) * FAST_WARPS + warp;
    const bool active = unit < nunits;
    if (!STAGED && !active) return;
    if (active) {
        const long long n = unit / units_per_img;
        const int rem = static_cast<int>(unit % units_per_img);
        const int cw = rem % Cw;
        const int hw0 = (rem / Cw) * 128;
        const int pix = hw0 + 4 * lane;
        const bool pvalid = pix < HW;
        const int nvalid = min(32, C - cw * 32);
        uint32_t v[32];
        if constexpr (ALIGNED) {           // the four pixels of a lane are inside or outside together
            const uint32_t* xin = reinterpret_cast<const uint32_t*>(x + (static_cast<size_t>(n) * C + cw * 32) * HW + (pvalid ? pix : hw0));
            const size_t row = static_cast<size_t>(HW / 4);
            if (nvalid == 32) {
#pragma unroll
                for (int u = 0; u < 32; ++u) v[u] = codes4<BITS>(__ldcs(xin + u * row), bipolar);
            } else {
#pragma unroll
                for (int u = 0; u < 32; ++u) v[u] = u < nvalid ? codes4<BITS>(__ldcs(xin + u * row), bipolar) : 0u;
            }
        } else {
            const long long at = (n * C + cw * 32) * HW + (pvalid ? pix : hw0);
            // only whole words inside the tensor are loaded; its last, partial word is put together from bytes
            const long long whole = bytes >> 2;
            uint32_t tail = 0u;
            const long long reach = (n * C + cw * 32 + nvalid - 1) * HW + hw0 + 136;
            if (reach > 4 * whole)
                for (int k = 0; k < (bytes & 3); ++k) tail |= static_cast<uint32_t>(static_cast<uint8_t>(x[4 * whole + k])) << (8 * k);
            const uint32_t* xw = reinterpret_cast<const uint32_t*>(x);
#pragma unroll
            for (int u = 0; u < 32; ++u) {
                const long long byte = at + static_cast<long long>(u < nvalid ? u : 0) * HW, i = byte >> 2;
                const uint32_t lo = i < whole ? __ldg(xw + i) : tail, hi = i + 1 < whole ? __ldg(xw + i + 1) : tail;
                v[u] = __funnelshift_r(lo, hi, static_cast<int>(byte & 3) * 8);
            }
#pragma unroll
            for (int u = 0; u < 32; ++u) v[u] = u < nvalid ? codes4<BITS>(v[u], bipolar) : 0u;
        }
        uint32_t w[4][BITS];
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int j = 0; j < BITS; ++j) w[k][j] = 0u;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            uint32_t a[BITS];
#pragma unroll
            for (int j = 0; j < BITS; ++j) a[j] = 0u;
#pragma unroll
            for (int i = 7; i >= 0; --i) {
                const uint32_t r = v[8 * g + i];
#pragma unroll
                for (int j = 0; j < BITS; ++j) a[j] = a[j] * 2u + ((r >> j) & 0x01010101u);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int j = 0; j < BITS; ++j)      // byte k of a[j] becomes byte g of the plane word of pixel k
                    w[k][j] = __byte_perm(w[k][j], a[j], (0x3210u & ~(0xfu << (4 * g))) | ((4u + k) << (4 * g)));
        }
        if constexpr (STAGED) {
#pragma unroll
            for (int j = 0; j < BITS; ++j)
                *reinterpret_cast<uint4*>(stage + (warp * BITS + j) * 128 + 4 * lane) = make_uint4(w[0][j], w[1][j], w[2][j], w[3][j]);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (pix + k < HW) store_planes<BITS>(out + ((static_cast<size_t>(n) * HW + pix + k) * Cw + cw) * BITS, w[k]);
        }
    }
    if constexpr (STAGED) {
        __syncthreads();
        // the block's first unit is a multiple of 4, hence of CW: warp t * CW + c holds channel word c of the block's tile t
        constexpr int REC = CW * BITS;                 // words of a pixel record
        constexpr int PIECE = REC % 4 == 0 ? 4 : (REC % 2 == 0 ? 2 : 1);     // words per store
#pragma unroll
        for (int t = 0; t < FAST_WARPS / CW; ++t) {
            const long long unit_t = static_cast<long long>(blockIdx.x) * FAST_WARPS + t * CW;
            if (unit_t >= nunits) break;
            const long long n = unit_t / units_per_img;
            const int hw0 = (static_cast<int>(unit_t % units_per_img) / CW) * 128;
            const int nwords = min(128, HW - hw0) * REC;            // a multiple of 4: H*W and the tile start are
            uint32_t* dst = out + (static_cast<size_t>(n) * HW + hw0) * REC;
            for (int i = threadIdx.x * PIECE; i < nwords; i += FAST_THREADS * PIECE) {
                uint32_t piece[PIECE];
#pragma unroll
                for (int e = 0; e < PIECE; ++e) {
                    const int idx = i + e, p = idx / REC, r = idx % REC;          // (pixel, word of its record)
                    piece[e] = stage[((t * CW + r / BITS) * BITS + r % BITS) * 128 + p];
                }
                if constexpr (PIECE == 4) *reinterpret_cast<uint4*>(dst + i) = make_uint4(piece[0], piece[1], piece[2], piece[3]);
                else if constexpr (PIECE == 2) *reinterpret_cast<uint2*>(dst + i) = make_uint2(piece[0], piece[1]);
                else dst[i] = piece[0];
            }
        }
    }
}

// int8 codes, NHWC, C a multiple of 32: the 32 channels of a (pixel, channel word) are 32 contiguous, aligned bytes.
// Lane = pixel; a warp takes 128 pixels x one channel word (four pixels per lane, eight 128-bit loads in flight).  For
// each word of four codes, ((q >> j) & 0x01010101) * 0x01020408 gathers bit j of the four bytes in bits 24..27 (all
// partial products fall on distinct bits, so nothing carries).  About 2.5 instructions per element for 2-bit codes.
template <int BITS>
__global__ void __launch_bounds__(FAST_THREADS, 8)
bitpack_nhwc_i8_kernel(const int8_t* __restrict__ x_in, uint32_t* __restrict__ out, int C, int HW, int Cw, long long nunits,
                       int units_per_img)
{
    const int8_t* x = dependent_begin(x_in);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long unit = static_cast<long long>(blockIdx.x) * FAST_WARPS + warp;
    if (unit >= nunits) return;
    const long long n = unit / units_per_img;
    const int rem = static_cast<int>(unit % units_per_img);
    const int cw = rem % Cw;
    const int hw0 = (rem / Cw) * 128;
    uint4 q[4][2];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const int pix = min(hw0 + 32 * t + lane, HW - 1);       // clamped: always in bounds, stored only when inside
        const uint4* src = reinterpret_cast<const uint4*>(x + (static_cast<size_t>(n) * HW + pix) * C + cw * 32);
        q[t][0] = __ldcs(src);
        q[t][1] = __ldcs(src + 1);
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const uint32_t words[8] = {q[t][0].x, q[t][0].y, q[t][0].z, q[t][0].w, q[t][1].x, q[t][1].y, q[t][1].z, q[t][1].w};
        uint32_t w[BITS];
#pragma unroll
        for (int j = 0; j < BITS; ++j) w[j] = 0u;
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < BITS; ++j)
                w[j] |= ((((words[i] >> j) & 0x01010101u) * 0x01020408u) >> 24) << (4 * i);
        const int pix = hw0 + 32 * t + lane;
        if (pix < HW) store_planes<BITS>(out + ((static_cast<size_t>(n) * HW + pix) * Cw + cw) * BITS, w);
    }
}

// int8 codes, NHWC, any C and any code: the whole tensor is one run of N*H*W records of C bytes, so a block takes `pix` consecutive
// pixels (64, fewer where C is large) = one contiguous run of bytes (no image boundary), staged into shared memory by 16-byte asynchronous copies from the
// 16-byte boundary at or below its start.  A thread then takes one (pixel, channel word): nine words of the stage from the one its
// first byte lies in, joined by funnel shifts, and the same plane gathering as above; bits of channels past C are masked out of the
// finished words, so what the stage holds behind the last record does not matter.  Neighbouring threads take neighbouring
// channel words of a pixel: the packed records leave as one contiguous run.  Byte loads with votes took 10 times as long
// (48 x 45 x 61 pixels of 50 channels, 2 bits: 18.2 -> 3.9 us a call).
constexpr int RAGGED_PIX = 64, RAGGED_BYTES = 40 * 1024;

template <int BITS>
__global__ void __launch_bounds__(FAST_THREADS)
bitpack_nhwc_ragged_i8_kernel(const int8_t* __restrict__ x_in, uint32_t* __restrict__ out, int C, int Cw, long long npix, int pix, int bipolar)
{
    extern __shared__ __align__(16) uint32_t ragged_smem[];
    const int8_t* x = dependent_begin(x_in);
    const long long p0 = static_cast<long long>(blockIdx.x) * pix;
    const int np = static_cast<int>(npix - p0 < pix ? npix - p0 : pix);
    const long long first = p0 * C, begin = first & ~15LL, end = first + static_cast<long long>(np) * C;
    const int lead = static_cast<int>(first - begin), span = static_cast<int>(end - begin);
    const int8_t* src = x + begin;
    int8_t* stage = reinterpret_cast<int8_t*>(ragged_smem);
    const int whole = end < npix * C ? (span + 15) / 16 : span / 16;       // 16-byte pieces inside the tensor
    for (int i = threadIdx.x; i < whole; i += FAST_THREADS) {
        const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(stage + 16 * i));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src + 16 * i) : "memory");
    }
    for (int i = 16 * whole + threadIdx.x; i < span; i += FAST_THREADS) stage[i] = src[i];
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const int nwords = np * Cw;
    uint32_t* dst = out + static_cast<size_t>(p0) * Cw * BITS;
    for (int i = threadIdx.x; i < nwords; i += FAST_THREADS) {
        const int p = i / Cw, cw = i - p * Cw;
        const int byte = lead + p * C + cw * 32;
        const uint32_t* q = ragged_smem + (byte >> 2);
        const int sh = (byte & 3) * 8;
        const int nvalid = C - cw * 32;
        const uint32_t valid = nvalid >= 32 ? 0xffffffffu : (1u << nvalid) - 1u;
        uint32_t w[BITS];
#pragma unroll
        for (int j = 0; j < BITS; ++j) w[j] = 0u;
        uint32_t lo = q[0];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t hi = q[k + 1];
            const uint32_t r = codes4<BITS>(__funnelshift_r(lo, hi, sh), bipolar);
            lo = hi;
#pragma unroll
            for (int j = 0; j < BITS; ++j) w[j] |= ((((r >> j) & 0x01010101u) * 0x01020408u) >> 24) << (4 * k);
        }
#pragma unroll
        for (int j = 0; j < BITS; ++j) w[j] &= valid;
        store_planes<BITS>(dst + static_cast<size_t>(i) * BITS, w);
    }
}

__global__ void bitunpack_kernel(const uint32_t* __restrict__ packed, int8_t* __restrict__ codes, long long total,
                                 int C, int HW, int Cw, int bits, int sign, int nhwc)
{
    const long long idx = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    // idx enumerates the OUTPUT layout
    long long n, c, hw;
    if (nhwc) { c = idx % C; hw = (idx / C) % HW; n = idx / (static_cast<long long>(C) * HW); }
    else      { hw = idx % HW; c = (idx / HW) % C; n = idx / (static_cast<long long>(C) * HW); }
    const uint32_t* rec = packed + ((n * HW + hw) * Cw + c / 32) * bits;
    unsigned pat = 0;
    for (int j = 0; j < bits; ++j) pat |= ((rec[j] >> (c % 32)) & 1u) << j;
    codes[idx] = static_cast<int8_t>(pattern_value(pat, bits, sign));
}

// One thread per packed word group (o, tap, cw): reads 32 channel codes, emits `bits` plane words.
__global__ void pack_weights_kernel(const int8_t* __restrict__ w, uint32_t* __restrict__ out, long long ngroups,
                                    int C, int RS, int Cw, int bits, int sign, int ohwi)
{
    const long long g = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (g >= ngroups) return;
    const int cw = static_cast<int>(g % Cw);
    const int tap = static_cast<int>((g / Cw) % RS);
    const long long o = g / (static_cast<long long>(Cw) * RS);
    unsigned words[4] = {0, 0, 0, 0};
    for (int b = 0; b < 32; ++b) {
        const int c = cw * 32 + b;
        if (c >= C) break;
        const long long src = ohwi ? ((o * RS + tap) * C + c) : ((o * C + c) * RS + tap);
        const unsigned pat = stored_pattern(w[src], bits, sign);
#pragma unroll
        for (int i = 0; i < 4; ++i) words[i] |= ((pat >> i) & 1u) << b;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (i < bits) out[g * bits + i] = words[i];
}

}  // namespace bs

using namespace bs;

extern "C" size_t bs_packed_act_bytes(int N, int C, int H, int W, int a_bits)
{
    if (N <= 0 || C <= 0 || H <= 0 || W <= 0 || a_bits < 1 || a_bits > 4) return 0;
    return static_cast<size_t>(N) * H * W * ceil_div(C, 32) * a_bits * sizeof(uint32_t);
}

extern "C" size_t bs_packed_wgt_bytes(int O, int C, int R, int S, int w_bits)
{
    if (O <= 0 || C <= 0 || R <= 0 || S <= 0 || w_bits < 1 || w_bits > 4) return 0;
    return static_cast<size_t>(O) * R * S * ceil_div(C, 32) * w_bits * sizeof(uint32_t);
}

extern "C" size_t bs_packed_rows_bytes(int rows, int K, int bits)
{
    if (rows <= 0 || K <= 0 || bits < 1 || bits > 4) return 0;
    return static_cast<size_t>(rows) * ceil_div(K, 32) * bits * sizeof(uint32_t);
}

// Host copy of the Section IV quantiser (IEEE binary32 division, clip, round-half-even) used to derive the bounds.
static int host_quantize(float x, float s, int qmin, int qmax)
{
    volatile float t = x / s;
    float c = fminf(fmaxf(t, static_cast<float>(qmin)), static_cast<float>(qmax));
    return static_cast<int>(nearbyintf(c));
}

// Ordered integer key of a float (monotone in the float order) and back.
static uint32_t float_key(float f)
{
    uint32_t u;
    memcpy(&u, &f, 4);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
static float key_float(uint32_t k)
{
    uint32_t u = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
    float f;
    memcpy(&f, &u, 4);
    return f;
}

// Comparison-form quantiser for scale s: below[k] = the binary32 value just under bound[k], the smallest input whose code
// is >= qmin + k + 1 (bounds are never -inf: -inf always quantises to the lowest code; unreachable levels get +inf).
// bound[k], k = 0 .. 14: smallest binary32 input whose code is >= qmin + k + 1; +inf for levels that do not exist.
static void quantiser_bounds(float s, int bits, int sign, float (&bound)[15])
{
    int qmin, qmax;
    code_limits(bits, sign, qmin, qmax);
    for (int k = 0; k < 15; ++k) bound[k] = INFINITY;
    if (sign == BS_BIPOLAR) {                 // +1 iff x >= 0
        bound[0] = 0.0f;
        return;
    }
    const uint32_t lo_key = float_key(-INFINITY), hi_key = float_key(INFINITY);
    for (int k = 1; k <= qmax - qmin; ++k) {
        // smallest x (in float order) with code >= qmin + k; the code is monotone in x and reaches qmax at +inf
        uint32_t lo = lo_key, hi = hi_key;
        while (lo < hi) {
            const uint32_t mid = lo + (hi - lo) / 2;
            if (host_quantize(key_float(mid), s, qmin, qmax) >= qmin + k) hi = mid;
            else lo = mid + 1;
        }
        bound[k - 1] = key_float(lo);
    }
}

static QuantParams make_quant_params(float s, int bits, int sign)
{
    QuantParams q{};
    q.bits = bits; q.sign = sign;
    float bound[15];
    quantiser_bounds(s, bits, sign, bound);
    for (int k = 0; k < 15; ++k) {
        float p = bound[k] == 0.0f ? -1.401298464e-45f : key_float(float_key(bound[k]) - 1u);
        if (p == 0.0f) p = fabsf(p);          // drops the sign of a zero
        q.below[k] = p;
    }
    q.below[15] = INFINITY;
    // the estimate needs 1 / s and its products with the inputs near the bounds to be normal numbers
    q.estimate = bits >= 3 && s > 1e-30f && s < 1e30f;
    if (q.estimate) {
        int qmin, qmax;
        code_limits(bits, sign, qmin, qmax);
        for (int k = qmax - qmin; k < 16; ++k) q.below[k] = INFINITY;     // no level above the top one
        q.inv = 1.0f / s;
        q.offset = static_cast<float>(-qmin) - 0x1p-10f;
    }
    return q;
}

extern "C" int bs_quantiser_bounds(float act_scale, int a_bits, bs_sign_t a_sign, float* bounds_out)
{
    if (!bounds_out || !bits_ok(a_bits, a_sign) || !(act_scale > 0.0f && act_scale < 3.0e38f)) return BS_ERR_INVALID_ARG;
    float bound[15];
    quantiser_bounds(act_scale, a_bits, a_sign, bound);
    const int n = a_sign == BS_BIPOLAR ? 1 : (1 << a_bits) - 1;
    for (int k = 0; k < n; ++k) bounds_out[k] = bound[k];
    return BS_OK;
}

// NHWC codes of more channels than this start behind the kernel before, not beside its end.  Up to 128 channels the early start is
// faster at every size measured (14 x 14 pixels, 2 bits, back to back; 8 M codes of 64 channels: 6.1 -> 4.4 us a call, of 128: 7.1 -> 5.8;
// 0.5 M: 3.7 -> 3.5).  Above, most sizes gain as much (8 M of 256: 8.2 -> 6.2, of 384: 7.0 -> 6.0), but some lose, and not the same ones for
// neighbouring widths (8 M of 300: 6.2 -> 7.3; 4 M of 384: 6.2 -> 6.6, of 512: 6.2 -> 7.2): the line stands where none does.
constexpr int NHWC_DEPENDENT_C = 128;

template <int BITS>
static int launch_bitpack_nhwc_ragged(const int8_t* x, uint32_t* out, int N, int C, int HW, int bipolar, cudaStream_t st)
{
    const int Cw = ceil_div(C, 32);
    int pix = RAGGED_PIX;
    while (pix > 1 && static_cast<long long>(pix) * C > RAGGED_BYTES) pix /= 2;
    const long long npix = static_cast<long long>(N) * HW, blocks = ceil_div_ll(npix, pix);
    // the run of bytes, the part of a piece before it, and the nine words read from the last channel word on
    const long long smem = (static_cast<long long>(pix) * C + 15 + 15) / 16 * 16 + 64;
    if (blocks > 0x7fffffffLL || smem > 48 * 1024) return BS_ERR_UNSUPPORTED;
    auto kern = bitpack_nhwc_ragged_i8_kernel<BITS>;
    if (C <= NHWC_DEPENDENT_C)
        return launch_dependent(kern, dim3(static_cast<unsigned>(blocks)), dim3(FAST_THREADS), static_cast<size_t>(smem), st, x, out, C, Cw, npix, pix, bipolar);
    kern<<<static_cast<unsigned>(blocks), FAST_THREADS, static_cast<size_t>(smem), st>>>(x, out, C, Cw, npix, pix, bipolar);
    return cudaGetLastError() == cudaSuccess ? BS_OK : BS_ERR_CUDA;
}

template <typename P, typename... R> static P first_param(void (*)(P, R...));

// Launch of a kernel whose warps each take `pix_per_unit` pixels x one channel word.
template <bool DEPENDENT = true, typename K, typename... Extra>
static int launch_units(K kern, const void* x, uint32_t* out, int N, int C, int HW, int pix_per_unit, cudaStream_t st, Extra... extra)
{
    const int Cw = ceil_div(C, 32);
    const long long units_per_img = static_cast<long long>(ceil_div(HW, pix_per_unit)) * Cw;
    const long long nunits = N * units_per_img;
    const long long blocks = ceil_div_ll(nunits, FAST_WARPS);
    if (units_per_img > 0x7fffffffLL || blocks > 0x7fffffffLL) return BS_ERR_UNSUPPORTED;
    const auto in = static_cast<decltype(first_param(kern))>(x);
    if (DEPENDENT)
        return launch_dependent(kern, dim3(static_cast<unsigned>(blocks)), dim3(FAST_THREADS), 0, st, in, out, C, HW, Cw, nunits,
                                static_cast<int>(units_per_img), extra...);
    kern<<<static_cast<unsigned>(blocks), FAST_THREADS, 0, st>>>(in, out, C, HW, Cw, nunits, static_cast<int>(units_per_img), extra...);
    return cudaGetLastError() == cudaSuccess ? BS_OK : BS_ERR_CUDA;
}

template <int BITS>
static int launch_bitpack_nchw_i8(const void* x, uint32_t* out, int N, int C, int HW, int bipolar, cudaStream_t st)
{
    const long long bytes = static_cast<long long>(N) * C * HW;
    // a plain launch: with all its blocks begun at once this one takes 10 to 20 % longer (46 x 173 x 43 x 27: 6.7 -> 8.1 us)
    if (HW % 4 != 0) return launch_units<false>(bitpack_nchw_i8_kernel<BITS, 0, false>, x, out, N, C, HW, 128, st, bytes, bipolar);
    switch (ceil_div(C, 32)) {      // records of 1, 2 or 4 channel words leave through the block-staged stores
        case 1: return launch_units(bitpack_nchw_i8_kernel<BITS, 1, true>, x, out, N, C, HW, 128, st, bytes, bipolar);
        case 2: return launch_units(bitpack_nchw_i8_kernel<BITS, 2, true>, x, out, N, C, HW, 128, st, bytes, bipolar);
        case 4: return launch_units(bitpack_nchw_i8_kernel<BITS, 4, true>, x, out, N, C, HW, 128, st, bytes, bipolar);
        default: return launch_units(bitpack_nchw_i8_kernel<BITS, 0, true>, x, out, N, C, HW, 128, st, bytes, bipolar);
    }
}

// NHWC codes: 16-byte loads straight from the records where these are whole channel words (C a multiple of 32, the planes the
// low bits of the byte), staged through shared memory otherwise.
template <int BITS>
static int launch_bitpack_nhwc_i8(const void* x, uint32_t* out, int N, int C, int HW, int bipolar, cudaStream_t st)
{
    if (C % 32 == 0 && !bipolar)
        return C <= NHWC_DEPENDENT_C ? launch_units(bitpack_nhwc_i8_kernel<BITS>, x, out, N, C, HW, 128, st)
                                     : launch_units<false>(bitpack_nhwc_i8_kernel<BITS>, x, out, N, C, HW, 128, st);
    return launch_bitpack_nhwc_ragged<BITS>(static_cast<const int8_t*>(x), out, N, C, HW, bipolar, st);
}

template <bool NHWC>
static int launch_bitpack_i8(const void* x, uint32_t* out, int N, int C, int HW, int bits, int bipolar, cudaStream_t st)
{
    switch (bits) {
        case 1: return NHWC ? launch_bitpack_nhwc_i8<1>(x, out, N, C, HW, bipolar, st) : launch_bitpack_nchw_i8<1>(x, out, N, C, HW, bipolar, st);
        case 2: return NHWC ? launch_bitpack_nhwc_i8<2>(x, out, N, C, HW, bipolar, st) : launch_bitpack_nchw_i8<2>(x, out, N, C, HW, bipolar, st);
        case 3: return NHWC ? launch_bitpack_nhwc_i8<3>(x, out, N, C, HW, bipolar, st) : launch_bitpack_nchw_i8<3>(x, out, N, C, HW, bipolar, st);
        default: return NHWC ? launch_bitpack_nhwc_i8<4>(x, out, N, C, HW, bipolar, st) : launch_bitpack_nchw_i8<4>(x, out, N, C, HW, bipolar, st);
    }
}

// fp32 tensors: one (32 pixels, channel word) unit per warp.
template <int BITS, bool LEVELS>
static int launch_f32(bool nhwc, const void* x, uint32_t* out, int N, int C, int HW, const QuantParams& q, cudaStream_t st)
{
    return nhwc ? launch_units(bitpack_nhwc_f32_kernel<BITS, LEVELS>, x, out, N, C, HW, 32, st, q)
                : launch_units(bitpack_nchw_f32_kernel<BITS, LEVELS>, x, out, N, C, HW, 32, st, q, NoOper{});
}

static int launch_bitpack_f32(bool nhwc, const void* x, uint32_t* out, int N, int C, int HW, const QuantParams& q, cudaStream_t st)
{
    switch (q.bits) {
        case 1: return launch_f32<1, false>(nhwc, x, out, N, C, HW, q, st);
        case 2: return launch_f32<2, false>(nhwc, x, out, N, C, HW, q, st);
        case 3: return q.estimate ? launch_f32<3, true>(nhwc, x, out, N, C, HW, q, st) : launch_f32<3, false>(nhwc, x, out, N, C, HW, q, st);
        default: return q.estimate ? launch_f32<4, true>(nhwc, x, out, N, C, HW, q, st) : launch_f32<4, false>(nhwc, x, out, N, C, HW, q, st);
    }
}

// The bisection of the bounds takes several microseconds: a thread keeps the last one it made.
static const QuantParams& quant_params(float act_scale, int bits, int sign)
{
    static thread_local QuantParams q;
    static thread_local float q_scale = 0.0f;
    if (q_scale != act_scale || q.bits != bits || q.sign != sign) {
        q = make_quant_params(act_scale, bits, sign);
        q_scale = act_scale;
    }
    return q;
}

extern "C" int bitpack_activations_operands(const float* x, int N, int C, int H, int W, float act_scale, int a_bits, uint32_t* packed_out,
                                            const bs_operand_tensor* operands, void* stream)
{
    const OperTensor* o = reinterpret_cast<const OperTensor*>(operands);
    if (!o) return bitpack_activations(x, 1, BS_NCHW, N, C, H, W, act_scale, a_bits, BS_UNSIGNED, packed_out, stream);
    if (!x || !packed_out || packed_out != o->packed || N != o->N || C != o->Cw * 32 || H != o->H || W != o->W || a_bits != o->bits) return BS_ERR_INVALID_ARG;
    if (!(act_scale > 0.0f && act_scale < 3.0e38f)) return BS_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(packed_out)) return BS_ERR_ALIGNMENT;
    const QuantParams& q = quant_params(act_scale, a_bits, BS_UNSIGNED);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return a_bits == 1 ? launch_units(bitpack_nchw_f32_kernel<1, false, OperTensor>, x, packed_out, N, C, H * W, 32, st, q, *o)
                       : launch_units(bitpack_nchw_f32_kernel<2, false, OperTensor>, x, packed_out, N, C, H * W, 32, st, q, *o);
}

extern "C" int bitpack_activations(const void* x, int x_is_fp32, bs_layout_t layout, int N, int C, int H, int W,
                                   float act_scale, int a_bits, bs_sign_t a_sign, uint32_t* packed_out, void* stream)
{
    if (!x || !packed_out || N <= 0 || C <= 0 || H <= 0 || W <= 0) return BS_ERR_INVALID_ARG;
    if (!bits_ok(a_bits, a_sign) || (layout != BS_NCHW && layout != BS_NHWC)) return BS_ERR_INVALID_ARG;
    if (x_is_fp32 && !(act_scale > 0.0f && act_scale < 3.0e38f)) return BS_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(packed_out)) return BS_ERR_ALIGNMENT;
    if (static_cast<long long>(H) * W > 0x7fffffffLL) return BS_ERR_UNSUPPORTED;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int HW = H * W;
    if (x_is_fp32) return launch_bitpack_f32(layout == BS_NHWC, x, packed_out, N, C, HW, quant_params(act_scale, a_bits, a_sign), st);
    return layout == BS_NHWC ? launch_bitpack_i8<true>(x, packed_out, N, C, HW, a_bits, a_sign == BS_BIPOLAR, st)
                             : launch_bitpack_i8<false>(x, packed_out, N, C, HW, a_bits, a_sign == BS_BIPOLAR, st);
}

extern "C" int bitunpack_activations(const uint32_t* packed, int N, int C, int H, int W, int a_bits, bs_sign_t a_sign,
                                     bs_layout_t layout, int8_t* codes_out, void* stream)
{
    if (!packed || !codes_out || N <= 0 || C <= 0 || H <= 0 || W <= 0) return BS_ERR_INVALID_ARG;
    if (!bits_ok(a_bits, a_sign) || (layout != BS_NCHW && layout != BS_NHWC)) return BS_ERR_INVALID_ARG;
    if (!aligned16(packed) || !aligned16(codes_out)) return BS_ERR_ALIGNMENT;
    const long long total = static_cast<long long>(N) * C * H * W;
    const long long blocks = ceil_div_ll(total, 256);
    if (blocks > 0x7fffffffLL) return BS_ERR_UNSUPPORTED;
    bitunpack_kernel<<<static_cast<unsigned>(blocks), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        packed, codes_out, total, C, H * W, ceil_div(C, 32), a_bits, a_sign, layout == BS_NHWC);
    return cudaGetLastError() == cudaSuccess ? BS_OK : BS_ERR_CUDA;
}

static int launch_pack_weights(const int8_t* w, int ohwi, long long O, int C, int RS, int bits, int sign,
                               uint32_t* out, cudaStream_t st)
{
    const int Cw = ceil_div(C, 32);
    const long long ngroups = O * RS * Cw;
    const long long blocks = ceil_div_ll(ngroups, 128);
    if (blocks > 0x7fffffffLL) return BS_ERR_UNSUPPORTED;
    pack_weights_kernel<<<static_cast<unsigned>(blocks), 128, 0, st>>>(w, out, ngroups, C, RS, Cw, bits, sign, ohwi);
    return cudaGetLastError() == cudaSuccess ? BS_OK : BS_ERR_CUDA;
}

extern "C" int pack_weights(const int8_t* w_codes, bs_layout_t layout, int O, int C, int R, int S, int w_bits,
                            bs_sign_t w_sign, uint32_t* packed_out, void* stream)
{
    if (!w_codes || !packed_out || O <= 0 || C <= 0 || R <= 0 || S <= 0) return BS_ERR_INVALID_ARG;
    if (!bits_ok(w_bits, w_sign) || (layout != BS_NCHW && layout != BS_NHWC)) return BS_ERR_INVALID_ARG;
    if (!aligned16(w_codes) || !aligned16(packed_out)) return BS_ERR_ALIGNMENT;
    return launch_pack_weights(w_codes, layout == BS_NHWC, O, C, R * S, w_bits, w_sign, packed_out,
                               static_cast<cudaStream_t>(stream));
}

extern "C" int bs_pack_rows(const int8_t* codes, int rows, int K, int bits, bs_sign_t sign, uint32_t* packed_out,
                            void* stream)
{
    if (!codes || !packed_out || rows <= 0 || K <= 0) return BS_ERR_INVALID_ARG;
    if (!bits_ok(bits, sign)) return BS_ERR_INVALID_ARG;
    if (!aligned16(codes) || !aligned16(packed_out)) return BS_ERR_ALIGNMENT;
    return launch_pack_weights(codes, 1, rows, K, 1, bits, sign, packed_out, static_cast<cudaStream_t>(stream));
}
