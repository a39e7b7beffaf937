// The stem of a mixed-precision classifier in one kernel: 7 x 7 stride-2 convolution of three channels to 64, ReLU, 3 x 3 stride-2
// max pooling and the 2-bit quantiser, images in, packed codes out.  The codes are those of the separate layers (bs_conv2d_f32,
// bs_maxpool2d_f32, bitpack_activations) bit for bit, but few outputs need their float value:
//
//   A code asks only between which of three bounds a value lies, and pooling commutes with that (the largest value exceeds a bound if any
//   does).  So every output of the convolution is quantised first, and the pooled code is the largest of nine.  The quantiser's decision
//   comes from an integer convolution on the tensor cores: images and filters in fixed point with three signed digits of eight bits each
//   (x = sx X + dx, |X| <= 2^22), digit products in int32, exact.  What separates its result from the layer's chain of binary32
//   multiply-adds is bounded: |dx| and |dw|, the digit products left out, and the roundings of the chain, at most 148 * 2^-24 *
//   (|bias| + |patch|_2 |filter|_2) by Cauchy and Schwarz.  An output closer to a bound than the sum of these is undecided between two codes:
//   about 0.08 % of normalised images.  Most windows have another output that reaches the higher of the two for certain; in the others
//   the chain itself is evaluated, tap by tap in the layer's order.  A slab whose values have no useful common scale (infinities, NaN,
//   above 2^20) takes the chain for every output: right, but slower than the separate layers.  64 images of 224 x 224: 1500 us where every
//   slab is like that, 1650 where half of all outputs sit on a bound, 378 with one infinity an image, against 386 for the layers.
//
// What bounds it: 24 MMAs of 128 positions x (192, 128, 64) columns x 32 digits per tile, 1650 cycles alone, of which 1540 are
// shared-memory reads of the operands, so every other access to shared memory shows: 2080 cycles a tile in the steady state, and
// pooling with the chains keeps just up.  64 images of 224 x 224: 77 us a call (convolution, pooling and quantiser apart: 326 + 40 +
// 14, the convolution bound by the FP32 pipe: 203 at its full rate), 16 images 29, one 15.  On the way here, 64 images: bounds of each filter
// read from shared memory 107 us (an LDS.128 that all lanes share still takes four wavefronts: half as much shared-memory time as the
// MMAs), listed outputs by single lanes 126, by shuffles 107, all undecided outputs instead of those that matter 110.
//
// Layout.  The image is read as cells of 2 x 2 pixels x 3 channels, 12 of 16 bytes per digit, so the stride-2 window becomes 4 x 4 cells at
// stride 1 (its eighth row and column have zero weights).  Positions (conv row, column) are numbered linearly over cell rows of Q + 3
// cells; a tap is then a constant shift of the operand's start address.  A K = 32 step is two cells two rows apart.
// A CTA owns a run of pooled rows and walks it in slabs of five tiles of 128 positions:
//   7 producer warps   float cells -> scale of the slab -> digits
//   8 epilogue warps   digit sums -> codes and undecided outputs as bits of words, kept for the rows of a window
//   4 finish warps     pooling, the chain for undecided outputs, codes out; one slab behind the epilogue
//   1 MMA warp         24 MMAs a tile into one of two accumulators (high, middle and low digit sums of 64 filters)
#include <cmath>

#include "mma_kernel.cuh"

namespace bs {

constexpr int ST_TILES = 5, ST_SLAB = ST_TILES * 128;      // positions per slab
constexpr int ST_RING = 2048;                              // positions whose bits are kept: two slabs and three rows
constexpr int ST_CAP = 512;                                // undecided codes listed at a time
constexpr int ST_PW = 7, ST_EW = 8, ST_FW = 4;             // producer, epilogue, finish warps; the MMA warp comes last
constexpr int ST_THREADS = (ST_PW + ST_EW + ST_FW + 1) * 32;
constexpr int ST_CELLS_PER_THREAD = 5;
constexpr int ST_TAPS = 147, ST_B_HALF = 192 * 16 + 16, ST_B_BYTES = 8 * 2 * ST_B_HALF;      // 16 bytes more than its rows: cells of a filter lie in different banks
constexpr int ST_SMEM_MAX = 226 * 1024;

struct StemArgs {
    const float* x;
    const float* w;
    const float* bias;
    uint32_t* out;
    OperDst dst1, dst2;             // the codes as operand tensors of the layers that read them, or null
    int* status;
    int H, W, P, Q, P2, Q2;
    int share, extra;           // pooled rows of a CTA, CTAs with one more
    int pitch, plane;           // cells per cell row; bytes of one digit of a slab's cells
    FastDiv d_pitch, d_q2, d_p2;
    float below[3];             // a value reaches level k + 1 exactly when it exceeds below[k]
    double scale, third;        // of a code step; 1 / (3 * scale)
    int off_cells, off_ring, off_energy, off_slab, off_list, off_own, off_stat, off_bar;
};

// Largest values over the filters, what the bounds need (shared memory; bits of non-negative floats, which order like integers).
struct StemFilters {
    unsigned top, bias;                 // |weight|, |bias|; an infinity or a NaN shows here
    unsigned norm, fixed;               // |filter|_2; error of the fixed-point product in its own units
    int wide;                           // a filter whose low digit sum could leave the accumulators' range
    float scale, inv;                   // step of the weights, a power of two, and its reciprocal
    int fine;
};

// A CTA's run of pooled rows: segments within one image, each walked in slabs.
struct StemWalk {
    int g, g1, n, y0, ny, tiles, slabs, slab, count;      // count: slabs so far
    int ring;                                             // ring slot of the segment's position 0, not reduced
    __device__ __forceinline__ StemWalk(const StemArgs& a) : slab(0), count(0), ring(0)
    {
        const int b = static_cast<int>(blockIdx.x);
        g = b * a.share + min(b, a.extra);
        g1 = g + a.share + (b < a.extra);
        ny = 0;
        segment(a);
    }
    __device__ __forceinline__ void segment(const StemArgs& a)
    {
        if (g >= g1) return;
        n = fdiv(g, a.d_p2);
        y0 = g - n * a.P2;
        ny = min(a.P2 - y0, g1 - g);
        tiles = ((2 * ny + 1) * a.pitch + 127) >> 7;
        slabs = (tiles + ST_TILES - 1) / ST_TILES;
    }
    __device__ __forceinline__ bool live() const { return g < g1; }
    __device__ __forceinline__ int slab_tiles() const { return min(ST_TILES, tiles - slab * ST_TILES); }
    __device__ __forceinline__ void next(const StemArgs& a)
    {
        ++count;
        if (++slab < slabs) return;
        slab = 0;
        ring = (ring + slabs * ST_SLAB) & (ST_RING - 1);
        g += ny;
        segment(a);
    }
    __device__ __forceinline__ int buf() const { return count & 1; }
    __device__ __forceinline__ unsigned phase() const { return (count >> 1) & 1; }
};

__device__ __forceinline__ float4 st_lds(uint32_t addr)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void st_st8(uint32_t taddr, const uint32_t (&v)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]) : "memory");
}
// a * b + c of both halves, clamped to [0, 1]
__device__ __forceinline__ u64 st_fma_sat(u64 a, float b, float c)
{
    uint32_t a0, a1;
    f2_split(a, a0, a1);
    return f2_pack(__float_as_uint(__saturatef(fmaf(__uint_as_float(a0), b, c))), __float_as_uint(__saturatef(fmaf(__uint_as_float(a1), b, c))));
}
// x in steps, rounded to a whole number (|.| <= 2^22), as three signed digits of eight bits in the low bytes + 128 each.
__device__ __forceinline__ uint32_t st_fixed(float x, float inv) { return __float_as_uint(fmaf(x, inv, 12582912.0f)) + (0x00808080u - 0x4B400000u); }
// Four such numbers -> a word of their high, middle and low digits.
__device__ __forceinline__ void st_digits(const uint32_t (&t)[4], uint32_t& high, uint32_t& middle, uint32_t& low)
{
    const uint32_t l0 = __byte_perm(t[0], t[1], 0x5140), l1 = __byte_perm(t[2], t[3], 0x5140);
    const uint32_t h0 = __byte_perm(t[0], t[1], 0x0062), h1 = __byte_perm(t[2], t[3], 0x0062);
    low = __byte_perm(l0, l1, 0x5410) ^ 0x80808080u;
    middle = __byte_perm(l0, l1, 0x7632) ^ 0x80808080u;
    high = __byte_perm(h0, h1, 0x5410) ^ 0x80808080u;
}
__device__ __forceinline__ unsigned st_max(unsigned v) { return __reduce_max_sync(0xffffffffu, v); }

// The layer's chain for every undecided output of eight filters at positions m0 .. m1 of a segment, by a warp: bias first, taps by channel,
// row, column; taps outside the image multiply zero.  A lane takes two positions at a time, the filters' taps lie in shared memory
// (`own`, [tap][8]).  `words`: the ring's arrays of the filters' half, `byte`: their place in its words.
__device__ __forceinline__ void stem_chains(const StemArgs& a, const float* x_img, const float* w, const float* biases, float* own, unsigned char* words, int byte, int ring0,
                                         int y0, int m0, int m1, int lane)
{
    __syncwarp();
    for (int t = lane; t < ST_TAPS * 8; t += 32) own[t] = w[(t & 7) * ST_TAPS + (t >> 3)];
    __syncwarp();
    for (int base = m0; base < m1; base += 64) {
        unsigned und[2];
        int p[2], q[2], at[2];
        unsigned any = 0;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int m = base + j * 32 + lane, row = fdiv(m, a.d_pitch);
            q[j] = m - row * a.pitch;
            p[j] = 2 * y0 - 1 + row;
            at[j] = ((ring0 + m) & (ST_RING - 1)) * 4 + byte;
            und[j] = m < m1 && q[j] < a.Q && p[j] >= 0 && p[j] < a.P ? words[at[j] + 16 * ST_RING] : 0u;
            any |= und[j];
        }
        if (!__any_sync(0xffffffffu, any != 0)) continue;
        float acc[2][8];
#pragma unroll
        for (int f = 0; f < 8; ++f) {
            const float b = biases ? biases[f] : 0.0f;
#pragma unroll
            for (int j = 0; j < 2; ++j) acc[j][f] = b;
        }
        const float* tap = own;
#pragma unroll 1
        for (int k = 0; k < 21; ++k) {
            const int c = k / 7, r = k - 7 * c - 3;
            const float* src[2];
            bool row[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int y = 2 * p[j] + r;
                row[j] = und[j] && y >= 0 && y < a.H;
                src[j] = x_img + (static_cast<ptrdiff_t>(c) * a.H + (row[j] ? y : 0)) * a.W + 2 * q[j] - 3;
            }
#pragma unroll
            for (int s = 0; s < 7; ++s, tap += 8) {
                const float4 lo = *reinterpret_cast<const float4*>(tap), hi = *reinterpret_cast<const float4*>(tap + 4);
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const int x = 2 * q[j] - 3 + s;
                    const float v = row[j] && x >= 0 && x < a.W ? src[j][s] : 0.0f;
                    acc[j][0] = fmaf(v, lo.x, acc[j][0]); acc[j][1] = fmaf(v, lo.y, acc[j][1]); acc[j][2] = fmaf(v, lo.z, acc[j][2]); acc[j][3] = fmaf(v, lo.w, acc[j][3]);
                    acc[j][4] = fmaf(v, hi.x, acc[j][4]); acc[j][5] = fmaf(v, hi.y, acc[j][5]); acc[j][6] = fmaf(v, hi.z, acc[j][6]); acc[j][7] = fmaf(v, hi.w, acc[j][7]);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            unsigned b0 = 0, b1 = 0;
#pragma unroll
            for (int f = 0; f < 8; ++f) {
                const unsigned code = (acc[j][f] > a.below[0]) + (acc[j][f] > a.below[1]) + (acc[j][f] > a.below[2]);
                b0 |= (code & 1u) << f;
                b1 |= (code >> 1) << f;
            }
            if (und[j]) {
                words[at[j]] = static_cast<unsigned char>((words[at[j]] & ~und[j]) | (b0 & und[j]));
                words[at[j] + 8 * ST_RING] = static_cast<unsigned char>((words[at[j] + 8 * ST_RING] & ~und[j]) | (b1 & und[j]));
                words[at[j] + 16 * ST_RING] = 0;
            }
        }
    }
}

// One output's chain by eight lanes (l of them this one) through 296 floats of shared memory of their own: the operands come at once.  A lane that
// walks alone waits for memory seven times; handing operands round by shuffles took 4000 cycles.  Called by whole warps; live: there is a
// chain to walk.
__device__ __forceinline__ float stem_chain_eight(const float* x_img, const float* w, float acc, int H, int W, int p, int q, int l, bool live, float* own)
{
    const uint32_t dst = smem_u32(own);
    __syncwarp();
    if (live && l < 7) {
        // lane = column; rows follow one another in the image and in both operands
        const int x = 2 * q - 3 + l, y = 2 * p - 3;
        const bool xin = x >= 0 && x < W;
        uint32_t d = dst + static_cast<uint32_t>(l * 4);
        const float* from = w + l;
#pragma unroll 1
        for (int c = 0; c < 3; ++c) {
            const float* row = x_img + (static_cast<ptrdiff_t>(c) * H + y) * W + x;
#pragma unroll
            for (int r = 0; r < 7; ++r, d += 28, from += 7, row += W) {
                const bool in = xin && static_cast<unsigned>(y + r) < static_cast<unsigned>(H);
                mm_cp<4>(d, in ? row : x_img, in ? 4 : 0);
                mm_cp<4>(d + 148 * 4, from, 4);
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
#pragma unroll 6
    for (int k = 0; k < 36; ++k) {
        const float4 x = st_lds(dst + k * 16), u = st_lds(dst + 148 * 4 + k * 16);
        acc = fmaf(x.w, u.w, fmaf(x.z, u.z, fmaf(x.y, u.y, fmaf(x.x, u.x, acc))));
    }
    return fmaf(own[146], own[294], fmaf(own[145], own[293], fmaf(own[144], own[292], acc)));
}

// Filters -> digits in the B operand [K step][half][digit * 64 + filter][16], and what their bounds need.  One step for all filters, so that
// the epilogue needs no constants of a filter (read by every lane from shared memory they cost as much of its bandwidth as half the MMAs).
// The bias is the weight of 64 inputs of value one in the operand's padding.  The caller synchronises before and after.
// Sixteen lanes take a filter, a cell of the window each; the producers are at the first slab meanwhile.
__device__ __forceinline__ void stem_filters(const StemArgs& a, const float* wgt, const float* biases, unsigned char* smem, int t)
{
    constexpr int THREADS = ST_THREADS - ST_PW * 32, AT_ONCE = THREADS / 16, ROUNDS = (64 + AT_ONCE - 1) / AT_ONCE;
    StemFilters* all = reinterpret_cast<StemFilters*>(smem + a.off_stat);
    // cell (row, column) of the 4 x 4: the operand's K step takes rows 0 and 2 or 1 and 3 of a column
    const int l = t & 15, row = (l & 1) * 2 + (l >> 3), col = l >> 1 & 3;
    float v[ROUNDS][12], b[ROUNDS];
    unsigned top = 0, top_bias = 0;
#pragma unroll
    for (int i = 0; i < ROUNDS; ++i) {
        const int f = (t >> 4) + i * AT_ONCE;
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const int y = 2 * row + (k >> 1 & 1) - 1, x = 2 * col + (k & 1) - 1;
            v[i][k] = f < 64 && y >= 0 && x >= 0 ? wgt[f * ST_TAPS + (k >> 2) * 49 + y * 7 + x] : 0.0f;
        }
        b[i] = f < 64 && biases ? biases[f] : 0.0f;
    }
#pragma unroll
    for (int i = 0; i < ROUNDS; ++i) {
#pragma unroll
        for (int k = 0; k < 12; ++k) top = max(top, __float_as_uint(v[i][k]) & 0x7fffffffu);
        top_bias = max(top_bias, __float_as_uint(b[i]) & 0x7fffffffu);
    }
    top = st_max(top);
    top_bias = st_max(top_bias);
    if ((t & 31) == 0) { atomicMax(&all->top, top); atomicMax(&all->bias, top_bias); }
    asm volatile("bar.sync 3, %0;" ::"n"(THREADS) : "memory");
    const int e = static_cast<int>(all->top >> 23), eb = static_cast<int>(all->bias >> 23);      // biased exponents
    // |w| < 2^(e - 126) and |bias| / 64 < 2^(eb - 132): steps of 2^-22 of the larger
    const int es = max(all->top == 0 ? 100 : e, eb - 6);
    const bool fine = es > 67 && es < 187;
    const float scale = __uint_as_float(static_cast<unsigned>(fine ? es - 21 : 106) << 23), inv = __uint_as_float(static_cast<unsigned>(254 - (fine ? es - 21 : 106)) << 23);
    if (t == 0) { all->scale = scale; all->inv = inv; all->fine = fine; }
    float most_norm = 0.0f, most_fixed = 0.0f;
    bool wide = false;
#pragma unroll 1
    for (int f = t >> 4; f < AT_ONCE * ROUNDS; f += AT_ONCE) {           // the same number of rounds for every lane
        float sq = 0.0f;
        uint32_t d[3][4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            uint32_t n[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (c < 3) sq = fmaf(v[0][c < 3 ? 4 * c + k : 0], v[0][c < 3 ? 4 * c + k : 0], sq);
                n[k] = st_fixed(c < 3 ? v[0][c < 3 ? 4 * c + k : 0] : b[0], c < 3 ? inv : inv * 0.015625f);
            }
            st_digits(n, d[0][c], d[1][c], d[2][c]);
        }
        int squares[3] = {0, 0, 0};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (f < 64) mm_sts(smem_u32(smem) + static_cast<uint32_t>(l * ST_B_HALF + (k * 64 + f) * 16), d[k][0], d[k][1], d[k][2], d[k][3]);
#pragma unroll
            for (int c = 0; c < 4; ++c) squares[k] = __dp4a(static_cast<int>(d[k][c]), static_cast<int>(d[k][c]), squares[k]);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
#pragma unroll
            for (int k = 0; k < 3; ++k) squares[k] += __shfl_xor_sync(0xffffffffu, squares[k], o);
            sq += __shfl_xor_sync(0xffffffffu, sq, o);
        }
        const float norm = sqrtf(sq) * 1.001f;
        most_norm = fmaxf(most_norm, norm);
        // sums of |digit| over the 211 places by Cauchy and Schwarz
        const float m0 = sqrtf(211.0f * static_cast<float>(squares[2])) * 1.001f, m1 = sqrtf(211.0f * static_cast<float>(squares[1])) * 1.001f,
                    m2 = sqrtf(211.0f * static_cast<float>(squares[0])) * 1.001f;
        // the accumulators are read as floats (2^22); the high and the middle sum cannot leave that range: 211 * 64 * 64, 2 * 211 * 64 * 128
        wide |= 64.0f * m0 + 128.0f * m1 + 128.0f * m2 > 4100000.0f;
        // |dx| <= 1/2 against sum |W| <= 12.2 (|filter|_2 / scale + 6.1), |dw| <= 1/2 against |X| <= 2^22, and the digit products left out, over 2^16
        most_fixed = fmaxf(most_fixed, (6.1f * (norm * inv + 6.1f) + 0.5f * (ST_TAPS + 64) * 4194304.0f + 32768.0f * (m0 + m1) + 128.0f * m0) * (1.001f / 65536.0f));
        // rolled: the registers move up instead
#pragma unroll
        for (int i = 0; i + 1 < ROUNDS; ++i) {
#pragma unroll
            for (int k = 0; k < 12; ++k) v[i][k] = v[i + 1][k];
            b[i] = b[i + 1];
        }
    }
    most_norm = __uint_as_float(st_max(__float_as_uint(most_norm)));
    most_fixed = __uint_as_float(st_max(__float_as_uint(most_fixed)));
    if ((t & 31) == 0) {
        atomicMax(&all->norm, __float_as_uint(most_norm));
        atomicMax(&all->fixed, __float_as_uint(most_fixed));
    }
    if (wide) atomicOr(&all->wide, 1);
    fence_proxy_async();
}

struct StemSlab { float mul, off, lim; unsigned coarse; };

// What turns the digit sums of a slab into a third of the code, less the error, and what rounding may take off where the code is certain.
__device__ __forceinline__ StemSlab stem_bounds(const StemArgs& a, const StemFilters& q, float sx, float patch)
{
    // one unit of the sum 65536 D0 + 256 D1 + D2 is sx * scale * 2^16, powers of two: the reciprocal by the exponents
    const double u = static_cast<double>(sx) * q.scale * 65536.0;
    const double iu = static_cast<double>(__uint_as_float((254u << 23) - __float_as_uint(sx))) * q.inv * (1.0 / 65536.0);
    const double eps = 5.9604644775390625e-08;             // 2^-24
    // chain of 147 fused multiply-adds (148 with slack for the higher-order terms): 148 eps (|bias| + |patch| |w|)
    const double chain = 148.0 * 1.001 * eps * (__uint_as_float(q.bias) + static_cast<double>(patch) * __uint_as_float(q.norm)) * iu;
    // The epilogue's binary32: sums of floats near 12582912 * 257 (an ulp is 256), the constant that takes this off again, the multiplier
    const double offset = 12582912.0 * 257.0, arith = 130.0 + eps * (2.0 * offset + 9.0 * a.scale * iu);
    const float mul = static_cast<float>(u * a.third);
    // in codes; the rest covers the bounds' distance from whole codes + 1/2 (an ulp) and the roundings below
    const double dist = (chain + __uint_as_float(q.fixed) + arith + 4.0) * 1.01 * u * (3.0 * a.third) + 4e-6;
    const bool ok = q.fine && !q.wide && dist < 0.49 && mul > 1e-30f && mul < 1e20f;
    return StemSlab{mul, static_cast<float>(-offset * mul - dist * (1.0 / 3.0)), static_cast<float>(0.5 - 2.0 * dist), ok ? 0u : 0xffffffffu};
}

__global__ void __launch_bounds__(ST_THREADS, 1) stem_codes_kernel(const __grid_constant__ StemArgs a)
{
    extern __shared__ __align__(1024) unsigned char st_smem[];
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const uint32_t smem0 = smem_u32(st_smem);
    uint64_t* bars = reinterpret_cast<uint64_t*>(st_smem + a.off_bar);
    uint64_t* full_cells = bars;            // [2] digits and constants of a slab
    uint64_t* empty_cells = bars + 2;       // [2] its MMAs are done
    uint64_t* empty_slab = bars + 4;        // [2] ... and the epilogue is done with its constants
    uint64_t* slab_done = bars + 6;         // [2] bits of a slab written
    uint64_t* fin_done = bars + 8;          // [2] ... and pooled
    uint64_t* full_acc = bars + 10;         // [2]
    uint64_t* empty_acc = bars + 12;        // [2]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 14);
    unsigned* count = reinterpret_cast<unsigned*>(bars + 15);           // listed codes
    unsigned* coarse = reinterpret_cast<unsigned*>(bars + 30);          // [2] a slab is undecided as a whole
    unsigned* red = reinterpret_cast<unsigned*>(bars + 16);             // [2][2][ST_PW]
    StemSlab* slabs = reinterpret_cast<StemSlab*>(st_smem + a.off_slab);     // [2]
    uint32_t* ring = reinterpret_cast<uint32_t*>(st_smem + a.off_ring);    // [code bit 0, code bit 1, undecided][half][ST_RING]

    if (tid == 0) {
        for (int s = 0; s < 2; ++s) {
            mbar_init(&full_cells[s], ST_PW); mbar_init(&empty_cells[s], 1); mbar_init(&empty_slab[s], ST_EW);
            mbar_init(&slab_done[s], ST_EW); mbar_init(&fin_done[s], ST_FW);
            mbar_init(&full_acc[s], 1); mbar_init(&empty_acc[s], ST_EW);
        }
        *count = 0;
        *reinterpret_cast<StemFilters*>(st_smem + a.off_stat) = StemFilters{};
        fence_barrier_init();
        fence_proxy_async();
    }
    constexpr int WARP_MMA = ST_PW + ST_EW + ST_FW;
    if (warp == WARP_MMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    mm_fence_before();
    __syncthreads();                    // the tensor memory is ours before the next launch may begin
    mm_fence_after();
    const float* xs = dependent_begin(a.x);
    const float* ws = a.w;
    const float* biases = a.bias;
    asm volatile("" : "+l"(ws), "+l"(biases)::"memory");        // read behind the wait, like the images
    if (warp >= ST_PW) {
        stem_filters(a, ws, biases, st_smem, tid - ST_PW * 32);
        __syncthreads();
    }
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    bool ok = true;

    if (warp < ST_PW) {
        // ------------------------------------------------------------------ producers
        for (StemWalk w(a); w.live(); w.next(a)) {
            const int b = w.buf(), cells = w.slab_tiles() * 128 + 3 * a.pitch + 3, base = w.slab * ST_SLAB;
            float* energy = reinterpret_cast<float*>(st_smem + a.off_energy);
            float2 v[ST_CELLS_PER_THREAD][6];
            float top = 0.0f;
#pragma unroll
            for (int i = 0; i < ST_CELLS_PER_THREAD; ++i) {
                const int c = tid + i * ST_PW * 32;
                const int crow = fdiv(base + c, a.d_pitch), ccol = base + c - crow * a.pitch;
                const int y = 2 * (2 * w.y0 - 3 + crow), x = 2 * (ccol - 2);
                const bool xin = c < cells && x >= 0 && x < a.W;
                const float* src = xs + (static_cast<ptrdiff_t>(w.n) * 3 * a.H + y) * a.W + x;
#pragma unroll
                for (int ch = 0; ch < 3; ++ch)
#pragma unroll
                    for (int dy = 0; dy < 2; ++dy) {
                        const bool in = xin && y + dy >= 0 && y + dy < a.H;
                        v[i][ch * 2 + dy] = in ? *reinterpret_cast<const float2*>(src + (static_cast<ptrdiff_t>(ch) * a.H + dy) * a.W) : make_float2(0.0f, 0.0f);
                    }
            }
#pragma unroll
            for (int i = 0; i < ST_CELLS_PER_THREAD; ++i) {
                const int c = tid + i * ST_PW * 32;
                float e = 0.0f;
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    top = fmaxf(top, fmaxf(fabsf(v[i][k].x), fabsf(v[i][k].y)));
                    e = fmaf(v[i][k].y, v[i][k].y, fmaf(v[i][k].x, v[i][k].x, e));
                }
                if (c < cells) energy[c] = e;
            }
            const unsigned wtop = st_max(__float_as_uint(top));
            if (lane == 0) red[b * 2 * ST_PW + warp] = wtop;
            asm volatile("bar.sync 1, %0;" ::"n"(ST_PW * 32) : "memory");
            // largest energy of a 4 x 4 window of cells, 29 windows a warp; an infinity or a NaN among the cells shows in its bits
            unsigned most = 0;
            for (int m = warp * 29 + lane; m - lane < w.slab_tiles() * 128; m += ST_PW * 29) {
                float e = 0.0f;
#pragma unroll
                for (int r = 0; r < 4; ++r) e += m + r * a.pitch < cells ? energy[m + r * a.pitch] : 0.0f;
                e += __shfl_down_sync(0xffffffffu, e, 1);
                e += __shfl_down_sync(0xffffffffu, e, 2);
                if (lane < 29) most = max(most, __float_as_uint(e));
            }
            most = st_max(most);
            if (lane == 0) red[(b * 2 + 1) * ST_PW + warp] = most;
            asm volatile("bar.sync 1, %0;" ::"n"(ST_PW * 32) : "memory");
            unsigned tops = 0, mosts = 0;
#pragma unroll
            for (int k = 0; k < ST_PW; ++k) {
                tops = max(tops, red[b * 2 * ST_PW + k]);
                mosts = max(mosts, red[(b * 2 + 1) * ST_PW + k]);
            }
            // |x| < 2^(es - 126): steps of 2^(es - 126 - 22); the value one has to be among them
            const int e = static_cast<int>(tops >> 23);
            const bool fine = e < 147 && mosts < 0x7f000000u;
            const int es = fine ? max(e, 126) : 126;
            const float inv = fine ? __uint_as_float(static_cast<unsigned>(254 - (es - 21)) << 23) : 0.0f;
            if (w.count == 0) __syncthreads();          // the filters are there
            if (ok) ok = mm_wait(&empty_slab[b], w.phase() ^ 1u);
            if (tid == 0) {
                StemSlab q = stem_bounds(a, *reinterpret_cast<const StemFilters*>(st_smem + a.off_stat), __uint_as_float(static_cast<unsigned>(es - 21) << 23),
                                         sqrtf(__uint_as_float(fine ? mosts : 0u)) * 1.001f);
                if (!fine) q.coarse = 0xffffffffu;
                slabs[b] = q;
            }
            if (ok) ok = mm_wait(&empty_cells[b], w.phase() ^ 1u);
            const uint32_t dst = smem0 + a.off_cells + static_cast<uint32_t>(b * 3 * a.plane);
            // the value one in the padding
            const uint32_t one = static_cast<uint32_t>(static_cast<int>(inv) + 0x00808080) ^ 0x00808080u;
            const uint32_t pad[3] = {(one >> 16 & 255u) * 0x01010101u, (one >> 8 & 255u) * 0x01010101u, (one & 255u) * 0x01010101u};
#pragma unroll
            for (int i = 0; i < ST_CELLS_PER_THREAD; ++i) {
                const int c = tid + i * ST_PW * 32;
                uint32_t d[3][3];
#pragma unroll
                for (int ch = 0; ch < 3; ++ch) {
                    const float2 p = v[i][ch * 2], q = v[i][ch * 2 + 1];
                    const uint32_t t[4] = {st_fixed(p.x, inv), st_fixed(p.y, inv), st_fixed(q.x, inv), st_fixed(q.y, inv)};
                    st_digits(t, d[0][ch], d[1][ch], d[2][ch]);
                }
                if (c < cells)
#pragma unroll
                    for (int k = 0; k < 3; ++k) mm_sts(dst + static_cast<uint32_t>(k * a.plane + c * 16), d[k][0], d[k][1], d[k][2], pad[k]);
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mm_arrive(&full_cells[b]);
        }
    } else if (warp < ST_PW + ST_EW) {
        // ------------------------------------------------------------------ epilogue
        const int ew = warp - ST_PW, quad = warp & 3, half = ew >> 2;
        const uint32_t acc0 = tmem + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(half * 32);
        uint32_t preset[8];                 // in registers of their own: eight constants would be moved into place before every store
#pragma unroll
        for (int k = 0; k < 8; ++k) { preset[k] = MM_PRESET; asm volatile("" : "+r"(preset[k])); }
#pragma unroll 1
        for (int k = 0; k < 24; ++k) st_st8(acc0 + static_cast<uint32_t>(k / 12 * 256 + k % 12 / 4 * 64 + k % 4 * 8), preset);
        mm_st_wait();
        mm_fence_before();
        __syncwarp();
        if (lane == 0) { mm_arrive(&empty_acc[0]); mm_arrive(&empty_acc[1]); }
        // The accumulators are the floats 12582912 + sum.  (256 D1 + D2) + 65536 D0, in steps of the slab and clamped to [0, 1], is a third of
        // the code before rounding, less the error: adding 1.5 * 2^23 leaves the least code it can be in the low bits, sixteen of which one
        // shifted addition each collects in a word; where rounding took off most of a half, the code may be one more.
        const u64 k256 = f2_pack(0x43800000u, 0x43800000u), k65536 = f2_pack(0x47800000u, 0x47800000u), off0 = f2_pack(0xD3400000u, 0xD3400000u), three = f2_pack(0x40400000u, 0x40400000u);
        const u64 magic = f2_pack(preset[0], preset[1]), unmagic = f2_pack(0xCB400000u, 0xCB400000u), minus3 = f2_pack(0xC0400000u, 0xC0400000u);
        uint32_t collected = 0;             // what sixteen times 1.5 * 2^23 adds up to
#pragma unroll
        for (int k = 0; k < 16; ++k) collected = collected * 4u + MM_PRESET;
        int ia = 0;
        unsigned pa = 0;
        for (StemWalk w(a); w.live(); w.next(a)) {
            const int b = w.buf();
            if (ok) ok = mm_wait(&full_cells[b], w.phase());          // the bounds are there
            if (ok) ok = mm_wait(&fin_done[b], w.phase() ^ 1u);       // the ring is free
            const float mul = slabs[b].mul, off = slabs[b].off;
            const uint32_t whole = slabs[b].coarse;
            if (ew == 0 && lane == 0) coarse[b] = whole;
            const u64 lim = f2_pack(__float_as_uint(slabs[b].lim), __float_as_uint(slabs[b].lim));
            const int tiles = w.slab_tiles();
            uint32_t* dst = ring + half * ST_RING;
            for (int t = 0; t < tiles; ++t) {
                if (ok) ok = mm_wait(&full_acc[ia], pa);
                mm_fence_after();
                uint32_t even = 0, odds = 0, und = 0;
                const uint32_t acc = acc0 + static_cast<uint32_t>(ia * 256);
                // eight filters at a time, the sums of the next eight on their way
                uint32_t D[2][3][8];
#pragma unroll
                for (int d = 0; d < 3; ++d) mm_ld8(acc + d * 64 + 24, D[0][d]);
#pragma unroll 1
                for (int pair = 1; pair >= 0; --pair)
#pragma unroll
                for (int odd = 1; odd >= 0; --odd) {
                    const int piece = pair * 2 + odd;
                    uint32_t (&E)[3][8] = D[odd ^ 1];
                    mm_ld_wait();
                    mm_landed(E[0]); mm_landed(E[1]); mm_landed(E[2]);
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        if (odd || pair) mm_ld8(acc + d * 64 + (piece - 1) * 8, D[odd][d]);
                        st_st8(acc + d * 64 + piece * 8, preset);
                    }
                    if (!odd && !pair) {            // all is in registers: the next tile's MMAs may begin
                        mm_st_wait();
                        mm_fence_before();
                        __syncwarp();
                        if (lane == 0) mm_arrive(&empty_acc[ia]);
                        if (++ia == 2) { ia = 0; pa ^= 1u; }
                    }
#pragma unroll
                    for (int j = 3; j >= 0; --j) {
                        const u64 high = f2_fma(f2_pack(E[0][2 * j], E[0][2 * j + 1]), k65536, off0);
                        const u64 sum = f2_add(high, f2_fma(f2_pack(E[1][2 * j], E[1][2 * j + 1]), k256, f2_pack(E[2][2 * j], E[2][2 * j + 1])));
                        const u64 z = st_fma_sat(sum, mul, off);
                        const u64 code = f2_fma(z, three, magic);
                        uint32_t x, y, ux, uy;
                        f2_split(code, x, y);
                        f2_split(f2_fma(z, minus3, f2_add(f2_add(code, unmagic), lim)), ux, uy);          // negative: undecided
                        even = even * 4u + x;
                        odds = odds * 4u + y;
                        und = __funnelshift_l(uy, und, 1);
                        und = __funnelshift_l(ux, und, 1);
                    }
                }
                const int slot = (w.ring + w.slab * ST_SLAB + t * 128 + quad * 32 + lane) & (ST_RING - 1);
                und |= whole;
                even -= collected;
                odds -= collected;
                dst[slot] = ((even & 0x55555555u) | ((odds << 1) & 0xAAAAAAAAu)) & ~whole;
                dst[2 * ST_RING + slot] = (((even >> 1) & 0x55555555u) | (odds & 0xAAAAAAAAu)) & ~whole;
                dst[4 * ST_RING + slot] = und;
            }
            __syncwarp();
            if (lane == 0) { mm_arrive(&empty_slab[b]); mm_arrive(&slab_done[b]); }
        }
    } else if (warp < WARP_MMA) {
        // ------------------------------------------------------------------ finish
        const int ft = tid - (ST_PW + ST_EW) * 32;
        uint32_t* list = reinterpret_cast<uint32_t*>(st_smem + a.off_list);
        int done = 0;                          // pooled rows of the segment that are out
        for (StemWalk w(a); w.live(); w.next(a)) {
            const int b = w.buf();
            if (w.slab == 0) done = 0;
            if (ok) ok = mm_wait(&slab_done[b], w.phase());
            // pooled rows whose three conv rows are complete
            const int have = w.slab * ST_SLAB + w.slab_tiles() * 128;
            int ready = done;
            while (ready < w.ny && (2 * ready + 2) * a.pitch + a.Q <= have) ++ready;
            const float* image = xs + static_cast<size_t>(w.n) * 3 * a.H * a.W;
            uint32_t* out = a.out + (static_cast<size_t>(w.n) * a.P2 + w.y0) * a.Q2 * 4;
            const int i0 = done * a.Q2 * 2, i1 = ready * a.Q2 * 2;
            // the chain for every undecided output of positions m0 .. m1
            auto resolve = [&](int m0, int m1) {
                for (int octet = ft >> 5; octet < 8; octet += ST_FW)
                    stem_chains(a, image, ws + octet * 8 * ST_TAPS, biases ? biases + octet * 8 : nullptr, reinterpret_cast<float*>(st_smem + a.off_own) + (ft >> 5) * 1184,
                                reinterpret_cast<unsigned char*>(ring + (octet >> 2) * ST_RING), octet & 3, w.ring, w.y0, m0, m1, lane);
                asm volatile("bar.sync 2, %0;" ::"n"(ST_FW * 32) : "memory");
            };
            const bool whole = *reinterpret_cast<volatile unsigned*>(&coarse[b]) != 0;
            if (whole) resolve(w.slab * ST_SLAB, have);
            for (bool again = true; again;) {
                for (int i = i0 + ft; i < i1; i += ST_FW * 32) {
                    uint32_t o1 = 0, o2 = 0, o3 = 0, u0 = 0, u1 = 0, u2 = 0;         // codes of at least 1, 2, 3; undecided ones of at least 0, 1, 2
                    const uint32_t* src = ring + (i & 1) * ST_RING;
                    // rows and columns outside the image repeat the window's own
                    const int r = fdiv(i >> 1, a.d_q2), x = (i >> 1) - r * a.Q2, p0 = 2 * (w.y0 + r) - 1;
                    const int row1 = w.ring + (2 * r + 1) * a.pitch + 2 * x;
                    const int rows[3] = {p0 < 0 ? row1 : row1 - a.pitch, row1, p0 + 2 < a.P ? row1 + a.pitch : row1};
                    const int cols[3] = {x == 0 ? 0 : -1, 0, 2 * x + 1 < a.Q ? 1 : 0};
#pragma unroll
                    for (int dr = 0; dr < 3; ++dr)
#pragma unroll
                        for (int dc = 0; dc < 3; ++dc) {
                            const uint32_t* at = src + ((rows[dr] + cols[dc]) & (ST_RING - 1));
                            const uint32_t b0 = at[0], b1 = at[2 * ST_RING];
                            const uint32_t und = at[4 * ST_RING];
                            o1 |= b0 | b1; o2 |= b1; o3 |= b0 & b1;
                            u0 |= und & ~(b0 | b1); u1 |= und & b0; u2 |= und & b1 & ~b0;
                        }
                    // an undecided output matters where none is certain to reach the code it may have
                    uint32_t und = (u0 & ~o1) | (u1 & ~o2) | (u2 & ~o3);
                    const uint32_t c0 = ((o1 & ~o2) | o3) & ~und, c1 = o2 & ~und;
                    *reinterpret_cast<uint2*>(out + i * 2) = make_uint2(c0, c1);
                    if (a.dst1.base || a.dst2.base) {
                        uint32_t even, odd;
                        oper_pairs(c0, c1, even, odd);
                        oper_put(a.dst1, a.dst2, i & 1, oper_at1(a.dst1, w.n, w.y0 + r, x), oper_at2(a.dst2, w.n, w.y0 + r, x), even, odd);
                    }
                    while (und) {
                        const unsigned f = static_cast<unsigned>(__ffs(und)) - 1;
                        und &= und - 1;
                        if (*reinterpret_cast<volatile unsigned*>(count) > ST_CAP) break;
                        const unsigned at = atomicAdd(count, 1u);
                        if (at < ST_CAP) list[at] = static_cast<uint32_t>(i) << 5 | f;
                    }
                }
                asm volatile("bar.sync 2, %0;" ::"n"(ST_FW * 32) : "memory");
                const unsigned n = *reinterpret_cast<volatile unsigned*>(count);
                asm volatile("bar.sync 2, %0;" ::"n"(ST_FW * 32) : "memory");
                if (ft == 0) *count = 0;
                again = n > ST_CAP;
                if (!again) {
                    // eight lanes per code: the chain of every undecided output of its window
                    const int l = lane & 7;
                    float* own = reinterpret_cast<float*>(st_smem + a.off_own) + (ft >> 3) * 296;
                    for (unsigned k0 = ft >> 5 << 2; k0 < n; k0 += ST_FW * 4) {
                        const unsigned k = k0 + (lane >> 3);
                        const uint32_t entry = k < n ? list[k] : 0u;
                        const int i = static_cast<int>(entry >> 5), f = static_cast<int>(entry & 31u), filter = (i & 1) * 32 + f;
                        const int r = fdiv(i >> 1, a.d_q2), p0 = 2 * (w.y0 + r) - 1, q0 = 2 * ((i >> 1) - r * a.Q2) - 1;
                        const uint32_t* src = ring + (i & 1) * ST_RING;
                        const float bias = biases ? biases[filter] : 0.0f;
                        uint32_t codes = 0, members = 0;              // two bits a position
#pragma unroll
                        for (int m = 0; m < 9; ++m) {
                            const int p = p0 + m / 3, q = q0 + m % 3;
                            const uint32_t* at = src + ((w.ring + (2 * r + m / 3) * a.pitch + q) & (ST_RING - 1));
                            if (k < n && p >= 0 && p < a.P && q >= 0 && q < a.Q) {
                                codes |= ((at[0] >> f & 1u) | (at[2 * ST_RING] >> f & 1u) << 1) << (2 * m);
                                members |= (at[4 * ST_RING] >> f & 1u) << m;
                            }
                        }
                        uint32_t top = 0;
#pragma unroll
                        for (int m = 0; m < 9; ++m) top = max(top, codes >> (2 * m) & 3u);
#pragma unroll
                        for (int m = 0; m < 9; ++m)
                            if ((codes >> (2 * m) & 3u) != top) members &= ~(1u << m);
                        const float below = top == 0 ? a.below[0] : top == 1 ? a.below[1] : a.below[2];
                        while (__any_sync(0xffffffffu, members != 0)) {
                            const bool live = members != 0;
                            const int m = live ? __ffs(members) - 1 : 0;
                            members &= members - 1;
                            const float v = stem_chain_eight(image, ws + filter * ST_TAPS, bias, a.H, a.W, p0 + m / 3, q0 + m % 3, l, live, own);
                            if (live && v > below) { ++top; members = 0; }
                        }
                        if (k < n && l < 2 && (top >> l & 1u)) {
                            atomicOr(out + i * 2 + l, 1u << f);
                            const int y = w.y0 + r, x = (i >> 1) - r * a.Q2;
                            const uint32_t bit = 1u << (4 * (f >> 2) + l);          // nibble f / 4 of word f % 4
                            if (a.dst1.base) atomicOr(oper_words(a.dst1, i & 1, oper_at1(a.dst1, w.n, y, x)) + (f & 3), bit);
                            if (a.dst2.base) atomicOr(oper_words(a.dst2, i & 1, oper_at2(a.dst2, w.n, y, x)) + (f & 3), bit);
                        }
                    }
                } else {
                    resolve(2 * done * a.pitch, 2 * ready * a.pitch + a.Q);         // too many for the list: all of these rows, then once more
                }
                asm volatile("bar.sync 2, %0;" ::"n"(ST_FW * 32) : "memory");
            }
            done = ready;
            __syncwarp();
            if (lane == 0) mm_arrive(&fin_done[b]);
        }
    } else {
        // ------------------------------------------------------------------ MMA issuer (all lanes in step)
        const uint32_t pitch = static_cast<uint32_t>(a.pitch), plane16 = static_cast<uint32_t>(a.plane) >> 4;
        const uint32_t a_hi = (128u >> 4) | (1u << 14), b_hi = (128u >> 4) | (1u << 14);
        const uint32_t a_lo = (2u * pitch) << 16, b_lo = static_cast<uint32_t>(ST_B_HALF >> 4) << 16;
        const uint32_t cells0 = (smem0 & 0x3FFFFu) + a.off_cells, b0 = (smem0 & 0x3FFFFu) >> 4;
        const uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | (static_cast<unsigned>(128 >> 4) << 24);
        const uint32_t i192 = idesc | (24u << 17), i128 = idesc | (16u << 17), i64 = idesc | (8u << 17);
        unsigned limit = 1u << 20;
        int ia = 0;
        unsigned pa = 0;
        for (StemWalk w(a); w.live(); w.next(a)) {
            const int b = __shfl_sync(0xffffffffu, w.buf(), 0), tiles = __shfl_sync(0xffffffffu, w.slab_tiles(), 0);
            mm_wait_uniform(&full_cells[b], w.phase(), limit);
            mm_fence_after();
            const uint32_t cells = (cells0 >> 4) + static_cast<uint32_t>(b * 3) * plane16;
            for (int t = 0; t < tiles; ++t) {
                mm_wait_uniform(&empty_acc[ia], pa, limit);
                mm_fence_after();
                const uint32_t d = tmem + static_cast<uint32_t>(ia * 256);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const uint32_t at = a_lo | (cells + static_cast<uint32_t>(t * 128) + (k >> 2) * pitch + (k & 3)), bt = b_lo | (b0 + static_cast<uint32_t>(k * 2 * (ST_B_HALF >> 4)));
                    mm_mma(d, at, a_hi, bt, b_hi, i192, 1u);
                    mm_mma(d + 64u, at + plane16, a_hi, bt, b_hi, i128, 1u);
                    mm_mma(d + 128u, at + 2u * plane16, a_hi, bt, b_hi, i64, 1u);
                }
                mm_commit(&full_acc[ia]);
                if (++ia == 2) { ia = 0; pa ^= 1u; }
            }
            mm_commit(&empty_cells[b]);
        }
        ok = limit != 1u;
        __syncwarp();
    }
    if (!ok && lane == 0) atomicOr(a.status, STATUS_TIMEOUT);
    mm_fence_before();
    __syncthreads();
    if (warp == WARP_MMA) {
        mm_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

}  // namespace bs

namespace bs {

// What does not depend on the tensors: sizes, shared-memory layout, bounds.  `bytes`: dynamic shared memory.
static int stem_plan(StemArgs& g, int& bytes, int N, int C, int H, int W, int O, int R, int S, int stride, int pad, float act_scale, int a_bits)
{
    if (N <= 0 || C <= 0 || H <= 0 || W <= 0 || O <= 0 || R <= 0 || S <= 0 || stride < 1 || pad < 0) return BS_ERR_INVALID_ARG;
    if (H + 2 * pad < R || W + 2 * pad < S || !bits_ok(a_bits, BS_UNSIGNED) || !(act_scale > 0.0f && act_scale < 3.0e38f)) return BS_ERR_INVALID_ARG;
    if (C != 3 || O != 64 || R != 7 || S != 7 || stride != 2 || pad != 3 || a_bits != 2 || W % 2 != 0) return BS_ERR_UNSUPPORTED;
    g.H = H; g.W = W;
    g.P = (H - 1) / 2 + 1; g.Q = W / 2;
    g.P2 = (g.P - 1) / 2 + 1; g.Q2 = (g.Q - 1) / 2 + 1;
    g.pitch = g.Q + 3;
    const int cells = ST_SLAB + 3 * g.pitch + 3;
    // the cells a thread holds, and the rows of bits the ring holds beside two slabs
    if (cells > ST_CELLS_PER_THREAD * ST_PW * 32 || 2 * ST_SLAB + 2 * g.pitch + g.Q > ST_RING) return BS_ERR_UNSUPPORTED;
    if (static_cast<long long>(N) * g.P2 > 0x7fffffffLL || static_cast<long long>(2 * g.P2 + 2) * g.pitch > 0x3ffffffLL) return BS_ERR_UNSUPPORTED;
    g.d_pitch = make_div(g.pitch);
    g.d_q2 = make_div(g.Q2);
    g.d_p2 = make_div(g.P2);
    g.plane = (cells * 16 + 127) / 128 * 128;
    int off = ST_B_BYTES;
    g.off_cells = off;  off += 6 * g.plane;
    g.off_ring = off;   off += 6 * ST_RING * 4;
    g.off_energy = off; off += (cells * 4 + 15) / 16 * 16;
    g.off_slab = off;   off += 2 * static_cast<int>(sizeof(StemSlab));
    g.off_list = off;   off += ST_CAP * 4;
    g.off_own = off;    off += ST_FW * 4 * 296 * 4;
    g.off_stat = off;   off += (static_cast<int>(sizeof(StemFilters)) + 15) / 16 * 16;
    g.off_bar = off;    off += 512;
    if (off > ST_SMEM_MAX) return BS_ERR_UNSUPPORTED;
    bytes = off;
    float bound[15];
    if (const int rc = bs_quantiser_bounds(act_scale, a_bits, BS_UNSIGNED, bound)) return rc;
    for (int k = 0; k < 3; ++k) {
        g.below[k] = nextafterf(bound[k], -INFINITY);
        // ReLU leaves what exceeds a bound alone only when the bounds are positive
        if (!(g.below[k] >= 0.0f) || !std::isfinite(g.below[k])) return BS_ERR_UNSUPPORTED;
    }
    g.scale = act_scale;
    g.third = 1.0 / (3.0 * act_scale);
    return BS_OK;
}

}  // namespace bs

extern "C" int bs_stem_codes_supported(int N, int C, int H, int W, int O, int R, int S, int stride, int pad, float act_scale, int a_bits)
{
    bs::StemArgs g{};
    int bytes = 0;
    return bs::stem_plan(g, bytes, N, C, H, W, O, R, S, stride, pad, act_scale, a_bits) == BS_OK;
}

extern "C" int bs_stem_codes_f32(const float* x, const float* w, const float* bias, int N, int C, int H, int W, int O, int R, int S, int stride, int pad,
                                 float act_scale, int a_bits, uint32_t* out, void* stream)
{
    return bs_stem_codes_operands_f32(x, w, bias, N, C, H, W, O, R, S, stride, pad, act_scale, a_bits, out, nullptr, stream);
}

extern "C" int bs_stem_codes_operands_f32(const float* x, const float* w, const float* bias, int N, int C, int H, int W, int O, int R, int S, int stride, int pad,
                                          float act_scale, int a_bits, uint32_t* out, const bs_operand_tensor* operands, void* stream)
{
    using namespace bs;
    if (!x || !w || !out) return BS_ERR_INVALID_ARG;
    StemArgs g{};
    int bytes = 0;
    const int rc = stem_plan(g, bytes, N, C, H, W, O, R, S, stride, pad, act_scale, a_bits);
    if (rc == BS_ERR_INVALID_ARG) return rc;
    if (!aligned16(x) || !aligned16(w) || !aligned16(out) || (bias && (reinterpret_cast<uintptr_t>(bias) & 3u))) return BS_ERR_ALIGNMENT;
    if (rc != BS_OK) return rc;
    if (const OperTensor* o = reinterpret_cast<const OperTensor*>(operands)) {
        if (out != o->packed || N != o->N || O != o->Cw * 32 || g.P2 != o->H || g.Q2 != o->W || a_bits != o->bits) return BS_ERR_INVALID_ARG;
        g.dst1 = o->dst1;
        g.dst2 = o->dst2;
    }
    g.x = x; g.w = w; g.bias = bias; g.out = out;
    g.status = status_device_ptr();
    const int sms = device_sm_count();
    if (!g.status || sms <= 0) return BS_ERR_CUDA;
    if (cudaFuncSetAttribute(stem_codes_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, ST_SMEM_MAX) != cudaSuccess) {
        cudaGetLastError();
        return BS_ERR_CUDA;
    }
    const long long rows = static_cast<long long>(N) * g.P2;
    const unsigned grid = static_cast<unsigned>(rows < sms ? rows : sms);
    g.share = static_cast<int>(rows / grid);
    g.extra = static_cast<int>(rows % grid);
    return launch_dependent(stem_codes_kernel, dim3(grid), dim3(ST_THREADS), static_cast<size_t>(bytes), static_cast<cudaStream_t>(stream), g);
}
