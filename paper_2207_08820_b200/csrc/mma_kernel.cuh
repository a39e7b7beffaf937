// Exact integer convolution of packed bitplanes on the tensor cores (tcgen05.mma kind::mxf4 and kind::i8, accumulators in tensor memory).
//
// The Section V plane-pair popcount sum equals the integer dot product of the unpacked codes, so the same whole numbers come out of a
// matrix product of the codes: as nibbles (codes of one and two bits on both sides, see below) or as int8.  Both operands stay
// bit-packed in memory (filters optionally as operand tiles prepared once) and are expanded on chip.  A CTA walks over work items =
// 128 * PT accumulator rows x TN filters:
//
//   expander warps   packed pixels -> nibbles or int8 in the K-major core-matrix layout [channel group][pixel][16 bytes]
//   one MMA warp     R*S taps x channel blocks of K = 64 nibbles or 32 int8; a tap is only another start address of the pixel operand
//   epilogue warps   accumulators -> requantised, re-packed codes or int32, overlapping the MMAs of the next item
//   one copy warp    prepared filters by bulk copies, once (resident) or chunk by chunk (streamed)
//
// Accumulator rows are numbered linearly over (image, strip, row, column) with the zero padding between the rows of a strip
// and between images as rows of their own.  A tap then shifts the row index by a constant, any 128 consecutive positions
// form a tile, and small or odd images waste W / (W + pad) instead of whole 16 x 8 blocks: 64 images of 28 x 28 make
// 421 tiles (512 with rectangular ones).  Wide images are cut into strips so that the halo of a tile stays short.
// Stride 2 keeps one such plane per parity of row and column.
//
// Codes of one and two bits on both sides run as tcgen05.mma kind::mxf4 (F4): two-bit codes are the small e2m1 floats 0, 0.5, 1, 1.5 with a
// sign, so a nibble holds the code (sign and magnitude), scale factors of 2 in both operands make the products whole numbers, and
// the sums stay exact in binary32 (below 2^22 by mma_nibbles; compared up to 3999744 in tests/test_gpu_nibbles.py).  A K = 64 step takes as long
// and reads as many bytes as a K = 32 step of kind::i8, so operands, filter traffic and MMA time are all half as large.
//
// Codes of three bits: signed ones, -4 .. 3, are halves as they are.  Of unsigned activations 5 and 7 are not, so the operand holds a - 4 (the top plane
// inverted; padding, whose code is 0, becomes -4 like every zero) and the epilogue adds four times the sum of a filter's codes, as many as the
// tile holds: sum (a - 4) w + 4 sum w = sum a w.  The sums are collected where resident packed filters are expanded; other plans of such
// layers are int8 (mma_conv.cu has the rules).  32 x 256 x 28 x 28, 256 filters, three bits both: 30.6 -> 22.9 us.
//
// Every wait on an mbarrier is bounded; a wait that runs out sets the device status word and the CTA drains.
#pragma once
#include "conv_kernel.cuh"
#include "mma_conv.h"
#include "oper_tensor.cuh"

namespace bs {

constexpr int MM_STAGES = 8;         // most stages of packed words in front of the expanders

struct MmaArgs {
    CUtensorMap tmA, tmB;           // flat tiles with aligned rows: packed pixels (words, rows), packed filters (words, filters)
    const uint32_t* act;
    const int8_t* wgt;              // prepared filters [C/32][filters, padded to 128][R*S][32 bytes] in core-matrix order (nibbles: C/64), or null
    const uint32_t* wgt_packed;     // packed filters [O][R*S][Cw][WB], used when wgt is null
    int32_t* out_i32;
    uint32_t* out_packed;
    const float* scale;
    const float* bias;
    const uint32_t* residual;
    int* status;
    float res_scale;
    int has_residual;
    int N, H, W, O, R, RS, P, Q, stride, Cw;
    int a_kind, w_kind;         // 0 unsigned, 1 two's complement, 2 bipolar
    int relu, out_bits, out_sign, out_cw_off, out_cw_total;
    int res_bits, res_sign, res_c_off, res_cw_total;
    int i32_nhwc;
    float acc_bound;                // largest possible |accumulator|
    // position numbering
    int flat;                       // positions are the pixels themselves (1x1, stride 1)
    int total;                      // positions in all
    FastDiv d_img, d_pitch, d_strips;       // positions of one (image, strip), positions of a row, strips
    int strip_q, xoff, hstart;      // outputs per strip row, plane column of position 0, halo start relative to the tile
    int HL, nplanes, NI;            // halo pixels per parity plane, parity planes, pixels expanded per item (HL * nplanes)
    int pitch, img_rows;            // positions per row, rows per (image, strip)
    int rmin, smin;                 // smallest row / column shift of a tap
    int pad;
    // tiling
    int TN, PT, units, nunits, nchunks;     // filters and row tiles per item, 64-channel units per chunk / in all
    int nse, nsb;                   // stages of the expanded ring; the same when filters are streamed through it, 0: filters resident
    int split, split_log;           // CTAs (a cluster) that share the chunks of an item
    int groups, nsp;                // expander groups (chunk n belongs to group n mod groups), stages of packed words in all
    int tiles_m, tiles_o;
    FastDiv d_rs;
    int tma;                        // rows of pixels (and of packed, streamed filters) arrive by TMA boxes
    int rowA, rowB, swzA, swzB;     // bytes of a box row, 16-byte pieces of a row - 1 (the swizzle of the box)
    int bulk_b;                     // resident packed filters: the tile is fetched with one bulk copy
    int psz, bpsz;                  // bytes per cp.async of pixels, of packed filters
    int nslots, bslots;             // (pixel, unit) and (filter row, unit) items per expander thread and chunk
    int e_bytes, b_bytes, stg_bytes, bstg_bytes;    // per stage
    int off_e, off_stg, off_bstg, off_pix, off_brow, off_tab, off_bar, off_out, off_red;
    int tmem_cols, nacc;
    int f4;                         // kind::mxf4: operands of nibbles, float accumulators
    int nblk, sf_col;               // K steps of all channels per tap; column of the scale factors
    int one_word;                   // a unit has one channel word (32 channels in all): the second half of a K step meets zero filters
    int preset;                     // the fast requantisation applies; integer accumulators then start at the bit pattern of 1.5 * 2^23 (see the epilogue)
    int epi;                        // which instantiation of the fast requantisation: odd ones read a residual and its multipliers
    int early_b;                    // filters may be read before the preceding kernel has finished
    int opad;
    unsigned idesc;
};

// ----------------------------------------------------------------------------- timeline trace (-DBS_TRACE builds only)
//
// Built with -DBS_TRACE, the first 148 CTAs of a launch record the SM cycle counter at the hand-offs between their roles;
// bs_tc_trace_read copies the table to the host.  Compiled out of the normal library.
enum { TR_START = 0, TR_SETUP, TR_PDL, TR_WGT, TR_XBEG, TR_XEND, TR_MBEG, TR_MEND, TR_EBEG, TR_EEND, TR_END, TR_XWAIT };
#ifdef BS_TRACE
constexpr int MM_TRACE_EVENTS = 12, MM_TRACE_SEQ = 48, MM_TRACE_CTAS = 148;
static __device__ long long g_mm_trace[MM_TRACE_CTAS * MM_TRACE_EVENTS * MM_TRACE_SEQ];
__device__ __forceinline__ void mm_trace(int ev, int seq)
{
    if (blockIdx.x < MM_TRACE_CTAS && seq < MM_TRACE_SEQ) g_mm_trace[(blockIdx.x * MM_TRACE_EVENTS + ev) * MM_TRACE_SEQ + seq] = clock64();
}
#define MM_TRACE(cond, ev, seq) do { if (cond) mm_trace(ev, seq); } while (0)
#else
#define MM_TRACE(cond, ev, seq) do { } while (0)
#endif

// ----------------------------------------------------------------------------- PTX wrappers

__device__ __forceinline__ void mm_arrive(uint64_t* bar) { asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory"); }
// Bounded wait: an attempt parks the thread for at most about 2 us, 2^20 attempts end after about two seconds.
__device__ __forceinline__ bool mm_wait(uint64_t* bar, unsigned parity)
{
    const uint32_t addr = smem_u32(bar);
    for (unsigned it = 0; it < (1u << 20); ++it) {
        unsigned ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok) : "r"(addr), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}
__device__ __forceinline__ void mm_pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void mm_pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void mm_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void mm_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// The MMA warp stays converged: its waits loop inside one asm statement and a wait that ran out is only recorded (later waits
// then poll once), so every branch the compiler sees is warp-uniform and descriptors live in uniform registers; the MMAs
// themselves go out under elect.sync.  Measured at M = 128, K = 32: 40 / 48 / 64 / 128 cycles per MMA for N = 32 / 64 / 128 /
// 256, which is the shared-memory read of both operands (128 B/clk) or the arithmetic; issued by a lone diverged thread or
// under an ordinary predicate the operands move through vector registers first: 53 - 134 cycles whatever N is.
__device__ __forceinline__ bool mm_elect()
{
    uint32_t r;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
    return r != 0;
}
__device__ __forceinline__ void mm_wait_uniform(uint64_t* bar, unsigned parity, unsigned& limit)
{
    unsigned left;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mov.u32 %0, %3;\n\t"
        "MM_WAIT:\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "@p bra MM_DONE;\n\t"
        "sub.u32 %0, %0, 1;\n\t"
        "setp.ne.u32 p, %0, 0;\n\t"
        "@p bra MM_WAIT;\n\t"
        "MM_DONE:\n\t}"
        : "=&r"(left) : "r"(smem_u32(bar)), "r"(parity), "r"(limit) : "memory");
    limit = left == 0 ? 1u : limit;
}
__device__ __forceinline__ void mm_commit(uint64_t* bar)
{
    if (mm_elect()) asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mm_mma(uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc, uint32_t acc)
{
    if (mm_elect())
        asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d), "l"((static_cast<uint64_t>(a_hi) << 32) | a_lo), "l"((static_cast<uint64_t>(b_hi) << 32) | b_lo), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void mm_mma4(uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc, uint32_t acc, uint32_t sf)
{
    if (mm_elect())
        asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%5], [%5], p;\n\t}"
        ::"r"(d), "l"((static_cast<uint64_t>(a_hi) << 32) | a_lo), "l"((static_cast<uint64_t>(b_hi) << 32) | b_lo), "r"(idesc), "r"(acc), "r"(sf) : "memory");
}
__device__ __forceinline__ void mm_ld32(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void mm_ld16(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void mm_ld8(uint32_t taddr, uint32_t (&v)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void mm_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// Values loaded from tensor memory may be touched only after the wait: arithmetic on them must not move above it.
__device__ __forceinline__ void mm_landed(uint32_t (&v)[8])
{
    asm volatile("" : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]));
}
__device__ __forceinline__ void mm_landed(uint32_t (&v)[16])
{
    asm volatile("" : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                      "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]));
}
__device__ __forceinline__ void mm_landed(uint32_t (&v)[32])
{
    mm_landed(*reinterpret_cast<uint32_t (*)[16]>(&v[0]));
    mm_landed(*reinterpret_cast<uint32_t (*)[16]>(&v[16]));
}
__device__ __forceinline__ void mm_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void mm_st8(uint32_t taddr, uint32_t x)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(taddr), "r"(x) : "memory");
}
__device__ __forceinline__ void mm_bulk(void* dst, const void* src, unsigned bytes, uint64_t* bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* tm, uint64_t* bar, int c0, int c1)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(tm)), "r"(smem_u32(bar)), "r"(c0), "r"(c1) : "memory");
}
template <int PSZ>
__device__ __forceinline__ void mm_cp(uint32_t dst, const void* src, int bytes)     // bytes of the PSZ that exist, the rest is zero
{
    if (PSZ == 16) asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
    else if (PSZ == 8) asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mm_sts(uint32_t dst, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void mm_st16(uint32_t taddr, const uint32_t* v)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
                 ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
                   "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}
__device__ __forceinline__ void mm_cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Shared-memory address `addr` of this CTA in the CTA of rank 0 of the cluster.
__device__ __forceinline__ uint32_t mm_leader(uint32_t addr)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
    return r;
}
// Bounded wait for arrivals of other CTAs of the cluster.
__device__ __forceinline__ bool mm_wait_cluster(uint64_t* bar, unsigned parity)
{
    const uint32_t addr = smem_u32(bar);
    for (unsigned it = 0; it < (1u << 20); ++it) {
        unsigned ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok) : "r"(addr), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}
typedef unsigned long long u64;
__device__ __forceinline__ u64 f2_pack(uint32_t lo, uint32_t hi) { u64 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi)); return r; }
__device__ __forceinline__ void f2_split(u64 v, uint32_t& lo, uint32_t& hi) { asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(v)); }
__device__ __forceinline__ u64 f2_add(u64 a, u64 b) { u64 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ u64 f2_fma(u64 a, u64 b, u64 c) { u64 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }

// ----------------------------------------------------------------------------- expansion: plane words -> int8 or nibbles

// 32 codes of NB planes -> 32 bytes, byte 4 m + k = channel 8 k + m: bytes are cut out of the words with a shift and a mask, no
// look-up (a 256-entry table in shared memory cost eight loads with bank conflicts per word).  Two planes are first merged
// into words of 2-bit fields (even and odd channels apart), four planes into words of nibbles.  NB = 2: 18 operations.
template <int NB>
__device__ __forceinline__ void expand_word(const uint32_t* p, int kind, uint32_t (&o)[8])
{
    if (NB == 1) {
#pragma unroll
        for (int m = 0; m < 8; ++m) o[m] = (p[0] >> m) & 0x01010101u;
        if (kind == 2) {
#pragma unroll
            for (int m = 0; m < 8; ++m) o[m] = ~(o[m] * 254u);
        }
    } else if (NB == 2) {
        const uint32_t e = (p[0] & 0x55555555u) | ((p[NB - 1] << 1) & 0xAAAAAAAAu);
        const uint32_t d = ((p[0] >> 1) & 0x55555555u) | (p[NB - 1] & 0xAAAAAAAAu);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            o[2 * m] = (e >> (2 * m)) & 0x03030303u;
            o[2 * m + 1] = (d >> (2 * m)) & 0x03030303u;
        }
    } else {
        const uint32_t p2 = p[NB >= 3 ? 2 : 0], p3 = NB == 4 ? p[NB - 1] : 0u, p1 = p[NB >= 2 ? 1 : 0];
        const uint32_t e = (p[0] & 0x55555555u) | ((p1 << 1) & 0xAAAAAAAAu), d = ((p[0] >> 1) & 0x55555555u) | (p1 & 0xAAAAAAAAu);
        const uint32_t f = (p2 & 0x55555555u) | ((p3 << 1) & 0xAAAAAAAAu), g = ((p2 >> 1) & 0x55555555u) | (p3 & 0xAAAAAAAAu);
        const uint32_t s[4] = {(e & 0x33333333u) | ((f << 2) & 0xCCCCCCCCu), (d & 0x33333333u) | ((g << 2) & 0xCCCCCCCCu),
                               ((e >> 2) & 0x33333333u) | (f & 0xCCCCCCCCu), ((d >> 2) & 0x33333333u) | (g & 0xCCCCCCCCu)};
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            o[m] = s[m] & 0x0F0F0F0Fu;
            o[m + 4] = (s[m] >> 4) & 0x0F0F0F0Fu;
        }
    }
    if (kind == 1) {
        // two's complement: 256 - 2^NB added to the bytes whose top plane is set (no carry leaves a byte)
        constexpr uint32_t top = 0x01010101u << (NB - 1);
        constexpr uint32_t mul = (256u - (1u << NB)) >> (NB - 1);
#pragma unroll
        for (int m = 0; m < 8; ++m) o[m] += (o[m] & top) * mul;
    }
}

// 32 codes of one to three planes -> 32 nibbles, nibble j of word m = channel 4 j + m, sign and magnitude (magnitude in halves).  NB = 2: 10
// operations, and half the bytes.
template <int NB>
__device__ __forceinline__ void expand_nibbles(const uint32_t* p, int kind, uint32_t (&o)[4])
{
    if (NB == 1) {
#pragma unroll
        for (int m = 0; m < 4; ++m) o[m] = (p[0] >> m) & 0x11111111u;
        if (kind == 1) {            // the only plane weighs -1
#pragma unroll
            for (int m = 0; m < 4; ++m) o[m] *= 9u;
        } else if (kind == 2) {
#pragma unroll
            for (int m = 0; m < 4; ++m) o[m] = 0x99999999u ^ (o[m] << 3);
        }
    } else if (NB == 3) {
        // two's complement, of unsigned codes less 4: sign and 4 - (the other two bits) where the top bit is set
        const uint32_t p1 = p[NB > 1 ? 1 : 0], s = kind == 0 ? ~p[NB - 1] : p[NB - 1];
        const uint32_t m1 = p1 ^ (p[0] & s), m2 = s & ~(p1 | p[0]);
        const uint32_t e = (p[0] & 0x55555555u) | ((m1 << 1) & 0xAAAAAAAAu), d = ((p[0] >> 1) & 0x55555555u) | (m1 & 0xAAAAAAAAu);
        const uint32_t f = (m2 & 0x55555555u) | ((s << 1) & 0xAAAAAAAAu), h = ((m2 >> 1) & 0x55555555u) | (s & 0xAAAAAAAAu);
        o[0] = (e & 0x33333333u) | ((f << 2) & 0xCCCCCCCCu); o[1] = (d & 0x33333333u) | ((h << 2) & 0xCCCCCCCCu);
        o[2] = ((e >> 2) & 0x33333333u) | (f & 0xCCCCCCCCu); o[3] = ((d >> 2) & 0x33333333u) | (h & 0xCCCCCCCCu);
    } else {
        const uint32_t p1 = p[NB > 1 ? 1 : 0];
        const uint32_t e = (p[0] & 0x55555555u) | ((p1 << 1) & 0xAAAAAAAAu), d = ((p[0] >> 1) & 0x55555555u) | (p1 & 0xAAAAAAAAu);
        o[0] = e & 0x33333333u; o[1] = d & 0x33333333u; o[2] = (e >> 2) & 0x33333333u; o[3] = (d >> 2) & 0x33333333u;
        if (kind == 1) {            // 2 -> -2, 3 -> -1
#pragma unroll
            for (int m = 0; m < 4; ++m) o[m] = ((o[m] << 2) & 0x88888888u) | (o[m] & 0x11111111u) | (o[m] & ~(o[m] << 1) & 0x22222222u);
        }
    }
}

// Two channel words (one 64-channel unit) of a staged row -> four 16-byte rows of the operand (two of nibbles), `g16` bytes apart.  one: the
// second word does not exist.
template <int NB, bool F4>
__device__ __forceinline__ void expand_unit(const uint32_t (&w)[2 * NB], int kind, uint32_t dst, uint32_t g16, bool one)
{
    if constexpr (F4) {
        uint32_t n[4];
        expand_nibbles<NB>(w, kind, n);
        mm_sts(dst, n[0], n[1], n[2], n[3]);
        if (one) return;
        expand_nibbles<NB>(w + NB, kind, n);
        mm_sts(dst + g16, n[0], n[1], n[2], n[3]);
        return;
    }
    uint32_t o[8];
    expand_word<NB>(w, kind, o);
    mm_sts(dst, o[0], o[1], o[2], o[3]);
    mm_sts(dst + g16, o[4], o[5], o[6], o[7]);
    expand_word<NB>(w + NB, kind, o);
    mm_sts(dst + 2 * g16, o[0], o[1], o[2], o[3]);
    mm_sts(dst + 3 * g16, o[4], o[5], o[6], o[7]);
}

// Staged pieces of one unit: piece k of a thread's slot sits `step` bytes after piece k - 1.
template <int NB>
__device__ __forceinline__ void load_unit(uint32_t src, uint32_t step, int psz, uint32_t (&w)[2 * NB], bool one = false)
{
    if (psz == 16 && (2 * NB) % 4 == 0) {
#pragma unroll
        for (int k = 0; k < 2 * NB / 4; ++k)
            if (!one || k < NB / 4)
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w[(4 * k) % (2 * NB)]), "=r"(w[(4 * k + 1) % (2 * NB)]), "=r"(w[(4 * k + 2) % (2 * NB)]),
                         "=r"(w[(4 * k + 3) % (2 * NB)]) : "r"(src + k * step));
    } else if (psz == 8) {
#pragma unroll
        for (int k = 0; k < NB; ++k)
            if (!one || 2 * k < NB) asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(w[2 * k]), "=r"(w[2 * k + 1]) : "r"(src + k * step));
    } else {
#pragma unroll
        for (int k = 0; k < 2 * NB; ++k)
            if (!one || k < NB) asm volatile("ld.shared.b32 %0, [%1];" : "=r"(w[k]) : "r"(src + k * step));
    }
}

// One unit of a box row: `off` bytes from the start of the stage (1024-byte aligned); the box swizzles the 16-byte pieces of its rows.
template <int NB>
__device__ __forceinline__ void load_row_unit(uint32_t stage, int off, int mask, uint32_t (&w)[2 * NB])
{
    const uint32_t o = static_cast<uint32_t>(off);
    const uint32_t x = static_cast<uint32_t>(mask);
    if (NB == 2 || NB == 4) {
#pragma unroll
        for (int k = 0; k < NB / 2; ++k) {
            const uint32_t a = o + 16u * k;
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w[(4 * k) % (2 * NB)]), "=r"(w[(4 * k + 1) % (2 * NB)]), "=r"(w[(4 * k + 2) % (2 * NB)]),
                         "=r"(w[(4 * k + 3) % (2 * NB)]) : "r"(stage + (a ^ (((a >> 7) & x) << 4))));
        }
    } else {
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            const uint32_t a = o + 8u * k;
            asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(w[2 * k]), "=r"(w[2 * k + 1]) : "r"(stage + (a ^ (((a >> 7) & x) << 4))));
        }
    }
}

// cp.async of one unit (two channel words, NB planes each) of a packed row; `left` words of it exist, the rest is zero.
template <int NB, int PSZ>
__device__ __forceinline__ void stage_unit_p(uint32_t dst, uint32_t step, const uint32_t* src, const uint32_t* safe, int left, bool one)
{
    constexpr int PW = PSZ / 4, NP = 2 * NB / PW > 0 ? 2 * NB / PW : 1;
    if (one) {                                  // one channel word: all of it, or none
#pragma unroll
        for (int k = 0; k < (NP + 1) / 2; ++k) mm_cp<PSZ>(dst + k * step, src + k * PW, left > 0 ? PSZ : 0);
        return;
    }
    if (left >= 2 * NB || left <= 0) {          // all of it, or none
        const int bytes = left > 0 ? PSZ : 0;
#pragma unroll
        for (int k = 0; k < NP; ++k) mm_cp<PSZ>(dst + k * step, src + k * PW, bytes);
        return;
    }
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const int words = max(0, min(left - k * PW, PW));
        mm_cp<PSZ>(dst + k * step, words > 0 ? src + k * PW : safe, words * 4);
    }
}
template <int NB>
__device__ __forceinline__ void stage_unit(int psz, uint32_t dst, uint32_t step, const uint32_t* src, const uint32_t* safe, int left, bool one = false)
{
    if (psz == 16) stage_unit_p<NB, 16>(dst, step, src, safe, left, one);
    else if (psz == 8) stage_unit_p<NB, 8>(dst, step, src, safe, left, one);
    else stage_unit_p<NB, 4>(dst, step, src, safe, left, one);
}

// ----------------------------------------------------------------------------- filters expanded in the kernel

// Row i of a filter tile is (filter group i / (8 R S), tap, filter i % 8): the core-matrix rows of the B operand in memory
// order, so the destination is linear in i.  Filter (within the tile) and offset of the row's packed record.
__device__ __forceinline__ int filter_row(const MmaArgs& g, int i, int WB, int& offset)
{
    const int t = i >> 3, grp = fdiv(t, g.d_rs), tap = t - grp * g.RS;
    const int col = grp * 8 + (i & 7);
    const int f = (col & ~31) + mma_filter_of_column(col & 31);
    offset = (f * g.RS + tap) * g.Cw * WB;
    return f;
}

// Sum of the 32 codes of a channel word as the operand holds them (a bipolar word has no missing ones).
template <int WB>
__device__ __forceinline__ int word_sum(const uint32_t* w, int kind)
{
    if (kind == 2) return 2 * __popc(w[0]) - 32;
    int s = 0;
#pragma unroll
    for (int k = 0; k < WB; ++k) s += (kind == 1 && k == WB - 1 ? -1 : 1) * (__popc(w[k]) << k);
    return s;
}

// One channel word of a filter row -> its two 16-byte core-matrix rows (one of nibbles); rows past the last filter are zero.
template <int WB, bool F4>
__device__ __forceinline__ void expand_filter_word(const uint32_t* w, int kind, bool live, uint32_t dst)
{
    if constexpr (F4) {
        uint32_t n[4];
        expand_nibbles<WB>(w, kind, n);
        if (kind == 2 && !live) {        // missing bits are no -1 (zeros as they are otherwise)
#pragma unroll
            for (int k = 0; k < 4; ++k) n[k] = 0u;
        }
        mm_sts(dst, n[0], n[1], n[2], n[3]);
        return;
    }
    uint32_t o[8];
    expand_word<WB>(w, kind, o);
    if (kind == 2 && !live) {            // a bipolar row must not turn missing bits into -1
#pragma unroll
        for (int k = 0; k < 8; ++k) o[k] = 0u;
    }
    mm_sts(dst, o[0], o[1], o[2], o[3]);
    mm_sts(dst + 128u, o[4], o[5], o[6], o[7]);
}

// `base`: packed records of the tile's filters, in shared memory (bulk copy) or global.  Nibbles: a K step is two channel words, the second
// of an odd number zero.  SUMS: the sum of each filter's codes is collected by column of the tile.
template <int WB, bool F4, bool SUMS>
__device__ __forceinline__ void expand_filters_resident(const MmaArgs& g, uint32_t b_base, const uint32_t* base, int o0, int t, int nt, int* sums)
{
    constexpr int BATCH = 4;                // loads in flight per thread
    const int rows = g.TN * g.RS, total = rows * (F4 ? 2 * g.nblk : g.Cw);
    const uint32_t blk = static_cast<uint32_t>(rows) * 32u;
    int i = t, cw = 0;
    while (i >= rows) { i -= rows; ++cw; }
    for (int j0 = t; j0 < total; j0 += BATCH * nt) {
        uint32_t w[BATCH][WB], dst[BATCH];
        bool live[BATCH];
        int col[BATCH];
#pragma unroll
        for (int b = 0; b < BATCH; ++b) {
            int off = 0;
            if (SUMS) col[b] = fdiv(i >> 3, g.d_rs) * 8 + (i & 7);
            live[b] = cw < g.Cw && o0 + filter_row(g, i, WB, off) < g.O;
            dst[b] = b_base + (F4 ? (cw >> 1) * blk + (cw & 1) * 128u : cw * blk) + static_cast<uint32_t>(i >> 3) * 256u + static_cast<uint32_t>(i & 7) * 16u;
#pragma unroll
            for (int k = 0; k < WB; ++k) w[b][k] = live[b] ? base[off + cw * WB + k] : 0u;
            i += nt;
            while (i >= rows) { i -= rows; ++cw; }
        }
#pragma unroll
        for (int b = 0; b < BATCH; ++b)
            if (j0 + b * nt < total) {
                expand_filter_word<WB, F4>(w[b], g.w_kind, live[b], dst[b]);
                if (SUMS && live[b]) atomicAdd(sums + col[b], word_sum<WB>(w[b], g.w_kind));
            }
    }
}

// ----------------------------------------------------------------------------- prepared filters of the other form

// Filters prepared for layers of other widths (bs_tc_prepare_weights: nibbles or int8, told apart by MM_NIBBLE_MARK) -> `nb` K steps from b0
// on in the form of this layer, by one warp: 16-byte vectors [K step][filter / 8][tap][half][filter % 8] at `dst`.  A layer with such filters
// is right but slow; preparing them for its widths is the remedy.
template <bool F4, class G>
static __device__ __noinline__ void convert_filters(const G& g, unsigned char* dst, int o0, int b0, int nb, int lane)
{
    const int per = g.TN * g.RS * 2;
    const size_t stride = static_cast<size_t>(g.opad) * g.RS * 2;
    const uint4* src = reinterpret_cast<const uint4*>(g.wgt) + static_cast<size_t>(o0) * g.RS * 2;
    for (int b = 0; b < nb; ++b)
#pragma unroll 4
        for (int r = lane; r < per; r += 32) {
            uint32_t o[4] = {0, 0, 0, 0};
            if (F4) {
                // a channel word is one vector here, two there
                const int cw = 2 * (b0 + b) + (r >> 3 & 1);
                if (cw < g.Cw) {
                    const uint4 lo = src[cw * stride + (r & ~8)], hi = src[cw * stride + (r | 8)];
                    const uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const uint32_t neg = (w[k] >> 7) & 0x01010101u, m = neg * 255u;
                        o[k & 3] |= ((__vsub4(w[k] ^ m, m) & 0x07070707u) | neg << 3) << (k & 4);
                    }
                }
            } else {
                const int cw = b0 + b, shift = r & 8 ? 4 : 0;
                const uint4 n = src[(cw >> 1) * stride + ((r & ~8) | (cw & 1) << 3)];
                const uint32_t w[4] = {n.x, n.y, n.z, n.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t v = w[k] >> shift, m = ((v >> 3) & 0x01010101u) * 255u;
                    o[k] = __vsub4((v & 0x07070707u) ^ m, m);
                }
            }
            mm_sts(smem_u32(dst) + static_cast<uint32_t>(b * per + r) * 16u, o[0], o[1], o[2], o[3]);
        }
    fence_proxy_async();
    __syncwarp();
}

// ----------------------------------------------------------------------------- MMA issue

// Fixed kernel sizes: the taps are unrolled, nothing but additions on uniform registers between the MMAs.
// a, b: descriptor words of the block's operands; PITCH and plane offsets in 16-byte units.
template <bool F4>
__device__ __forceinline__ void issue_mma(uint32_t d, uint32_t a, uint32_t a_hi, uint32_t b, uint32_t b_hi, uint32_t idesc, uint32_t acc, uint32_t sf)
{
    if constexpr (F4) mm_mma4(d, a, a_hi, b, b_hi, idesc, acc, sf);
    else mm_mma(d, a, a_hi, b, b_hi, idesc, acc);
}

template <int R, int ST, bool F4>
__device__ __forceinline__ void issue_taps(uint32_t d, uint32_t a, uint32_t a_hi, uint32_t b, uint32_t b_hi, uint32_t idesc, uint32_t acc, uint32_t pitch,
                                           uint32_t HL, uint32_t sf)
{
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int s = 0; s < R; ++s) {
            // 3x3, pad 1, stride 2: taps -1, 0, 1 -> parity 1, 0, 1, shift -1, 0, 0
            const uint32_t off = ST == 1 ? r * pitch + s
                                         : ((r != 1 ? 2u : 0u) + (s != 1 ? 1u : 0u)) * HL + (r > 0 ? pitch : 0u) + (s > 0 ? 1u : 0u);
            issue_mma<F4>(d, a + off, a_hi, b + static_cast<uint32_t>(r * R + s) * 16u, b_hi, idesc, (r == 0 && s == 0) ? acc : 1u, sf);
        }
}

enum { TAPS_1 = 0, TAPS_3S1, TAPS_3S2, TAPS_ANY };

template <int TAPS, bool F4>
__device__ __forceinline__ void issue_block(const MmaArgs& g, uint32_t d, uint32_t a, uint32_t a_hi, uint32_t b, uint32_t b_hi, uint32_t idesc, uint32_t acc,
                                            uint32_t pitch, uint32_t HL, uint32_t sf)
{
    if (TAPS == TAPS_1) issue_mma<F4>(d, a, a_hi, b, b_hi, idesc, acc, sf);
    else if (TAPS == TAPS_3S1) issue_taps<3, 1, F4>(d, a, a_hi, b, b_hi, idesc, acc, pitch, HL, sf);
    else if (TAPS == TAPS_3S2) issue_taps<3, 2, F4>(d, a, a_hi, b, b_hi, idesc, acc, pitch, HL, sf);
    else
        for (int r = 0; r < g.R; ++r)
            for (int s = 0; s < g.R; ++s) {
                const int rp = r - g.pad, sp = s - g.pad;
                uint32_t off;
                if (g.stride == 1) off = static_cast<uint32_t>(r * g.pitch + s);
                else off = static_cast<uint32_t>(((rp & 1) * 2 + (sp & 1)) * g.HL + ((rp >> 1) - g.rmin) * g.pitch + (sp >> 1) - g.smin);
                issue_mma<F4>(d, a + off, a_hi, b, b_hi, idesc, acc, sf);
                acc = 1u;
                b += 16u;
            }
}

// Chunks of this CTA: all of them, or its share of an item split over a cluster.
struct MmaChunks {
    int beg, n, rank;
    __device__ __forceinline__ MmaChunks(const MmaArgs& g, bool split) : beg(0), n(g.nchunks), rank(0)
    {
        if (!split) return;
        rank = blockIdx.x & (g.split - 1);
        beg = (rank * g.nchunks) >> g.split_log;
        n = (((rank + 1) * g.nchunks) >> g.split_log) - beg;
    }
};

struct MmaIssue {
    uint64_t *full_e, *empty_e, *full_acc, *empty_acc, *wgt_full, *form_ok;
    uint32_t smem0, tmem;
    int items;
    bool resident;
};

// The MMA warp's walk over items and chunks, in uniform code; every MMA and every commit elects its thread by itself (one elected region
// for a whole chunk was slower: its descriptors move through vector registers, 100 cycles per MMA against 85 to 90).
template <int TAPS, bool SPLIT, bool F4>
__device__ __forceinline__ void issue_items(const MmaArgs& g, const MmaIssue& m)
{
    const uint32_t NI16 = static_cast<uint32_t>(g.NI);
    // K-major, no swizzle: core matrices of 8 rows x 16 bytes; leading offset = next 16 channels, stride offset = next 8 rows
    const uint32_t a_hi = (128u >> 4) | (1u << 14), b_hi = static_cast<uint32_t>(g.RS * 16) | (1u << 14);
    // (32 channels as nibbles: the second half of the step reads the first again, against zeros)
    const uint32_t a_lo0 = F4 && g.one_word ? 0u : (NI16 & 0x3FFFu) << 16, b_lo0 = (128u >> 4) << 16;
    // descriptors take the offset within the CTA; in a cluster the upper bits of a shared address name the CTA
    const uint32_t smem_off = m.smem0 & 0x3FFFFu, e_base = (smem_off + g.off_e) >> 4, w_base = smem_off >> 4;
    const uint32_t blk16 = static_cast<uint32_t>(g.TN * g.RS * 2), idesc = g.idesc;
    const uint32_t pitch = static_cast<uint32_t>(g.pitch), HL = static_cast<uint32_t>(g.HL), TN = static_cast<uint32_t>(g.TN);
    const uint32_t e16 = static_cast<uint32_t>(g.e_bytes >> 4), b16 = static_cast<uint32_t>(g.b_bytes >> 4);
    const MmaChunks range(g, SPLIT);
    const int log = SPLIT ? g.split_log : 0;
    const int nchunks = range.n, PT = g.PT, per_chunk = F4 ? g.units : g.units * 2, blocks = g.nblk, nse = g.nse, nacc = g.nacc;
    const uint32_t sf = m.tmem + static_cast<uint32_t>(g.sf_col);
    unsigned limit = 1u << 20;
    if (m.resident) mm_wait_uniform(m.wgt_full, 0, limit);
    if (m.form_ok) mm_wait_uniform(m.form_ok, 0, limit);
    MM_TRACE((threadIdx.x & 31) == 0, TR_WGT, 0);
#ifdef BS_TRACE
    int mseq = 0;
#endif
    int ie = 0, ia = 0;
    unsigned pe = 0, pa = 0;
    const uint32_t acc0 = !F4 && g.preset ? 1u : 0u;
    for (int it = blockIdx.x >> log; it < m.items; it += gridDim.x >> log) {
        mm_wait_uniform(&m.empty_acc[ia], pa, limit);
        const uint32_t d0 = m.tmem + static_cast<uint32_t>(ia * PT) * TN;
        for (int c = 0; c < nchunks; ++c) {
            const int b0 = (range.beg + c) * per_chunk;
            const int nb = blocks - b0 < per_chunk ? blocks - b0 : per_chunk;
            const uint32_t wb = b_lo0 | (w_base + (m.resident ? static_cast<uint32_t>(b0) * blk16 : static_cast<uint32_t>(ie) * b16));
            const uint32_t eb = a_lo0 | (e_base + static_cast<uint32_t>(ie) * e16);
            mm_wait_uniform(&m.full_e[ie], pe, limit);
            mm_fence_after();
            MM_TRACE((threadIdx.x & 31) == 0, TR_MBEG, mseq);
            {
                uint32_t acc = c == 0 ? acc0 : 1u;
                uint32_t d = d0, at = eb;
                for (int t = 0; t < PT; ++t, d += TN, at += 128u) {
                    uint32_t a = at, b = wb;
                    issue_block<TAPS, F4>(g, d, a, a_hi, b, b_hi, idesc, acc, pitch, HL, sf);
#pragma unroll(TAPS == TAPS_1 ? 4 : 1)
                    for (int k = 1; k < nb; ++k) {
                        a += 2u * NI16;
                        b += blk16;
                        issue_block<TAPS, F4>(g, d, a, a_hi, b, b_hi, idesc, 1u, pitch, HL, sf);
                    }
                }
                mm_commit(&m.empty_e[ie]);
                if (c == nchunks - 1) mm_commit(&m.full_acc[ia]);
            }
#ifdef BS_TRACE
            MM_TRACE((threadIdx.x & 31) == 0, TR_MEND, mseq);
            ++mseq;
#endif
            if (++ie == nse) { ie = 0; pe ^= 1u; }
        }
        if (++ia == nacc) { ia = 0; pa ^= 1u; }
    }
    if (limit == 1u && (threadIdx.x & 31) == 0) atomicOr(g.status, STATUS_TIMEOUT);
    __syncwarp();
}

// ----------------------------------------------------------------------------- epilogue

constexpr int MM_SF_COLS = 32;                  // columns that hold scale factors (eight bytes a row and column of the operands need at most 16)
constexpr uint32_t MM_PRESET = 0x4B400000u;      // 1.5 * 2^23: an accumulator that starts here IS the float 12582912 + acc

// Fast requantisation of 16 accumulators of one pixel = half a group of 32 filters (codes of 1..4 bits, residual codes unsigned).
//   acc -> float: integer accumulators start at the bit pattern of 1.5 * 2^23, so one subtraction converts (|acc| < 2^22); those of F4 are floats.
//   t = fmaf(acc, scale, bias) and fmaf(res_scale, res, t) in the formula's order, two outputs per instruction (f32x2), all
//   scaled by 2^-24: an exact change of the exponents (the caller's table check keeps every value in the normal range).
//   rint: adding 0.75 (one ulp = 2^-24) leaves the rounded level in the low mantissa bits; two outputs are clamped as a pair
//   of 16-bit integers (|level| < 2^15, checked), which equals clip-then-round because the limits are integers.
//   Residual codes enter as denormals: code << p has the float value code * 2^(p - 149), and the multiplier of pair i
//   carries the missing power of two, so a code costs one AND.
// Half w holds the pairs (filter 2 i + w, filter 16 + 2 i + w), i = 0..7: shifting pair i by 2 i collects sixteen 2-bit codes in
// one word (4 i' and two words for wider codes), and a few operations per group de-interleave the words of both halves into
// planes.  About 4 instructions per output, a quarter of them loads and integer ALU; the threshold-table form it replaces
// took 8 (12 with a residual).
template <int OBC, int RESC, bool LO0, bool F4, bool OFS>
__device__ __forceinline__ void requant16(const uint32_t (&v)[16], uint32_t tab, uint32_t cor, uint32_t rtab, uint32_t z0, uint32_t z1, uint32_t lo2, uint32_t hi2,
                                          uint32_t (&W)[2])
{
    const u64 unbias = f2_pack(0xCB400000u, 0xCB400000u), magic = f2_pack(0x3F400000u, 0x3F400000u);
    const uint32_t z0h = z0 >> 16, z1h = z1 >> 16;
    uint32_t k[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        u64 s2, b2;
        asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(s2), "=l"(b2) : "r"(tab + i * 16));
        u64 acc = f2_pack(v[2 * i], v[2 * i + 1]);
        if (OFS) {
            u64 c2;
            asm volatile("ld.shared.b64 %0, [%1];" : "=l"(c2) : "r"(cor + i * 8));
            acc = f2_add(acc, c2);
        }
        u64 t = f2_fma(F4 ? acc : f2_add(acc, unbias), s2, b2);
        if (RESC) {
            u64 rmul;
            asm volatile("ld.shared.b64 %0, [%1];" : "=l"(rmul) : "r"(rtab + (RESC == 2 ? i : (i >> 1) * 2) * 8));
            const uint32_t m = RESC == 2 ? 3u << (2 * i) : 15u << (4 * (i >> 1));
            const bool odd = RESC == 4 && (i & 1);
            t = f2_fma(f2_pack((odd ? z1 : z0) & m, (odd ? z1h : z0h) & m), rmul, t);
        }
        uint32_t lo, hi;
        f2_split(f2_add(t, magic), lo, hi);
        k[i] = __byte_perm(lo, hi, 0x5410);
        if (LO0) {
            k[i] = __vimin_s16x2_relu(k[i], hi2);
        } else {
            asm("min.s16x2 %0, %0, %1;" : "+r"(k[i]) : "r"(hi2));
            asm("max.s16x2 %0, %0, %1;" : "+r"(k[i]) : "r"(lo2));
            k[i] &= OBC == 2 ? 0x00030003u : 0x000F000Fu;
        }
    }
    if (OBC == 2) {
        W[0] = ((k[0] + (k[1] << 2)) + ((k[2] + (k[3] << 2)) << 4)) + (((k[4] + (k[5] << 2)) + ((k[6] + (k[7] << 2)) << 4)) << 8);
    } else {
        W[0] = (k[0] + (k[2] << 4)) + ((k[4] + (k[6] << 4)) << 8);
        W[1] = (k[1] + (k[3] << 4)) + ((k[5] + (k[7] << 4)) << 8);
    }
}

// The documented formula, one output at a time: any scale, bias, residual format.
template <class G>
static __device__ __noinline__ void requant32_formula(const G& g, const uint32_t* v, int ob, const uint32_t* rw, uint32_t* ow)
{
    int qmin, qmax;
    code_limits(g.out_bits, g.out_sign, qmin, qmax);
    const float fqmin = static_cast<float>(qmin), fqmax = static_cast<float>(qmax);
    for (int f = 0; f < 32; ++f) {
        if (ob + f >= g.O) break;
        const int acc = static_cast<int>(v[mma_column_of_filter(f)]);
        float val = fmaf(static_cast<float>(acc), g.scale[ob + f], g.bias[ob + f]);
        if (g.residual) {
            unsigned rpat = 0;
            for (int j = 0; j < g.res_bits; ++j) rpat |= ((rw[j] >> f) & 1u) << j;
            val = fmaf(g.res_scale, static_cast<float>(pattern_value(rpat, g.res_bits, g.res_sign)), val);
        }
        if (g.relu) val = fmaxf(val, 0.0f);
        int code;
        if (g.out_sign == BS_BIPOLAR) code = val >= 0.0f ? 1 : -1;
        else code = small_float_to_int_rn(fminf(fmaxf(val, fqmin), fqmax));
        const unsigned pat = stored_pattern(code, g.out_bits, g.out_sign);
        for (int j = 0; j < g.out_bits; ++j) ow[j] |= ((pat >> j) & 1u) << f;
    }
}

// Work items of a CTA: item = pixel tile * tiles_o + filter tile, walked without divisions.
struct MmaWalk {
    int it, m, o, dm, dn, log;       // log: of the CTAs that share an item
    __device__ __forceinline__ MmaWalk(const MmaArgs& g, int log_) : log(log_)
    {
        it = blockIdx.x >> log;
        m = it / g.tiles_o; o = it - m * g.tiles_o;
        const int n = gridDim.x >> log;
        dm = n / g.tiles_o; dn = n - dm * g.tiles_o;
    }
    __device__ __forceinline__ void next(const MmaArgs& g)
    {
        it += gridDim.x >> log; m += dm; o += dn;
        if (o >= g.tiles_o) { o -= g.tiles_o; ++m; }
    }
};

struct MmaPixel { bool valid; int pix, n, rem; };       // output pixel index (n P Q + p Q + q), image, p Q + q

__device__ __forceinline__ MmaPixel mma_pixel(const MmaArgs& g, int pos)
{
    MmaPixel o;
    if (g.flat) {
        o.valid = pos < g.total; o.pix = pos;
        o.n = 0; o.rem = pos;
        if (g.out_i32 && !g.i32_nhwc) { o.n = fdiv(pos, g.d_img); o.rem = pos - o.n * g.d_img.d; }
        return o;
    }
    int u = fdiv(pos, g.d_img);
    int rem = pos - u * g.d_img.d;
    const int y = fdiv(rem, g.d_pitch), x = rem - y * g.d_pitch.d;
    const int n = fdiv(u, g.d_strips), q = (u - n * g.d_strips.d) * g.strip_q + x;
    o.valid = pos < g.total && y < g.P && x < g.strip_q && q < g.Q;
    o.n = n; o.rem = y * g.Q + q;
    o.pix = n * g.P * g.Q + o.rem;
    return o;
}

// Checks and lays out the (scale, bias) pairs of the CTA's filters: tab[16 * group + pair] = (s0, s1, b0, b1) scaled by 2^-24.
// *ok stays 1 when the fast form takes the formula's decision for every possible accumulator.
template <class G>
__device__ __forceinline__ void epilogue_tables(const G& g, float4* tab, float2* rtab, int* ok, int o0, int t, int nt)
{
    const float res_max = g.residual ? fabsf(g.res_scale) * 15.0f : 0.0f;
    for (int e = t; e < g.TN / 2; e += nt) {
        const int grp = e >> 4, pr = e & 15;
        float s[2] = {0.f, 0.f}, b[2] = {0.f, 0.f};
        for (int h = 0; h < 2; ++h) {
            const int o = o0 + grp * 32 + mma_filter_of_column(2 * pr + h);
            if (o >= g.O) continue;
            s[h] = g.scale[o];
            b[h] = g.bias[o];
            const float as = fabsf(s[h]), ab = fabsf(b[h]);
            const bool fine = (as == 0.f || as > 1e-18f) && (ab == 0.f || ab > 1e-18f) && as * g.acc_bound + ab + res_max < 32000.0f;
            if (!fine) *ok = 0;             // also catches NaN and infinities
        }
        const float k = 5.9604644775390625e-08f;        // 2^-24
        tab[e] = make_float4(s[0] * k, s[1] * k, b[0] * k, b[1] * k);
    }
    if (g.residual && t < 8) {
        // entry t multiplies a code << (2 t): 2^(149 - 24 - 2 t) (codes of 3-4 bits use every other entry)
        const float m = g.res_scale * __uint_as_float(static_cast<uint32_t>(127 + 125 - 2 * t) << 23);
        rtab[t] = make_float2(m, m);
    }
}

// What the epilogue warps share: the walk over the items and the hand-over of the accumulator buffers.
struct MmaEpi {
    unsigned char* smem;
    uint64_t* full_acc;
    uint64_t* empty_acc;
    int* fast_ok;
    uint32_t acc;            // tensor-memory address of the warp's lanes
    int row0;                // tile row of this thread
    int set;                 // 0 or 1: which of the two warps of a lane quadrant
    int tid, lane, warp;
    uint64_t* red_full;      // the partial sums of the other CTAs of a split item have arrived
};

// Whole number of an accumulator.
__device__ __forceinline__ uint32_t acc_int(bool f4, uint32_t v, uint32_t bias)
{
    return f4 ? __float_as_uint(__uint_as_float(v) + 12582912.0f) - MM_PRESET : v - bias;
}

// Split items.  CTAs of rank 1 and up send their accumulators to the shared memory of rank 0 ([rank - 1][column][row], so a warp
// stores 128 contiguous bytes), which adds them to its own in tensor memory and goes on as if it had done all the chunks.
template <int EW, bool F4>
__device__ __forceinline__ bool send_partials(const MmaArgs& g, const MmaEpi& e, int rank)
{
    if (!mm_wait(&e.full_acc[0], 0)) return false;
    mm_fence_after();
    const uint32_t bias = !F4 && g.preset ? MM_PRESET : 0u;
    const int columns = g.PT * g.TN;
    const uint32_t dst = mm_leader(smem_u32(e.smem + g.off_red)) + static_cast<uint32_t>(((rank - 1) * columns * 128 + e.row0) * 4);
    for (int c0 = e.set * 32; c0 < columns; c0 += EW / 4 * 32)
        for (int h = 0; h < 32; h += 16) {
            uint32_t v[16];
            mm_ld16(e.acc + static_cast<uint32_t>(c0 + h), v);
            mm_ld_wait();
            mm_landed(v);
#pragma unroll
            for (int c = 0; c < 16; ++c)
                asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(dst + static_cast<uint32_t>((c0 + h + c) * 512)), "r"(v[c] - bias) : "memory");
        }
    __syncwarp();
    if (e.lane == 0) asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(mm_leader(smem_u32(e.red_full))) : "memory");
    return true;
}
template <int EW, bool F4>
__device__ __forceinline__ bool merge_partials(const MmaArgs& g, const MmaEpi& e)
{
    if (!mm_wait_cluster(e.red_full, 0)) return false;
    const int columns = g.PT * g.TN;
    const uint32_t src = smem_u32(e.smem + g.off_red) + static_cast<uint32_t>(e.row0 * 4);
    for (int c0 = e.set * 32; c0 < columns; c0 += EW / 4 * 32)
        for (int h = 0; h < 32; h += 16) {
            uint32_t v[16];
            mm_ld16(e.acc + static_cast<uint32_t>(c0 + h), v);
            mm_ld_wait();
            mm_landed(v);
            for (int r = 0; r < g.split - 1; ++r)
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    uint32_t x;
                    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(x) : "r"(src + static_cast<uint32_t>((r * columns + c0 + h + c) * 512)));
                    v[c] = F4 ? __float_as_uint(__uint_as_float(v[c]) + __uint_as_float(x)) : v[c] + x;
                }
            mm_st16(e.acc + static_cast<uint32_t>(c0 + h), v);
        }
    mm_st_wait();
    return true;
}

template <class G>
__device__ __forceinline__ void store_codes(const G& g, int pix, int ob, uint32_t (&ow)[4])
{
    if (g.O - ob < 32) {
        const uint32_t m = (1u << (g.O - ob)) - 1u;
#pragma unroll
        for (int j = 0; j < 4; ++j) ow[j] &= m;
    }
    uint32_t* dst = g.out_packed + (static_cast<size_t>(pix) * g.out_cw_total + g.out_cw_off + (ob >> 5)) * g.out_bits;
    if (g.out_bits == 2) {
        *reinterpret_cast<uint2*>(dst) = make_uint2(ow[0], ow[1]);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (j < g.out_bits) dst[j] = ow[j];
    }
}

// Residual planes of (pixel, 32 filters from ob).
template <class G>
__device__ __forceinline__ void load_residual(const G& g, int pix, int ob, uint32_t (&rw)[4])
{
    const uint32_t* rp = g.residual + (static_cast<size_t>(pix) * g.res_cw_total + ((g.res_c_off + ob) >> 5)) * g.res_bits;
    if (g.res_bits == 2) {
        const uint2 t = *reinterpret_cast<const uint2*>(rp);
        rw[0] = t.x; rw[1] = t.y;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (j < g.res_bits) rw[j] = rp[j];
    }
}

// One group of 32 filters through the documented formula (any scale, bias, residual and output format).
static __device__ __noinline__ void epilogue_formula(const MmaArgs& g, uint32_t addr, bool live, int pix, int ob, uint32_t bias, const float* cor)
{
    uint32_t v[32], rw[4] = {0, 0, 0, 0}, ow[4] = {0, 0, 0, 0};
    mm_ld32(addr, v);
    mm_ld_wait();
    mm_landed(v);
    if (live) {
        for (int c = 0; c < 32; ++c) v[c] = acc_int(g.f4, cor ? __float_as_uint(__uint_as_float(v[c]) + cor[c]) : v[c], bias);
        if (g.residual) load_residual(g, pix, ob, rw);
        requant32_formula(g, v, ob, rw, ow);
        store_codes(g, pix, ob, ow);
    }
    __syncwarp();
}
// A whole item that way, its accumulators set back to the preset.
static __device__ __noinline__ void epilogue_item_formula(const MmaArgs& g, uint32_t acc, int base, int o0, int set, int step, const float* cor)
{
    const int groups = g.TN >> 5;
    for (int u = set; u < g.PT * groups; u += step) {
        const int t = u / groups, cc = u - t * groups;
        const MmaPixel px = mma_pixel(g, base + t * 128);
        const uint32_t col = acc + static_cast<uint32_t>(t * g.TN + cc * 32);
        epilogue_formula(g, col, px.valid && o0 + cc * 32 < g.O, px.pix, o0 + cc * 32, MM_PRESET, cor ? cor + cc * 32 : nullptr);
        if (!g.f4)
            for (int c = 0; c < 32; c += 8) mm_st8(col + c, MM_PRESET);
    }
}

// Codes out, fast form.  One warp's accumulators arrive 16 columns at a time; the next 16 are on their way from tensor memory
// while the current ones are computed, and the residual words of a group are fetched one group ahead.
template <int OBC, int RESC, bool LO0, int EW, bool SPLIT, bool F4, bool OFS, class Sums>
__device__ __forceinline__ bool epilogue_codes(const MmaArgs& g, const MmaEpi& e, const Sums& sums)
{
    constexpr int STEP = EW / 4;
    const uint32_t tab0 = smem_u32(e.smem + g.off_tab), rtab = tab0 + static_cast<uint32_t>(g.TN) * 8u, cor0 = rtab + 64u;
    int qmin, qmax;
    code_limits(g.out_bits, g.out_sign, qmin, qmax);
    const int lo = g.relu && qmin < 0 ? 0 : qmin;
    const uint32_t lo2 = (static_cast<uint32_t>(lo) & 0xFFFFu) * 0x10001u, hi2 = (static_cast<uint32_t>(qmax) & 0xFFFFu) * 0x10001u;
    const int groups = g.TN >> 5;
    int tab_o = -1, ia = 0;
    unsigned pa = 0;
    bool ok = true, fast = false, waited = !g.early_b;
    for (MmaWalk w(g, SPLIT ? g.split_log : 0); w.m < g.tiles_m; w.next(g)) {
        const int o0 = w.o * g.TN;
        if (w.o != tab_o) {
            if (tab_o >= 0) asm volatile("bar.sync 2, %0;" ::"n"(EW * 32) : "memory");     // every warp is done with the old table
            epilogue_tables(g, reinterpret_cast<float4*>(e.smem + g.off_tab), reinterpret_cast<float2*>(e.smem + g.off_tab + g.TN * 8), e.fast_ok, o0,
                            e.tid, EW * 32);
            if (OFS) sums();
            asm volatile("bar.sync 2, %0;" ::"n"(EW * 32) : "memory");
            fast = *reinterpret_cast<volatile int*>(e.fast_ok) != 0;
            tab_o = w.o;
        }
        if (!waited) { mm_pdl_wait(); waited = true; }
        const int base = w.m * 128 * g.PT + e.row0;
        int t = 0, cc = e.set;                        // row tile and filter group
        while (cc >= groups) { cc -= groups; ++t; }
        MmaPixel px = mma_pixel(g, base + t * 128);
        uint32_t rn[4] = {0, 0, 0, 0};
        if (RESC && t < g.PT && px.valid && o0 + cc * 32 < g.O) load_residual(g, px.pix, o0 + cc * 32, rn);
        if (ok) ok = mm_wait(&e.full_acc[ia], pa);    // after a wait that ran out the walk goes on without waiting, so the named barriers stay matched
        mm_fence_after();
        if (SPLIT && ok) ok = merge_partials<EW, F4>(g, e);
        MM_TRACE(e.tid == 0, TR_EBEG, (w.it - static_cast<int>(blockIdx.x)) / static_cast<int>(gridDim.x));
        const uint32_t acc = e.acc + static_cast<uint32_t>(ia * g.PT * g.TN);
        if (!fast) {
            epilogue_item_formula(g, acc, base, o0, e.set, STEP, OFS ? reinterpret_cast<const float*>(e.smem + g.off_tab + g.TN * 8 + 64) : nullptr);
            t = g.PT;
        }
        uint32_t A[16], B[16];
        if (t < g.PT) mm_ld16(acc + static_cast<uint32_t>(t * g.TN + cc * 32), A);
        while (t < g.PT) {
            const int ob = o0 + cc * 32, pix = px.pix;
            const bool live = px.valid && ob < g.O;
            const uint32_t col = acc + static_cast<uint32_t>(t * g.TN + cc * 32);
            const uint32_t tab = tab0 + static_cast<uint32_t>(cc) * 256u;
            uint32_t rw[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) rw[j] = rn[j];
            mm_ld_wait();
            mm_landed(A);
            mm_ld16(col + 16, B);
            if (!F4) { mm_st8(col, MM_PRESET); mm_st8(col + 8, MM_PRESET); }
            // the next group's place and residual
            cc += STEP;
            const int t_old = t;
            while (cc >= groups) { cc -= groups; ++t; }
            if (t != t_old && t < g.PT) px = mma_pixel(g, base + t * 128);
            if (RESC && t < g.PT && px.valid && o0 + cc * 32 < g.O) load_residual(g, px.pix, o0 + cc * 32, rn);
            uint32_t z[4] = {0, 0, 0, 0}, Wa[2], Wb[2];
            if (RESC == 2) {
                z[0] = (rw[0] & 0x55555555u) | ((rw[1] << 1) & 0xAAAAAAAAu);
                z[1] = ((rw[0] >> 1) & 0x55555555u) | (rw[1] & 0xAAAAAAAAu);
            } else if (RESC == 4) {
                const uint32_t p = (rw[0] & 0x55555555u) | ((rw[1] << 1) & 0xAAAAAAAAu), q = ((rw[0] >> 1) & 0x55555555u) | (rw[1] & 0xAAAAAAAAu);
                const uint32_t r = (rw[2] & 0x55555555u) | ((rw[3] << 1) & 0xAAAAAAAAu), s = ((rw[2] >> 1) & 0x55555555u) | (rw[3] & 0xAAAAAAAAu);
                z[0] = (p & 0x33333333u) | ((r << 2) & 0xCCCCCCCCu);          // filters 0, 4, .. (half 0, even pairs)
                z[1] = (q & 0x33333333u) | ((s << 2) & 0xCCCCCCCCu);          // 1, 5, .. (half 1, even pairs)
                z[2] = ((p >> 2) & 0x33333333u) | (r & 0xCCCCCCCCu);          // 2, 6, .. (half 0, odd pairs)
                z[3] = ((q >> 2) & 0x33333333u) | (s & 0xCCCCCCCCu);
            }
            requant16<OBC, RESC, LO0, F4, OFS>(A, tab, cor0 + static_cast<uint32_t>(ob - o0) * 4u, rtab, z[0], z[2], lo2, hi2, Wa);
            mm_ld_wait();
            mm_landed(B);
            if (t < g.PT) mm_ld16(acc + static_cast<uint32_t>(t * g.TN + cc * 32), A);
            if (!F4) { mm_st8(col + 16, MM_PRESET); mm_st8(col + 24, MM_PRESET); }
            requant16<OBC, RESC, LO0, F4, OFS>(B, tab + 128u, cor0 + static_cast<uint32_t>(ob - o0) * 4u + 64u, rtab, z[1], z[3], lo2, hi2, Wb);
            uint32_t ow[4] = {0, 0, 0, 0};
            if (OBC == 2) {
                ow[0] = (Wa[0] & 0x55555555u) | ((Wb[0] << 1) & 0xAAAAAAAAu);
                ow[1] = ((Wa[0] >> 1) & 0x55555555u) | (Wb[0] & 0xAAAAAAAAu);
            } else {
                const uint32_t M = 0x11111111u;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    ow[j] = ((Wa[0] >> j) & M) | (((Wb[0] >> j) & M) << 1) | (((Wa[1] >> j) & M) << 2) | (((Wb[1] >> j) & M) << 3);
            }
            if (live) store_codes(g, pix, ob, ow);
        }
        if (!F4) mm_st_wait();
        mm_fence_before();
        __syncwarp();
        if (e.lane == 0) mm_arrive(&e.empty_acc[ia]);
        MM_TRACE(e.tid == 0, TR_EEND, (w.it - static_cast<int>(blockIdx.x)) / static_cast<int>(gridDim.x));
        if (++ia == g.nacc) { ia = 0; pa ^= 1u; }
    }
    if (!waited) mm_pdl_wait();
    return ok;
}

// Nibbles, codes of at most two bits; items of two or four row tiles: two row tiles at a time (NT), so that the scales and biases of 32 filters are
// read once for both.  An LDS.128 costs four wavefronts of shared memory even when all lanes read the same address, and 16 of them for every
// 32 x 32 outputs (24 with the residual's multipliers, which are shifts here) took more of its bandwidth than the MMAs' operands.  Eight
// columns of each tile are computed while the next eight are on their way.
// conv2_x of 64 images: 14.1 -> 13.5 us without, 16.4 -> 15.1 us with a residual.  (Fragments of 16 x 256 bits, whose lanes need the
// constants of 8 filters only, made it 16.1 and 19.7: trading codes for plane words between lanes costs more than the loads.)
// Eight columns of two tiles: codes of pair i at bits 2 i of either half of W.  z: residual codes of the pairs from bit 0 of either half on.
template <bool RES, int NT>
__device__ __forceinline__ void requant8(const uint32_t (&v)[NT][8], uint32_t tab, const uint32_t (&z)[NT], u64 rmul, u64 rmul4, uint32_t hi2, uint32_t (&W)[NT])
{
    const u64 magic = f2_pack(0x3F400000u, 0x3F400000u);
    uint32_t k[NT][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        u64 s2, b2;
        asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(s2), "=l"(b2) : "r"(tab + i * 16));
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            u64 t = f2_fma(f2_pack(v[j][2 * i], v[j][2 * i + 1]), s2, b2);
            if (RES) {
                const uint32_t c = i < 2 ? z[j] : z[j] >> 4, m = i & 1 ? 12u : 3u;
                t = f2_fma(f2_pack(c & m, (c >> 16) & m), i & 1 ? rmul4 : rmul, t);
            }
            uint32_t lo, hi;
            f2_split(f2_add(t, magic), lo, hi);
            k[j][i] = __vimin_s16x2_relu(__byte_perm(lo, hi, 0x5410), hi2);
        }
    }
#pragma unroll
    for (int j = 0; j < NT; ++j) W[j] = (k[j][0] + (k[j][1] << 2)) + ((k[j][2] + (k[j][3] << 2)) << 4);
}
template <bool RES, int NT, int EW, bool SPLIT>
__device__ __forceinline__ bool epilogue_tiles(const MmaArgs& g, const MmaEpi& e)
{
    constexpr int STEP = EW / 4;
    const uint32_t tab0 = smem_u32(e.smem + g.off_tab);
    int qmin, qmax;
    code_limits(g.out_bits, g.out_sign, qmin, qmax);
    const uint32_t hi2 = (static_cast<uint32_t>(qmax) & 0xFFFFu) * 0x10001u;
    // a residual code in the low bits of a word is the denormal code * 2^-149; everything is scaled by 2^-24
    const uint32_t rm = __float_as_uint(g.res_scale * __uint_as_float(252u << 23)), rm4 = __float_as_uint(g.res_scale * __uint_as_float(250u << 23));
    const u64 rmul = f2_pack(rm, rm), rmul4 = f2_pack(rm4, rm4);
    const int groups = g.TN >> 5;
    int tab_o = -1, ia = 0;
    unsigned pa = 0;
    bool ok = true, fast = false, waited = !g.early_b;
    for (MmaWalk w(g, SPLIT ? g.split_log : 0); w.m < g.tiles_m; w.next(g)) {
        const int o0 = w.o * g.TN;
        if (w.o != tab_o) {
            if (tab_o >= 0) asm volatile("bar.sync 2, %0;" ::"n"(EW * 32) : "memory");     // every warp is done with the old table
            epilogue_tables(g, reinterpret_cast<float4*>(e.smem + g.off_tab), reinterpret_cast<float2*>(e.smem + g.off_tab + g.TN * 8), e.fast_ok, o0,
                            e.tid, EW * 32);
            asm volatile("bar.sync 2, %0;" ::"n"(EW * 32) : "memory");
            fast = *reinterpret_cast<volatile int*>(e.fast_ok) != 0;
            tab_o = w.o;
        }
        if (!waited) { mm_pdl_wait(); waited = true; }
        const int base = w.m * 128 * g.PT + e.row0;
        // units (NT tiles, group), group fastest
        int t = 0, cc = e.set;
        while (cc >= groups) { cc -= groups; t += NT; }
        int pix[NT];
        auto pixels = [&]() {
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                const MmaPixel px = mma_pixel(g, base + (t + j) * 128);
                pix[j] = px.valid ? px.pix : -1;
            }
        };
        uint32_t rn[NT][4];
        auto residual = [&](int ob) {
#pragma unroll
            for (int j = 0; j < NT; ++j) {
#pragma unroll
                for (int k = 0; k < 4; ++k) rn[j][k] = 0;
                if (RES && pix[j] >= 0 && ob < g.O) load_residual(g, pix[j], ob, rn[j]);
            }
        };
        if (t < g.PT) {
            pixels();
            residual(o0 + cc * 32);
        }
        if (ok) ok = mm_wait(&e.full_acc[ia], pa);    // after a wait that ran out the walk goes on without waiting, so the named barriers stay matched
        mm_fence_after();
        if (SPLIT && ok) ok = merge_partials<EW, true>(g, e);
        MM_TRACE(e.tid == 0, TR_EBEG, (w.it - static_cast<int>(blockIdx.x)) / static_cast<int>(gridDim.x));
        const uint32_t acc = e.acc + static_cast<uint32_t>(ia * g.PT * g.TN), TN = static_cast<uint32_t>(g.TN);
        if (!fast) {
            epilogue_item_formula(g, acc, base, o0, e.set, STEP, nullptr);
            t = g.PT;
        }
        uint32_t v[2][NT][8];           // [buffer][tile]
        uint32_t col = acc + static_cast<uint32_t>(t * g.TN + cc * 32);
        if (t < g.PT)
#pragma unroll
            for (int j = 0; j < NT; ++j) mm_ld8(col + j * TN, v[0][j]);
        while (t < g.PT) {
            const int ob = o0 + cc * 32;
            const uint32_t tab = tab0 + static_cast<uint32_t>(cc) * 256u;
            int to[NT];
            uint32_t z[2][NT];                             // [half of the filters][tile]
#pragma unroll
            for (int j = 0; j < NT; ++j) { to[j] = pix[j]; z[0][j] = z[1][j] = 0u; }
            if (RES)
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    z[0][j] = (rn[j][0] & 0x55555555u) | ((rn[j][1] << 1) & 0xAAAAAAAAu);
                    z[1][j] = ((rn[j][0] >> 1) & 0x55555555u) | (rn[j][1] & 0xAAAAAAAAu);
                }
            // the next unit's place and residual
            cc += STEP;
            const int t_old = t;
            while (cc >= groups) { cc -= groups; t += NT; }
            const bool more = t < g.PT;
            if (more) {
                if (t != t_old) pixels();
                residual(o0 + cc * 32);
            }
            const uint32_t next = acc + static_cast<uint32_t>(t * g.TN + cc * 32);
            uint32_t H[2][NT];                             // [half][tile]
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                mm_ld_wait();
#pragma unroll
                for (int j = 0; j < NT; ++j) mm_landed(v[p & 1][j]);
                if (p < 3 || more) {
                    const uint32_t from = p < 3 ? col + 8u * (p + 1) : next;
#pragma unroll
                    for (int j = 0; j < NT; ++j) mm_ld8(from + j * TN, v[(p & 1) ^ 1][j]);
                }
                uint32_t zp[NT], W[NT];
#pragma unroll
                for (int j = 0; j < NT; ++j) zp[j] = z[p >> 1][j] >> (8 * (p & 1));
                requant8<RES, NT>(v[p & 1], tab + 64u * p, zp, rmul, rmul4, hi2, W);
#pragma unroll
                for (int j = 0; j < NT; ++j) H[p >> 1][j] = p & 1 ? H[p >> 1][j] + (W[j] << 8) : W[j];
            }
            col = next;
#pragma unroll
            for (int j = 0; j < NT; ++j)
                if (to[j] >= 0 && ob < g.O) {
                    uint32_t ow[4] = {(H[0][j] & 0x55555555u) | ((H[1][j] << 1) & 0xAAAAAAAAu), ((H[0][j] >> 1) & 0x55555555u) | (H[1][j] & 0xAAAAAAAAu), 0u, 0u};
                    store_codes(g, to[j], ob, ow);
                }
        }
        mm_fence_before();
        __syncwarp();
        if (e.lane == 0) mm_arrive(&e.empty_acc[ia]);
        MM_TRACE(e.tid == 0, TR_EEND, (w.it - static_cast<int>(blockIdx.x)) / static_cast<int>(gridDim.x));
        if (++ia == g.nacc) { ia = 0; pa ^= 1u; }
    }
    if (!waited) mm_pdl_wait();
    return ok;
}

// Codes of at most two bits from zero on, residual codes of at most two bits.
template <bool RES, int EW, bool SPLIT, bool F4, bool OFS, class Sums>
__device__ __forceinline__ bool epilogue_two_bits(const MmaArgs& g, const MmaEpi& e, const Sums& sums)
{
    if constexpr (!F4 || OFS) return epilogue_codes<2, RES ? 2 : 0, true, EW, SPLIT, F4, OFS>(g, e, sums);
    else if constexpr (SPLIT) return epilogue_tiles<RES, 1, EW, true>(g, e);       // one row tile
    else return g.PT > 1 ? epilogue_tiles<RES, 2, EW, false>(g, e) : epilogue_tiles<RES, 1, EW, false>(g, e);
}

// int32 accumulators out (and codes through the formula where both are asked for or the fast form does not apply).
template <int EW, bool SPLIT, bool F4, bool OFS, class Sums>
__device__ __forceinline__ bool epilogue_general(const MmaArgs& g, const MmaEpi& e, const Sums& sums)
{
    const int groups = g.TN >> 5;
    const float* cor = OFS ? reinterpret_cast<const float*>(e.smem + g.off_tab + g.TN * 8 + 64) : nullptr;
    int ia = 0, sum_o = -1;
    unsigned pa = 0;
    bool ok = true;
    mm_pdl_wait();
    for (MmaWalk w(g, SPLIT ? g.split_log : 0); w.m < g.tiles_m; w.next(g)) {
        const int o0 = w.o * g.TN, base = w.m * 128 * g.PT + e.row0;
        if (OFS && w.o != sum_o) {
            if (sum_o >= 0) asm volatile("bar.sync 2, %0;" ::"n"(EW * 32) : "memory");      // every warp is done with the old ones
            sums();
            asm volatile("bar.sync 2, %0;" ::"n"(EW * 32) : "memory");
            sum_o = w.o;
        }
        if (ok) ok = mm_wait(&e.full_acc[ia], pa);
        mm_fence_after();
        if (SPLIT && ok) ok = merge_partials<EW, F4>(g, e);
        MM_TRACE(e.tid == 0, TR_EBEG, (w.it - static_cast<int>(blockIdx.x)) / static_cast<int>(gridDim.x));
        const uint32_t acc = e.acc + static_cast<uint32_t>(ia * g.PT * g.TN);
        int t = 0, cc = e.set;
        while (cc >= groups) { cc -= groups; ++t; }
        for (; t < g.PT;) {
            const MmaPixel px = mma_pixel(g, base + t * 128);
            const int ob = o0 + cc * 32;
            const uint32_t col = acc + static_cast<uint32_t>(t * g.TN + cc * 32);
            const bool live = px.valid && ob < g.O;
            if (g.out_i32) {
                uint32_t v[32];
                mm_ld32(col, v);
                mm_ld_wait();
                mm_landed(v);
                if (F4)
#pragma unroll
                    for (int c = 0; c < 32; ++c) v[c] = acc_int(true, OFS ? __float_as_uint(__uint_as_float(v[c]) + cor[cc * 32 + c]) : v[c], 0u);
                if (g.flat && g.i32_nhwc) {
                    // The 32 x 32 block of the warp goes through 4 KB of shared memory so that a store writes a run of a row: 16 bytes a lane where rows
                    // are multiples of that, else 4 (a lane's own row, word by word, touches 32 lines a store: 4059 x 1382 x 1518: 62.6 -> 23.3 us).
                    uint4* sw = reinterpret_cast<uint4*>(e.smem + g.off_out + e.warp * 4096);
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        sw[e.lane * 8 + (c ^ (e.lane & 7))] = make_uint4(v[mma_column_of_filter(4 * c)], v[mma_column_of_filter(4 * c + 1)],
                                                                        v[mma_column_of_filter(4 * c + 2)], v[mma_column_of_filter(4 * c + 3)]);
                    __syncwarp();
                    const int r0 = base + t * 128 - e.lane;
                    if ((g.O & 3) != 0 || g.O - ob < 32) {
                        const uint32_t* words = reinterpret_cast<const uint32_t*>(sw);
                        int32_t* dst = g.out_i32 + static_cast<size_t>(r0) * g.O + ob + e.lane;
                        const int rows = min(32, g.total - r0);
#pragma unroll 8
                        for (int rr = 0; rr < rows; ++rr, dst += g.O)
                            if (ob + e.lane < g.O) *dst = static_cast<int32_t>(words[rr * 32 + ((e.lane >> 2) ^ (rr & 7)) * 4 + (e.lane & 3)]);
                    } else
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const int rr = k * 4 + (e.lane >> 3), ch = e.lane & 7;
                        const uint4 val = sw[rr * 8 + (ch ^ (rr & 7))];
                        if (r0 + rr < g.total) *reinterpret_cast<uint4*>(g.out_i32 + static_cast<size_t>(r0 + rr) * g.O + ob + ch * 4) = val;
                    }
                    __syncwarp();
                } else if (live) {
                    int32_t* dst = g.i32_nhwc ? g.out_i32 + static_cast<size_t>(px.pix) * g.O + ob
                                              : g.out_i32 + (static_cast<size_t>(px.n) * g.O + ob) * g.P * g.Q + px.rem;
                    const size_t step = g.i32_nhwc ? 1 : static_cast<size_t>(g.P) * g.Q;
#pragma unroll
                    for (int f = 0; f < 32; ++f)
                        if (ob + f < g.O) dst[f * step] = static_cast<int32_t>(v[mma_column_of_filter(f)]);
                }
                __syncwarp();
            }
            if (g.out_packed) epilogue_formula(g, col, live, px.pix, ob, 0u, OFS ? cor + cc * 32 : nullptr);
            cc += EW / 4;
            while (cc >= groups) { cc -= groups; ++t; }
        }
        mm_fence_before();
        __syncwarp();
        if (e.lane == 0) mm_arrive(&e.empty_acc[ia]);
        MM_TRACE(e.tid == 0, TR_EEND, (w.it - static_cast<int>(blockIdx.x)) / static_cast<int>(gridDim.x));
        if (++ia == g.nacc) { ia = 0; pa ^= 1u; }
    }
    return ok;
}

// ----------------------------------------------------------------------------- the kernel

// A: activation bits.  WB: 0 = prepared filters, 1..4 = packed filters of that many bits, expanded here.
// HALF: four epilogue and four expander warps in half an SM (two CTAs per SM, or one with room for the next layer's set-up beside
// it); otherwise eight + eight warps that own the SM.
template <bool HALF>
struct MmaShape {
    static constexpr int EW = HALF ? 4 : 8, XW = HALF ? 4 : 8, THREADS = (EW + XW + 2) * 32, CPS = HALF ? 2 : 1;
};

// SPLIT: an item belongs to a cluster of CTAs, each with a share of its chunks.  F4: nibbles (A and WB at most 3).  OFS: unsigned activations of three bits
// on nibbles enter as a - 4, the filters (packed, resident) give their sums.
template <int A, int WB, bool HALF, bool SPLIT, bool F4, bool OFS>
__global__ void __launch_bounds__(MmaShape<HALF>::THREADS, MmaShape<HALF>::CPS) bitserial_mma_kernel(const __grid_constant__ MmaArgs g)
{
    extern __shared__ __align__(1024) unsigned char mm_smem[];
    constexpr int XW = MmaShape<HALF>::XW, EW = MmaShape<HALF>::EW, NXT = XW * 32, NET = EW * 32;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);          // warp-uniform for the compiler: the roles below are not divergent code
    const uint32_t smem0 = smem_u32(mm_smem);
    uint64_t* bars = reinterpret_cast<uint64_t*>(mm_smem + g.off_bar);
    uint64_t* full_e = bars;            // [4]
    uint64_t* empty_e = bars + 4;       // [4]
    uint64_t* full_acc = bars + 8;      // [2]
    uint64_t* empty_acc = bars + 10;    // [2]
    uint64_t* wgt_full = bars + 12;
    uint64_t* bulk_full = bars + 13;
    uint64_t* full_p = bars + 14;       // [MM_STAGES] packed rows landed
    uint64_t* empty_p = bars + 22;      // [MM_STAGES] ... and expanded
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 30);
    int* fast_ok = reinterpret_cast<int*>(bars + 31);
    uint64_t* red_full = bars + 32;     // partial sums of a split item
    uint64_t* form_ok = bars + 33;      // prepared filters are in the form of this layer, or have been brought into it

    constexpr bool packed_b = WB > 0;
    constexpr int WBX = WB > 0 ? WB : 1;
    int* sums_i = reinterpret_cast<int*>(mm_smem + g.off_tab + g.TN * 8 + 64);
    const bool resident = g.nsb == 0;
    const bool stream_prepared = !resident && !packed_b;      // a stage then holds expanded pixels and the filters of the same chunk
    const int items = g.tiles_m * g.tiles_o;
    const int BM = 128 * g.PT;

    MM_TRACE(tid == 0, TR_START, 0);
    if (OFS)
        for (int c = tid; c < g.TN; c += MmaShape<HALF>::THREADS) sums_i[c] = 0;
    if (tid == 0) {
        for (int s = 0; s < 4; ++s) {
            mbar_init(&full_e[s], XW / g.groups + (stream_prepared ? 1 : 0));
            mbar_init(&empty_e[s], 1);
        }
        for (int s = 0; s < 2; ++s) { mbar_init(&full_acc[s], 1); mbar_init(&empty_acc[s], EW); }
        mbar_init(wgt_full, packed_b ? XW + EW : 1);
        mbar_init(bulk_full, 1);
        mbar_init(form_ok, 1);
        if (SPLIT) mbar_init(red_full, (g.split - 1) * EW);
        for (int s = 0; s < MM_STAGES; ++s) { mbar_init(&full_p[s], 1); mbar_init(&empty_p[s], XW / g.groups); }
        *fast_ok = 1;
        fence_barrier_init();
        fence_proxy_async();
    }
    constexpr int WARP_COPY = EW + XW, WARP_MMA = EW + XW + 1;
    if (warp == WARP_MMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(g.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        // Only now: a CTA of a later launch may take tensor memory as soon as it runs, and keeps it until every launch before it has ended.  Released
        // while this CTA still waits for its columns, the two could wait for each other.
        mm_pdl_release();
    }
    mm_fence_before();
    __syncthreads();
    mm_fence_after();
    if (SPLIT) mm_cluster_sync();      // the barriers of rank 0 are initialised
    const MmaChunks range(g, SPLIT);
    const int walk_log = SPLIT ? g.split_log : 0;
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);      // uniform for the compiler, as above
    MM_TRACE(tid == 0, TR_SETUP, 0);

    // a CTA with resident filters keeps its filter tile; otherwise the filter tile runs fastest over the items
    if (warp == WARP_COPY) {
        // ------------------------------------------------------------------ copy warp: prepared filters, and packed rows by TMA
        // One lane issues the copies; with prepared filters the others follow, in case they are in the other form.
        if (!packed_b || lane == 0) {
            bool waited = false, ok = true;
            const size_t blk_stride = static_cast<size_t>(g.opad) * g.RS * 32;
            const unsigned blk_bytes = static_cast<unsigned>(g.TN * g.RS * 32);
            const int o0 = static_cast<int>(blockIdx.x % static_cast<unsigned>(g.tiles_o)) * g.TN;       // of resident filters
            if (!packed_b || (resident && g.bulk_b)) {
                if (!g.early_b) { mm_pdl_wait(); waited = true; }
                if (resident && lane == 0) {
                    if (packed_b) {
                        // the packed tile parks in the ring of expanded pixels, which nobody uses yet
                        const int words = (g.O - o0 < g.TN ? g.O - o0 : g.TN) * g.RS * g.Cw * WBX;
                        mbar_expect_tx(bulk_full, static_cast<unsigned>(words) * 4u);
                        mm_bulk(mm_smem + g.off_e, g.wgt_packed + static_cast<size_t>(o0) * g.RS * g.Cw * WBX, static_cast<unsigned>(words) * 4u, bulk_full);
                    } else {
                        const int8_t* src = g.wgt + static_cast<size_t>(o0) * g.RS * 32;
                        mbar_expect_tx(wgt_full, blk_bytes * g.nblk);
                        for (int b = 0; b < g.nblk; ++b) mm_bulk(mm_smem + static_cast<size_t>(b) * blk_bytes, src + b * blk_stride, blk_bytes, wgt_full);
                    }
                }
            }
            // The form is read beside the first copies, which are made as if it were the expected one: nothing waits for it that would not wait
            // for them.  Otherwise what has landed is overwritten before the MMAs may begin.
            uint32_t mark = 0;
            if (!packed_b) asm volatile("ld.global.b32 %0, [%1];" : "=r"(mark) : "l"(g.wgt + blk_stride * g.Cw - 4) : "memory");
            bool first = !packed_b, other = false;
            auto check_form = [&](uint64_t* landed, int o, int b0, int nb) {
                other = (mark == MM_NIBBLE_MARK) != F4;
                if (other) {
                    if (ok) ok = mm_wait(landed, 0);
                    convert_filters<F4>(g, mm_smem, o, b0, nb, lane);
                }
                if (lane == 0) mm_arrive(form_ok);
                first = false;
            };
            const bool stream = stream_prepared;
            if (stream || g.tma) {
                int ib = 0, ip = 0;
                unsigned pb = 0, pp = 0;
                for (MmaWalk w(g, walk_log); w.m < g.tiles_m && ok; w.next(g)) {
                    const int8_t* src = g.wgt + static_cast<size_t>(w.o) * g.TN * g.RS * 32;
                    for (int c = range.beg; c < range.beg + range.n && ok; ++c) {
                        const int step = F4 ? g.units : g.units * 2, b0 = c * step;
                        const int nb = g.nblk - b0 < step ? g.nblk - b0 : step;
                        if (stream) {
                            ok = mm_wait(&empty_e[ib], pb ^ 1u);
                            if (!ok) break;
                            unsigned char* dst = mm_smem + static_cast<size_t>(ib) * g.b_bytes;
                            if (other) {
                                convert_filters<F4>(g, dst, w.o * g.TN, b0, nb, lane);
                                if (lane == 0) mm_arrive(&full_e[ib]);
                            } else if (lane == 0) {
                                mbar_expect_tx(&full_e[ib], blk_bytes * nb);
                                for (int b = 0; b < nb; ++b) mm_bulk(dst + static_cast<size_t>(b) * blk_bytes, src + (b0 + b) * blk_stride, blk_bytes, &full_e[ib]);
                            }
                            if (++ib == g.nse) { ib = 0; pb ^= 1u; }
                        }
                        if (g.tma) {
                            if (!waited) { mm_pdl_wait(); waited = true; }
                            ok = mm_wait(&empty_p[ip], pp ^ 1u);
                            if (!ok) break;
                            if (lane == 0) {
                                const bool fb = packed_b && !resident;
                                mbar_expect_tx(&full_p[ip], static_cast<unsigned>(BM * g.rowA + (fb ? g.TN * g.rowB : 0)));
                                unsigned char* dst = mm_smem + g.off_stg + ip * g.stg_bytes;
                                const int rows = BM < 256 ? BM : 256;
                                for (int r = 0; r < BM; r += rows) tma_load_2d(dst + r * g.rowA, &g.tmA, &full_p[ip], c * (g.rowA >> 2), w.m * BM + r);
                                if (fb) tma_load_2d(mm_smem + g.off_bstg + ip * g.bstg_bytes, &g.tmB, &full_p[ip], c * (g.rowB >> 2), w.o * g.TN);
                            }
                            if (++ip == g.nsp) { ip = 0; pp ^= 1u; }
                        }
                        if (first) check_form(resident ? wgt_full : &full_e[0], resident ? o0 : w.o * g.TN, resident ? 0 : b0, resident ? g.nblk : nb);
                    }
                }
            }
            if (first && resident && ok) check_form(wgt_full, o0, 0, g.nblk);
            if (!ok && lane == 0) atomicOr(g.status, STATUS_TIMEOUT);
        }
        __syncwarp();
    } else if (warp == WARP_MMA) {
        // ------------------------------------------------------------------ MMA issuer (all lanes in step)
        const MmaIssue m{full_e, empty_e, full_acc, empty_acc, wgt_full, packed_b ? nullptr : form_ok, smem0, tmem, items, resident};
        if (g.R == 1) issue_items<TAPS_1, SPLIT, F4>(g, m);
        else if (g.R == 3 && g.stride == 1) issue_items<TAPS_3S1, SPLIT, F4>(g, m);
        else if (g.R == 3 && g.pad == 1) issue_items<TAPS_3S2, SPLIT, F4>(g, m);
        else issue_items<TAPS_ANY, SPLIT, F4>(g, m);
    } else if (warp >= EW && warp < WARP_COPY) {
        // ------------------------------------------------------------------ expanders
        const int xt = tid - NET;
        if (packed_b && resident) {
            if (!g.early_b) mm_pdl_wait();
            const int o0 = static_cast<int>(blockIdx.x % static_cast<unsigned>(g.tiles_o)) * g.TN;
            const uint32_t* src = g.wgt_packed + static_cast<size_t>(o0) * g.RS * g.Cw * WBX;
            if (g.bulk_b) {
                if (!mm_wait(bulk_full, 0)) atomicOr(g.status, STATUS_TIMEOUT);
                src = reinterpret_cast<const uint32_t*>(mm_smem + g.off_e);
            }
            expand_filters_resident<WBX, F4, OFS>(g, smem0, src, o0, tid, NXT + NET, sums_i);
            fence_proxy_async();
            // the parked tile has been read: the ring may be filled once every warp is here
            asm volatile("bar.sync 4, %0;" ::"n"(NXT + NET) : "memory");
            __syncwarp();
            if (lane == 0) mm_arrive(wgt_full);
        }
        // A chunk belongs to one group of warps.  The waits, the fence and the arrival of a chunk take several hundred cycles whatever its
        // size; with several groups they overlap (see make_plan for how many).
        const int G = g.groups, nx = NXT / G, xg = xt / nx, xl = xt - xg * nx;
        // bipolar filters of an odd number of channel words: the second half of the last K step of nibbles has to be zero, not -1
        const bool odd_tail = F4 && g.w_kind == 2 && (g.Cw & 1);
#ifdef BS_TRACE
        int xseq = 0;
#endif
        if (g.tma) {
            mm_pdl_wait();
            MM_TRACE(xt == 0, TR_PDL, 0);
            // Flat tiles: the copy warp fetches boxes of [row][units] with TMA (a thread-by-thread copy touches one 128-byte line per
            // lane: 32 tag cycles per instruction, a thousand cycles per 256 rows of 128 channels).  Items (unit, row), row
            // fastest; the 16-byte pieces of a row are swizzled by the box so that 32 rows read without bank conflicts.
            const bool stream_b = packed_b && !resident;
            const int rowsA = BM, shA = 31 - __clz(BM), shB = 31 - __clz(g.TN);
            int idx = xg, ip = xg;
            unsigned phase = 0, pp = 0;
            bool ok = true;
            const uint32_t g16 = static_cast<uint32_t>(g.NI) * 16u;
            int c = xg;
            MmaWalk w(g, walk_log);
            while (c >= range.n) { c -= range.n; w.next(g); }
            while (w.m < g.tiles_m) {
                {
                    MM_TRACE(xt == 0, TR_XWAIT, xseq);
                    ok = mm_wait(&full_p[ip], pp);
                    if (ok) ok = mm_wait(&empty_e[idx], phase ^ 1u);
                    if (!ok) break;
                    MM_TRACE(xt == 0, TR_XBEG, xseq);
                    const int nu = min(g.units, g.nunits - (range.beg + c) * g.units);
                    const uint32_t src = smem0 + g.off_stg + static_cast<uint32_t>(ip * g.stg_bytes);
                    const uint32_t e0 = smem0 + g.off_e + static_cast<uint32_t>(idx * g.e_bytes);
                    // two rows at a time: the second one's words are on their way while the first is expanded
                    for (int it = xl; it < nu << shA; it += 2 * nx) {
                        const int u0 = it >> shA, i0 = it & (rowsA - 1), u1 = (it + nx) >> shA, i1 = (it + nx) & (rowsA - 1);
                        const bool two = it + nx < nu << shA;
                        uint32_t wa[2 * A], wb[2 * A];
                        load_row_unit<A>(src, i0 * g.rowA + u0 * 8 * A, g.swzA, wa);
                        if (two) load_row_unit<A>(src, i1 * g.rowA + u1 * 8 * A, g.swzA, wb);
                        expand_unit<A, F4>(wa, g.a_kind, e0 + static_cast<uint32_t>(u0) * (F4 ? 2u : 4u) * g16 + static_cast<uint32_t>(i0) * 16u, g16, false);
                        if (two) expand_unit<A, F4>(wb, g.a_kind, e0 + static_cast<uint32_t>(u1) * (F4 ? 2u : 4u) * g16 + static_cast<uint32_t>(i1) * 16u, g16, false);
                    }
                    if (stream_b) {
                        const uint32_t bsrc = smem0 + g.off_bstg + static_cast<uint32_t>(ip * g.bstg_bytes);
                        const uint32_t bdst = smem0 + static_cast<uint32_t>(idx * g.b_bytes), blk = static_cast<uint32_t>(g.TN) * 32u;
                        for (int it = xl; it < nu << shB; it += nx) {
                            const int u = it >> shB, i = it & (g.TN - 1);
                            const int f = (i & ~31) + mma_filter_of_column(i & 31);
                            uint32_t wd[2 * WBX];
                            load_row_unit<WBX>(bsrc, f * g.rowB + u * 8 * WBX, g.swzB, wd);
                            const bool live = w.o * g.TN + f < g.O, both = !odd_tail || (range.beg + c) * g.units + u + 1 < g.nunits;
                            const uint32_t d = bdst + static_cast<uint32_t>(F4 ? u : 2 * u) * blk + static_cast<uint32_t>(i >> 3) * 256u + static_cast<uint32_t>(i & 7) * 16u;
                            expand_filter_word<WBX, F4>(wd, g.w_kind, live, d);
                            expand_filter_word<WBX, F4>(wd + WBX, g.w_kind, live && both, d + (F4 ? 128u : blk));
                        }
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) { mm_arrive(&full_e[idx]); mm_arrive(&empty_p[ip]); }
#ifdef BS_TRACE
                    MM_TRACE(xt == 0, TR_XEND, xseq);
                    ++xseq;
#endif
                    idx += G;
                    if (idx >= g.nse) { idx -= g.nse; phase ^= 1u; }
                    ip += G;
                    if (ip >= g.nsp) { ip -= g.nsp; pp ^= 1u; }
                    c += G;
                    while (c >= range.n) { c -= range.n; w.next(g); }
                }
            }
            if (!ok && lane == 0) atomicOr(g.status, STATUS_TIMEOUT);
        } else {
        // Packed words travel through a group's own stages of shared memory, one chunk (and one cp.async group) each, issued as many of
        // its chunks ahead as it has stages.  A thread copies and later expands the same items, so nothing needs a barrier.
        const bool stream_b = packed_b && !resident;
        const int rec = g.Cw * A, rows = g.TN * g.RS;
        constexpr int stages = 2;
        const uint32_t stg0 = smem0 + g.off_stg + static_cast<uint32_t>(xg * stages * g.stg_bytes + xl * g.psz);
        const uint32_t bstg0 = smem0 + g.off_bstg + static_cast<uint32_t>(xg * stages * g.bstg_bytes + xl * g.bpsz);
        const uint32_t step = static_cast<uint32_t>(g.nslots * nx * g.psz), bstep = static_cast<uint32_t>(g.bslots * nx * g.bpsz);
        const uint32_t rel0 = smem0 + g.off_pix, pix0 = rel0 + static_cast<uint32_t>((1 + xg * (stages + 1)) * g.NI) * 4u, brow0 = smem0 + g.off_brow;
        // Where row i of a halo sits relative to the halo's first position: rows and columns of the position grid, parity plane.
        // Found once per kernel; a tile adds its own origin.
        for (int i = xt; i < g.NI && !g.flat; i += NXT) {
            int h = i, pl = 0;
            if (g.nplanes > 1) {
                pl = (i >= g.HL) + (i >= 2 * g.HL) + (i >= 3 * g.HL);
                h = i - pl * g.HL;
            }
            const int hq = fdiv(h, g.d_pitch), hr = h - hq * g.d_pitch.d;
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(rel0 + static_cast<uint32_t>(i) * 4u), "r"((static_cast<uint32_t>(pl) << 30) | static_cast<uint32_t>((hq << 15) | hr)) : "memory");
        }
        // Packed record of filter row i: filter of the tile in the top byte, record below it (taps and tile filters number at most 2^14).
        if (stream_b && g.units == 1)
            for (int i = xt; i < rows; i += NXT) {
                int off;
                const int f = filter_row(g, i, 1, off);
                asm volatile("st.shared.b32 [%0], %1;" ::"r"(brow0 + static_cast<uint32_t>(i) * 4u), "r"((static_cast<uint32_t>(f) << 24) | static_cast<uint32_t>(off / g.Cw)) : "memory");
            }
        if (g.units > 1 || G > 1) asm volatile("bar.sync 3, %0;" ::"n"(NXT) : "memory");      // other threads' entries are read
        MmaWalk iw(g, walk_log);
        int ic = xg, ibuf = 0, iitem = -1, itab = 0;
        while (ic >= range.n) { ic -= range.n; iw.next(g); }
        int lc = ic, litem = -1, ltab = 0;
        MmaWalk lw = iw;
        int oy = 0, ox = 0, on = 0, ostrip = 0;              // origin of a halo: row, column, image, strip
        const int PH = g.img_rows;
        auto origin = [&](int m) {
            // (image, strip) and row of the first position; a halo may start above the first image
            const int b0 = m * BM + g.hstart + g.d_img.d;
            const int u = fdiv(b0, g.d_img), rem = b0 - u * g.d_img.d;
            oy = fdiv(rem, g.d_pitch);
            ox = rem - oy * g.d_pitch.d;
            on = fdiv(u - 1 < 0 ? 0 : u - 1, g.d_strips);
            ostrip = u - 1 - on * g.d_strips.d;
        };
        // input pixel of row i of the halo at the origin; -1: padding
        auto halo_pixel = [&](int i) -> int {
            uint32_t e;
            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(e) : "r"(rel0 + static_cast<uint32_t>(i) * 4u));
            int x = ox + static_cast<int>(e & 0x7FFFu), y = oy + static_cast<int>((e >> 15) & 0x7FFFu);
            if (x >= g.d_pitch.d) { x -= g.d_pitch.d; ++y; }
            int n = on, strip = ostrip;
            while (y >= PH) { y -= PH; if (++strip == g.d_strips.d) { strip = 0; ++n; } }
            const int Y = y * g.stride + static_cast<int>(e >> 31), X = (x + g.xoff + strip * g.strip_q) * g.stride + static_cast<int>((e >> 30) & 1u);
            const bool in = n < g.N && strip >= 0 && Y < g.H && static_cast<unsigned>(X) < static_cast<unsigned>(g.W);
            return in ? (n * g.H + Y) * g.W + X : -1;
        };
        auto flat_pixel = [&](int m, int i) -> int { return m * BM + i < g.total ? m * BM + i : -1; };
        // The pixels of a thread's rows are found one chunk before their copies are issued, the first ones while the preceding kernel
        // still runs, and kept in shared memory for all chunks of the item: about 40 instructions a row that would otherwise
        // stand in front of every chunk's copies (a thousand cycles a chunk, more than the MMAs of 64 channels take).
        auto locate = [&]() {
            if (g.flat || g.units > 1) return;
            if (lw.m < g.tiles_m && lw.it != litem) {
                litem = lw.it;
                origin(lw.m);
                const uint32_t t = pix0 + static_cast<uint32_t>(ltab * g.NI) * 4u;
                for (int i = xl; i < g.NI; i += nx) asm volatile("st.shared.b32 [%0], %1;" ::"r"(t + static_cast<uint32_t>(i) * 4u), "r"(halo_pixel(i)) : "memory");
                if (++ltab > stages) ltab = 0;
            }
            lc += G;
            while (lc >= range.n) { lc -= range.n; lw.next(g); }
        };
        uint32_t ipix = 0;
        auto issue = [&]() {
            if (iw.m < g.tiles_m) {
                if (iw.it != iitem) {
                    iitem = iw.it;
                    if (g.units > 1 && !g.flat) origin(iw.m);
                    ipix = pix0 + static_cast<uint32_t>(itab * g.NI) * 4u;
                    if (++itab > stages) itab = 0;
                }
                uint32_t dst = stg0 + static_cast<uint32_t>(ibuf * g.stg_bytes);
                const int chunk = range.beg + ic;
                if (g.units == 1) {
                    const int left = (g.Cw - 2 * chunk) * A;
                    const uint32_t* src = g.act + 2 * chunk * A;
                    for (int i = xl; i < g.NI; i += nx, dst += nx * g.psz) {
                        int pixel;
                        if (g.flat) pixel = flat_pixel(iw.m, i);
                        else asm volatile("ld.shared.b32 %0, [%1];" : "=r"(pixel) : "r"(ipix + static_cast<uint32_t>(i) * 4u));
                        stage_unit<A>(g.psz, dst, step, src + static_cast<size_t>(static_cast<unsigned>(pixel < 0 ? 0 : pixel)) * rec, g.act, pixel >= 0 ? left : 0, F4 && g.one_word);
                    }
                } else {
                    // items (unit, pixel), pixel fastest
                    int u = 0, i = xl;
                    while (i >= g.NI) { i -= g.NI; ++u; }
                    for (; u < g.units; dst += nx * g.psz) {
                        const int pixel = g.flat ? flat_pixel(iw.m, i) : halo_pixel(i), unit = chunk * g.units + u;
                        stage_unit<A>(g.psz, dst, step, g.act + static_cast<size_t>(static_cast<unsigned>(pixel < 0 ? 0 : pixel)) * rec + 2 * unit * A, g.act,
                                      pixel >= 0 ? (g.Cw - 2 * unit) * A : 0);
                        i += nx;
                        while (i >= g.NI) { i -= g.NI; ++u; }
                    }
                }
                if (stream_b) {
                    const uint32_t* base = g.wgt_packed + static_cast<size_t>(iw.o) * g.TN * g.RS * g.Cw * WBX;
                    const int o0 = iw.o * g.TN;
                    dst = bstg0 + static_cast<uint32_t>(ibuf * g.bstg_bytes);
                    if (g.units == 1) {
                        const int left = (g.Cw - 2 * chunk) * WBX;
                        const uint32_t* src = base + 2 * chunk * WBX;
                        for (int i = xl; i < rows; i += nx, dst += nx * g.bpsz) {
                            uint32_t e;
                            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(e) : "r"(brow0 + static_cast<uint32_t>(i) * 4u));
                            const bool live = o0 + static_cast<int>(e >> 24) < g.O;
                            stage_unit<WBX>(g.bpsz, dst, bstep, src + (e & 0xFFFFFFu) * static_cast<unsigned>(g.Cw * WBX), g.wgt_packed, live ? left : 0);
                        }
                    } else {
                        int u = 0, i = xl;
                        while (i >= rows) { i -= rows; ++u; }
                        for (; u < g.units; dst += nx * g.bpsz) {
                            int off;
                            const bool live = o0 + filter_row(g, i, WBX, off) < g.O;
                            const int unit = chunk * g.units + u;
                            stage_unit<WBX>(g.bpsz, dst, bstep, base + off + 2 * unit * WBX, g.wgt_packed, live ? (g.Cw - 2 * unit) * WBX : 0);
                            i += nx;
                            while (i >= rows) { i -= rows; ++u; }
                        }
                    }
                }
                ic += G;
                while (ic >= range.n) { ic -= range.n; iw.next(g); }
            }
            cp_async_commit();
            if (++ibuf == stages) ibuf = 0;
        };
        int buf = 0, idx = xg;
        unsigned phase = 0;
        bool ok = true;
        for (int s = 0; s <= stages; ++s) locate();
        mm_pdl_wait();
        MM_TRACE(xt == 0, TR_PDL, 0);
        for (int s = 0; s < stages; ++s) issue();
        MmaWalk w(g, walk_log);
        int c = xg;
        while (c >= range.n) { c -= range.n; w.next(g); }
        while (w.m < g.tiles_m) {
            {
                asm volatile("cp.async.wait_group %0;" ::"n"(stages - 1) : "memory");
                MM_TRACE(xt == 0, TR_XWAIT, xseq);
                if (ok) ok = mm_wait(&empty_e[idx], phase ^ 1u);
                MM_TRACE(xt == 0, TR_XBEG, xseq);
                const int nu = min(g.units, g.nunits - (range.beg + c) * g.units);
                const uint32_t g16 = static_cast<uint32_t>(g.NI) * 16u;
                uint32_t src = stg0 + static_cast<uint32_t>(buf * g.stg_bytes);
                const uint32_t e0 = smem0 + g.off_e + static_cast<uint32_t>(idx * g.e_bytes);
                if (g.units == 1) {
                    uint32_t dst = e0 + static_cast<uint32_t>(xl) * 16u;
                    for (int i = xl; i < g.NI; i += nx, src += nx * g.psz, dst += nx * 16) {
                        uint32_t wd[2 * A];
                        load_unit<A>(src, step, g.psz, wd, F4 && g.one_word);
                        expand_unit<A, F4>(wd, g.a_kind, dst, g16, F4 && g.one_word);
                    }
                } else {
                    int u = 0, i = xl;
                    while (i >= g.NI) { i -= g.NI; ++u; }
                    for (; u < nu; src += nx * g.psz) {
                        uint32_t wd[2 * A];
                        load_unit<A>(src, step, g.psz, wd);
                        expand_unit<A, F4>(wd, g.a_kind, e0 + static_cast<uint32_t>(u) * (F4 ? 2u : 4u) * g16 + static_cast<uint32_t>(i) * 16u, g16, false);
                        i += nx;
                        while (i >= g.NI) { i -= g.NI; ++u; }
                    }
                }
                if (stream_b) {
                    src = bstg0 + static_cast<uint32_t>(buf * g.bstg_bytes);
                    const uint32_t bdst = smem0 + static_cast<uint32_t>(idx * g.b_bytes), blk = static_cast<uint32_t>(rows) * 32u;
                    const bool all_live = (w.o + 1) * g.TN <= g.O;
                    int u = 0, i = xl;
                    while (i >= rows) { i -= rows; ++u; }
                    for (; u < nu; src += nx * g.bpsz) {
                        uint32_t wd[2 * WBX];
                        load_unit<WBX>(src, bstep, g.bpsz, wd);
                        bool live = true;
                        int off;
                        if (!all_live) live = w.o * g.TN + filter_row(g, i, WBX, off) < g.O;
                        const bool both = !odd_tail || (range.beg + c) * g.units + u + 1 < g.nunits;
                        const uint32_t d = bdst + static_cast<uint32_t>(F4 ? u : 2 * u) * blk + static_cast<uint32_t>(i >> 3) * 256u + static_cast<uint32_t>(i & 7) * 16u;
                        expand_filter_word<WBX, F4>(wd, g.w_kind, live, d);
                        expand_filter_word<WBX, F4>(wd + WBX, g.w_kind, live && both, d + (F4 ? 128u : blk));
                        i += nx;
                        while (i >= rows) { i -= rows; ++u; }
                    }
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mm_arrive(&full_e[idx]);
#ifdef BS_TRACE
                MM_TRACE(xt == 0, TR_XEND, xseq);
                ++xseq;
#endif
                issue();                       // into the stage just read
                locate();
                idx += G;
                if (idx >= g.nse) { idx -= g.nse; phase ^= 1u; }
                if (++buf == stages) buf = 0;
                c += G;
                while (c >= range.n) { c -= range.n; w.next(g); }
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        if (!ok) atomicOr(g.status, STATUS_TIMEOUT);
        }
    } else if (warp < EW) {
        // ------------------------------------------------------------------ epilogue
        const int quad = warp & 3, set = warp >> 2;
        const uint32_t lane_addr = static_cast<uint32_t>(quad * 32) << 16;
        if (F4) {           // scale factors of 2 for every row, column and block
            for (int c = set * 8; c < MM_SF_COLS; c += 8 * (EW / 4)) mm_st8(tmem + lane_addr + static_cast<uint32_t>(g.sf_col + c), 0x80808080u);
            mm_st_wait();
        } else if (g.preset) {
            for (int c = set * 8; c < g.tmem_cols; c += 8 * (EW / 4)) mm_st8(tmem + lane_addr + static_cast<uint32_t>(c), MM_PRESET);
            mm_st_wait();
        }
        mm_fence_before();
        __syncwarp();
        if (lane == 0) { mm_arrive(&empty_acc[0]); if (g.nacc > 1) mm_arrive(&empty_acc[1]); }
        if (packed_b && resident) {
            if (!g.early_b) mm_pdl_wait();
            const int o0 = static_cast<int>(blockIdx.x % static_cast<unsigned>(g.tiles_o)) * g.TN;
            const uint32_t* src = g.wgt_packed + static_cast<size_t>(o0) * g.RS * g.Cw * WBX;
            if (g.bulk_b) {
                if (!mm_wait(bulk_full, 0)) atomicOr(g.status, STATUS_TIMEOUT);
                src = reinterpret_cast<const uint32_t*>(mm_smem + g.off_e);
            }
            expand_filters_resident<WBX, F4, OFS>(g, smem0, src, o0, tid, NXT + NET, sums_i);
            fence_proxy_async();
            // the parked tile has been read: the ring may be filled once every warp is here
            asm volatile("bar.sync 4, %0;" ::"n"(NXT + NET) : "memory");
            __syncwarp();
            if (lane == 0) mm_arrive(wgt_full);
        }
        if (!g.early_b) mm_pdl_wait();
        MmaEpi e;
        e.smem = mm_smem; e.full_acc = full_acc; e.empty_acc = empty_acc; e.fast_ok = fast_ok;
        e.acc = tmem + lane_addr; e.row0 = quad * 32 + lane; e.set = set;
        e.tid = tid; e.lane = lane; e.warp = warp; e.red_full = red_full;
        // what the epilogue adds to the accumulators of a filter: four times the sum of its codes
        auto sums = [&]() {
            if constexpr (OFS)
                for (int c = tid; c < g.TN; c += NET) reinterpret_cast<float*>(sums_i)[c] = 4.0f * static_cast<float>(sums_i[c]);
        };
        bool ok;
        if (SPLIT && range.rank > 0) ok = send_partials<EW, F4>(g, e, range.rank);
        else if (!g.preset) ok = epilogue_general<EW, SPLIT, F4, OFS>(g, e, sums);
        else if (g.epi == 0) ok = epilogue_two_bits<false, EW, SPLIT, F4, OFS>(g, e, sums);
        else if (g.epi == 1) ok = epilogue_two_bits<true, EW, SPLIT, F4, OFS>(g, e, sums);
        else if (g.epi == 2) ok = epilogue_codes<4, 0, true, EW, SPLIT, F4, OFS>(g, e, sums);
        else if (g.epi == 3) ok = epilogue_codes<4, 4, true, EW, SPLIT, F4, OFS>(g, e, sums);
        else if (g.epi == 4) ok = epilogue_codes<4, 0, false, EW, SPLIT, F4, OFS>(g, e, sums);
        else ok = epilogue_codes<4, 4, false, EW, SPLIT, F4, OFS>(g, e, sums);
        if (!ok && lane == 0) atomicOr(g.status, STATUS_TIMEOUT);
    }
    mm_fence_before();
    __syncthreads();
    if (SPLIT) mm_cluster_sync();      // shared memory of rank 0 stays until everything sent has arrived
    MM_TRACE(tid == 0, TR_END, 0);
    if (warp == WARP_MMA) {
        mm_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(g.tmem_cols) : "memory");
    }
}

typedef void (*MmaKernel)(MmaArgs);

// The instantiations for A activation bits, a translation unit each (mma_inst_a*.cu; nibbles: mma_inst_f*.cu): filters prepared (wb = 0)
// or packed in wb bits, half an SM or a whole one per CTA, a whole one with the item split over a cluster; offset: unsigned activations of three bits.
MmaKernel mma_kernel_a1(int wb, bool half, bool split);
MmaKernel mma_kernel_a2(int wb, bool half, bool split);
MmaKernel mma_kernel_a3(int wb, bool half, bool split);
MmaKernel mma_kernel_a4(int wb, bool half, bool split);
MmaKernel mma_kernel_f1(int wb, bool half, bool split);
MmaKernel mma_kernel_f2(int wb, bool half, bool split);
MmaKernel mma_kernel_f3(int wb, bool half, bool split, bool offset);

template <int A, int WB, bool F4>
MmaKernel mma_pick_shape(bool half, bool split)
{
    return split ? bitserial_mma_kernel<A, WB, false, true, F4, false> : half ? bitserial_mma_kernel<A, WB, true, false, F4, false>
                                                                              : bitserial_mma_kernel<A, WB, false, false, F4, false>;
}
// (resident filters are not split)
template <int WB>
MmaKernel mma_pick_offset(bool half) { return half ? bitserial_mma_kernel<3, WB, true, false, true, true> : bitserial_mma_kernel<3, WB, false, false, true, true>; }
template <int A>
MmaKernel mma_pick(int wb, bool half, bool split)
{
    switch (wb) {
        case 0: return mma_pick_shape<A, 0, false>(half, split);
        case 1: return mma_pick_shape<A, 1, false>(half, split);
        case 2: return mma_pick_shape<A, 2, false>(half, split);
        case 3: return mma_pick_shape<A, 3, false>(half, split);
        default: return mma_pick_shape<A, 4, false>(half, split);
    }
}
template <int A>
MmaKernel mma_pick_nibbles(int wb, bool half, bool split)
{
    switch (wb) {
        case 0: if constexpr (A <= 2) return mma_pick_shape<A, 0, true>(half, split); else return nullptr;        // prepared filters are int8 there
        case 1: return mma_pick_shape<A, 1, true>(half, split);
        case 2: return mma_pick_shape<A, 2, true>(half, split);
        default: return mma_pick_shape<A, 3, true>(half, split);
    }
}

}  // namespace bs
