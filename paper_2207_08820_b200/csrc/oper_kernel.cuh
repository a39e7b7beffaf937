// Layers of a bound sequence on operand tensors: activations that stay on the device as nibbles in the order the tensor cores read them.
//
// Inside a sequence the layer that writes a tensor can write, beside its packed codes, what the next layer's tensor-core operand will be: 32
// channels of a position as 16 bytes, [32-channel group][position][16 bytes], positions numbered as the accumulator rows of the reading
// layer are (mma_kernel.cuh: rows of an image with the zero padding between them as positions of their own, stride 2 a plane
// per parity).  The pixels of any tile and their halo are then one run of memory per channel group, so a layer has nothing to expand, no pixel
// to locate and no thread that copies: one warp fetches runs by bulk copies, one warp issues MMAs, eight warps requantise.
//
// What bounds it: the turn of MMAs and epilogue, and the start of a launch (a 56 x 56 layer of 64 images: 1000 cycles of MMA issue and 1800 to 2500 of
// epilogue an item, three items, 4000 cycles from a CTA's start to its first MMA; without its stores 5 %, without reads of scales 7 % faster).
// Half an SM's shared memory and tensor memory per CTA, so that two CTAs overlap each other's MMAs and epilogues, or the next layer's CTA sets up
// and fetches its filters beside the last one of this layer.
// Layers one after the other, calls on packed codes -> on operand tensors, us: 64 images, 64 channels of 56 x 56, 3 x 3: 13.4 -> 8.8, with a residual
// 15.1 -> 10.1; 256 of 14 x 14: 9.2 -> 6.3; one image of the former 3.7 -> 2.5; 512 of 7 x 7: 6.9 -> 4.6.
#pragma once
#include "mma_kernel.cuh"

namespace bs {

constexpr int OP_STAGES = 8, OP_EW = 8;         // stages at most; epilogue warps of an item
// FULL: one CTA per SM with all its tensor memory, 16 epilogue warps, of which eight take every other item.
constexpr int oper_threads(bool full) { return ((full ? 2 : 1) * OP_EW + 2) * 32; }

struct OperArgs {
    const unsigned char* src;       // operand tensor of the input, at the first halo position of tile 0 (of plane 0, group 0)
    long long src_group, src_plane; // bytes between channel groups, parity planes
    const int8_t* wgt;              // prepared filters (nibbles) [C/64][filters, padded to 128][R*S][32 bytes]
    uint32_t* out_packed;
    OperDst dst1, dst2;             // operand tensors of the output for readers of stride 1, of stride 2
    const float* scale;
    const float* bias;
    const uint32_t* residual;
    int* status;
    float res_scale, acc_bound;
    int N, O, R, RS, P, Q, stride, pad, Cw, opad;
    int relu, out_bits, out_sign, out_cw_off, out_cw_total;
    int res_bits, res_sign, res_c_off, res_cw_total;
    // positions
    int total, pitch, HL, nplanes, NI;      // positions, positions of a row, halo positions per plane and in all planes
    int rmin, smin;
    FastDiv d_img, d_pitch;
    // tiling
    int TN, PT, units, nunits, nchunks;     // filters and row tiles per item, K steps (64 channels) per chunk / in all
    int tiles_m, tiles_o, step_m;           // a CTA keeps its filter tile and walks pixel tiles m, m + step_m, ..
    int nse, resident;                      // stages; filters resident or in the stages
    int halves;                             // channel groups of a K step: 2, or 1 where there is one group in all (LBO 0: its second half meets zero filters)
    int a_bytes, stage_bytes;               // pixels of a stage, a stage
    int off_stage, off_tab, off_bar;
    int tmem_cols, nacc, sf_col;
    int early_b;                            // filters, scale and bias may be read before the preceding kernel has finished
    unsigned idesc;
};

// ----------------------------------------------------------------------------- epilogue

struct OperPos { int pix, at1, at2; };       // output pixel (-1: none), positions in the operand tensors of the output

__device__ __forceinline__ OperPos oper_position(const OperArgs& g, int pos)
{
    OperPos o;
    const int n = fdiv(pos, g.d_img), rem = pos - n * g.d_img.d, y = fdiv(rem, g.d_pitch), x = rem - y * g.d_pitch.d;
    o.pix = pos < g.total && y < g.P && x < g.Q ? (n * g.P + y) * g.Q + x : -1;
    o.at1 = oper_at1(g.dst1, n, y, x);
    o.at2 = oper_at2(g.dst2, n, y, x);
    return o;
}

// Codes of 32 filters from ob on: e, d = codes of the even and the odd filters, two bits each.
__device__ __forceinline__ void oper_store(const OperArgs& g, const OperPos& o, int ob, uint32_t e, uint32_t d)
{
    uint32_t ow[4] = {(e & 0x55555555u) | ((d << 1) & 0xAAAAAAAAu), ((e >> 1) & 0x55555555u) | (d & 0xAAAAAAAAu), 0u, 0u};
    store_codes(g, o.pix, ob, ow);
    oper_put(g.dst1, g.dst2, ob >> 5, o.at1, o.at2, e, d);
}

// An item through the documented formula, one output at a time (scales and biases outside the range of the fast form).
static __device__ __noinline__ void oper_item_formula(const OperArgs& g, uint32_t acc, int base, int o0, int set)
{
    const int groups = g.TN >> 5;
    for (int u = set; u < g.PT * groups; u += OP_EW / 4) {
        const int t = u / groups, cc = u - t * groups, ob = o0 + cc * 32;
        const OperPos px = oper_position(g, base + t * 128);
        uint32_t v[32];
        mm_ld32(acc + static_cast<uint32_t>(t * g.TN + cc * 32), v);
        mm_ld_wait();
        mm_landed(v);
        if (px.pix >= 0 && ob < g.O) {
            uint32_t rw[4] = {0, 0, 0, 0}, ow[4] = {0, 0, 0, 0};
            for (int c = 0; c < 32; ++c) v[c] = acc_int(true, v[c], 0u);
            if (g.residual) load_residual(g, px.pix, ob, rw);
            requant32_formula(g, v, ob, rw, ow);
            uint32_t even, odd;
            oper_pairs(ow[0], ow[1], even, odd);
            oper_store(g, px, ob, even, odd);
        }
        __syncwarp();
    }
}

// As epilogue_tiles (mma_kernel.cuh): NT row tiles share the loads of scales and biases, eight columns of each on their way while eight are computed.
template <bool RES, int NT, bool FULL>
__device__ __forceinline__ bool oper_epilogue(const OperArgs& g, const MmaEpi& e)
{
    constexpr int STEP = OP_EW / 4, TEAMS = FULL ? 2 : 1, EPI_THREADS = TEAMS * OP_EW * 32;
    const uint32_t tab0 = smem_u32(e.smem + g.off_tab);
    const uint32_t hi2 = ((1u << g.out_bits) - 1u) * 0x10001u;
    // a residual code in the low bits of a word is the denormal code * 2^-149; everything is scaled by 2^-24
    const uint32_t rm = __float_as_uint(g.res_scale * __uint_as_float(252u << 23)), rm4 = __float_as_uint(g.res_scale * __uint_as_float(250u << 23));
    const u64 rmul = f2_pack(rm, rm), rmul4 = f2_pack(rm4, rm4);
    const int groups = g.TN >> 5, o0 = static_cast<int>(blockIdx.x % static_cast<unsigned>(g.tiles_o)) * g.TN;
    epilogue_tables(g, reinterpret_cast<float4*>(e.smem + g.off_tab), reinterpret_cast<float2*>(e.smem + g.off_tab + g.TN * 8), e.fast_ok, o0, e.tid, EPI_THREADS);
    asm volatile("bar.sync 2, %0;" ::"n"(EPI_THREADS) : "memory");
    const bool fast = *reinterpret_cast<volatile int*>(e.fast_ok) != 0;
    if (g.early_b) mm_pdl_wait();
    const int team = FULL ? e.warp / OP_EW : 0;
    int ia = team;
    unsigned pa = 0;
    if (ia >= g.nacc) { ia -= g.nacc; pa ^= 1u; }
    bool ok = true;
#ifdef BS_TRACE
    int seq = 0;
#endif
    for (int m = static_cast<int>(blockIdx.x / static_cast<unsigned>(g.tiles_o)) + team * g.step_m; m < g.tiles_m; m += TEAMS * g.step_m) {
        const int base = m * 128 * g.PT + e.row0;
        // units (NT tiles, group), group fastest
        int t = 0, cc = e.set;
        while (cc >= groups) { cc -= groups; t += NT; }
        OperPos px[NT];
        auto pixels = [&]() {
#pragma unroll
            for (int j = 0; j < NT; ++j) px[j] = oper_position(g, base + (t + j) * 128);
        };
        uint32_t rn[NT][4];
        auto residual = [&](int ob) {
#pragma unroll
            for (int j = 0; j < NT; ++j) {
#pragma unroll
                for (int k = 0; k < 4; ++k) rn[j][k] = 0;
                if (RES && px[j].pix >= 0 && ob < g.O) load_residual(g, px[j].pix, ob, rn[j]);
            }
        };
        if (t < g.PT) {
            pixels();
            residual(o0 + cc * 32);
        }
        if (ok) ok = mm_wait(&e.full_acc[ia], pa);    // after a wait that ran out the walk goes on without waiting
        mm_fence_after();
        MM_TRACE(e.tid == 0, TR_EBEG, seq);
        const uint32_t acc = e.acc + static_cast<uint32_t>(ia * g.PT * g.TN), TN = static_cast<uint32_t>(g.TN);
        if (!fast) {
            oper_item_formula(g, acc, base, o0, e.set);
            t = g.PT;
        }
        bool released = false;
        uint32_t v[2][NT][8];           // [buffer][tile]
        uint32_t col = acc + static_cast<uint32_t>(t * g.TN + cc * 32);
        if (t < g.PT)
#pragma unroll
            for (int j = 0; j < NT; ++j) mm_ld8(col + j * TN, v[0][j]);
        while (t < g.PT) {
            const int ob = o0 + cc * 32;
            const uint32_t tab = tab0 + static_cast<uint32_t>(cc) * 256u;
            OperPos to[NT];
            uint32_t z[2][NT];                             // [half of the filters][tile]
#pragma unroll
            for (int j = 0; j < NT; ++j) { to[j] = px[j]; z[0][j] = z[1][j] = 0u; }
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
                } else {
                    // the last columns of the item are in registers: the MMAs of a later one may overwrite them
                    mm_fence_before();
                    __syncwarp();
                    if (e.lane == 0) mm_arrive(&e.empty_acc[ia]);
                    released = true;
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
                if (to[j].pix >= 0 && ob < g.O) oper_store(g, to[j], ob, H[0][j], H[1][j]);
        }
        if (!released) {                // no columns, or read by the formula
            mm_fence_before();
            __syncwarp();
            if (e.lane == 0) mm_arrive(&e.empty_acc[ia]);
        }
        MM_TRACE(e.tid == 0, TR_EEND, seq);
#ifdef BS_TRACE
        ++seq;
#endif
        for (ia += TEAMS; ia >= g.nacc; ia -= g.nacc) pa ^= 1u;
    }
    return ok;
}

// ----------------------------------------------------------------------------- MMA issue

struct OperIssue {
    uint64_t *full, *empty, *full_acc, *empty_acc, *wgt_full, *form_ok;
    uint32_t smem0, tmem;
};

// The nine taps of a K step under one elect.sync, in one asm statement: OFF advances the pixel operand to the next tap.
#define OP_MMA(A, B, P) "@p tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], " A ", " B ", %3, [%5], [%5], " P ";\n\t"
#define OP_STEP(OFF) "add.s64 a, a, " OFF ";\n\tadd.s64 b, b, 16;\n\t" OP_MMA("a", "b", "t")
template <int ST>
__device__ __forceinline__ void oper_taps(uint32_t d, uint32_t a, uint32_t a_hi, uint32_t b, uint32_t b_hi, uint32_t idesc, uint32_t acc, uint32_t pitch, uint32_t HL, uint32_t sf)
{
    const uint64_t da = (static_cast<uint64_t>(a_hi) << 32) | a, db = (static_cast<uint64_t>(b_hi) << 32) | b;
    if (ST == 1) {
        const uint64_t row = pitch - 2u;        // from the last tap of a row to the first of the next
        asm volatile(
            "{\n\t.reg .pred p, q, t;\n\t.reg .b64 a, b;\n\t"
            "elect.sync _|p, 0xffffffff;\n\t"
            "setp.ne.b32 q, %4, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
            "mov.b64 a, %1;\n\tmov.b64 b, %2;\n\t"
            OP_MMA("a", "b", "q") OP_STEP("1") OP_STEP("1") OP_STEP("%6") OP_STEP("1") OP_STEP("1") OP_STEP("%6") OP_STEP("1") OP_STEP("1")
            "}"
            ::"r"(d), "l"(da), "l"(db), "r"(idesc), "r"(acc), "r"(sf), "l"(row) : "memory");
    } else {
        // offsets of the taps (issue_taps): 3 HL, 2 HL + 1, 3 HL + 1; HL, 1, HL + 1 and 3 HL, 2 HL + 1, 3 HL + 1, these a row on
        const uint64_t back = 1ull - HL, fwd = HL, r1 = static_cast<uint64_t>(pitch) - 2ull * HL - 1ull, r2 = 2ull * HL - 1ull;
        asm volatile(
            "{\n\t.reg .pred p, q, t;\n\t.reg .b64 a, b;\n\t"
            "elect.sync _|p, 0xffffffff;\n\t"
            "setp.ne.b32 q, %4, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
            "mov.b64 a, %1;\n\tmov.b64 b, %2;\n\t"
            OP_MMA("a", "b", "q") OP_STEP("%6") OP_STEP("%7") OP_STEP("%8") OP_STEP("%6") OP_STEP("%7") OP_STEP("%9") OP_STEP("%6") OP_STEP("%7")
            "}"
            ::"r"(d), "l"(da + 3u * HL), "l"(db), "r"(idesc), "r"(acc), "r"(sf), "l"(back), "l"(fwd), "l"(r1), "l"(r2) : "memory");
    }
}

template <int TAPS>
__device__ __forceinline__ void oper_block(const OperArgs& g, uint32_t d, uint32_t a, uint32_t a_hi, uint32_t b, uint32_t b_hi, uint32_t acc, uint32_t sf)
{
    const uint32_t pitch = static_cast<uint32_t>(g.pitch), HL = static_cast<uint32_t>(g.HL), idesc = g.idesc;
    if (TAPS == TAPS_1) issue_mma<true>(d, a, a_hi, b, b_hi, idesc, acc, sf);
    else if (TAPS == TAPS_3S1) oper_taps<1>(d, a, a_hi, b, b_hi, idesc, acc, pitch, HL, sf);
    else if (TAPS == TAPS_3S2) oper_taps<2>(d, a, a_hi, b, b_hi, idesc, acc, pitch, HL, sf);
    else
        for (int r = 0; r < g.R; ++r)
            for (int s = 0; s < g.R; ++s) {
                const int rp = r - g.pad, sp = s - g.pad;
                uint32_t off;
                if (g.stride == 1) off = static_cast<uint32_t>(r * g.pitch + s);
                else off = static_cast<uint32_t>(((rp & 1) * 2 + (sp & 1)) * g.HL + ((rp >> 1) - g.rmin) * g.pitch + (sp >> 1) - g.smin);
                issue_mma<true>(d, a + off, a_hi, b, b_hi, idesc, acc, sf);
                acc = 1u;
                b += 16u;
            }
}

// In uniform code, as issue_items (mma_kernel.cuh).
template <int TAPS>
__device__ __forceinline__ void oper_issue(const OperArgs& g, const OperIssue& m)
{
    const uint32_t NI16 = static_cast<uint32_t>(g.NI);
    const uint32_t a_hi = (128u >> 4) | (1u << 14), b_hi = static_cast<uint32_t>(g.RS * 16) | (1u << 14);
    const uint32_t a_lo0 = g.halves == 1 ? 0u : (NI16 & 0x3FFFu) << 16, b_lo0 = (128u >> 4) << 16;
    const uint32_t smem_off = m.smem0 & 0x3FFFFu, s_base = (smem_off + g.off_stage) >> 4, w_base = smem_off >> 4;
    const uint32_t blk16 = static_cast<uint32_t>(g.TN * g.RS * 2), unit16 = NI16 * static_cast<uint32_t>(g.halves), TN = static_cast<uint32_t>(g.TN);
    const uint32_t stage16 = static_cast<uint32_t>(g.stage_bytes >> 4), a16 = static_cast<uint32_t>(g.a_bytes >> 4);
    const int nchunks = g.nchunks, PT = g.PT, units = g.units, nunits = g.nunits, nse = g.nse, nacc = g.nacc;
    const bool resident = g.resident != 0;
    const uint32_t sf = m.tmem + static_cast<uint32_t>(g.sf_col);
    unsigned limit = 1u << 20;
    if (resident) mm_wait_uniform(m.wgt_full, 0, limit);
    mm_wait_uniform(m.form_ok, 0, limit);
    MM_TRACE((threadIdx.x & 31) == 0, TR_WGT, 0);
#ifdef BS_TRACE
    int mseq = 0;
#endif
    int ie = 0, ia = 0;
    unsigned pe = 0, pa = 0;
    for (int it = static_cast<int>(blockIdx.x / static_cast<unsigned>(g.tiles_o)); it < g.tiles_m; it += g.step_m) {
        mm_wait_uniform(&m.empty_acc[ia], pa, limit);
        const uint32_t d0 = m.tmem + static_cast<uint32_t>(ia * PT) * TN;
        for (int c = 0; c < nchunks; ++c) {
            const int u0 = c * units;
            const int nu = nunits - u0 < units ? nunits - u0 : units;
            const uint32_t eb = s_base + static_cast<uint32_t>(ie) * stage16;
            const uint32_t wb = b_lo0 | (resident ? w_base + static_cast<uint32_t>(u0) * blk16 : eb + a16);
            mm_wait_uniform(&m.full[ie], pe, limit);
            mm_fence_after();
            MM_TRACE((threadIdx.x & 31) == 0, TR_MBEG, mseq);
            uint32_t d = d0, at = a_lo0 | eb;
            for (int t = 0; t < PT; ++t, d += TN, at += 128u) {
                uint32_t a = at, b = wb;
                oper_block<TAPS>(g, d, a, a_hi, b, b_hi, c == 0 ? 0u : 1u, sf);
#pragma unroll(TAPS == TAPS_1 ? 4 : 1)
                for (int k = 1; k < nu; ++k) {
                    a += unit16;
                    b += blk16;
                    oper_block<TAPS>(g, d, a, a_hi, b, b_hi, 1u, sf);
                }
            }
            mm_commit(&m.empty[ie]);
            if (c == nchunks - 1) mm_commit(&m.full_acc[ia]);
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

// ----------------------------------------------------------------------------- the kernel

template <bool FULL>
__global__ void __launch_bounds__(oper_threads(FULL), FULL ? 1 : 2) bitserial_oper_kernel(const __grid_constant__ OperArgs g)
{
    extern __shared__ __align__(1024) unsigned char op_smem[];
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const uint32_t smem0 = smem_u32(op_smem);
    uint64_t* bars = reinterpret_cast<uint64_t*>(op_smem + g.off_bar);
    uint64_t* full = bars;                      // [OP_STAGES] pixels (and filters) of a chunk landed
    uint64_t* empty = bars + OP_STAGES;         // [OP_STAGES]
    uint64_t* full_acc = empty + OP_STAGES;     // [4]
    uint64_t* empty_acc = full_acc + 4;         // [4]
    uint64_t* wgt_full = empty_acc + 4;
    uint64_t* form_ok = wgt_full + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(form_ok + 1);
    int* fast_ok = reinterpret_cast<int*>(form_ok + 2);
    constexpr int WARP_COPY = (FULL ? 2 : 1) * OP_EW, WARP_MMA = WARP_COPY + 1;

    MM_TRACE(tid == 0, TR_START, 0);
    if (tid == 0) {
        for (int s = 0; s < OP_STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int s = 0; s < 4; ++s) { mbar_init(&full_acc[s], 1); mbar_init(&empty_acc[s], OP_EW); }
        mbar_init(wgt_full, 1);
        mbar_init(form_ok, 1);
        *fast_ok = 1;
        fence_barrier_init();
        fence_proxy_async();
    }
    if (warp == WARP_MMA) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(g.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    mm_fence_before();
    __syncthreads();
    mm_fence_after();
    // only now: a CTA of the next launch may take tensor memory as soon as it runs, and it keeps it until this launch has ended
    mm_pdl_release();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    MM_TRACE(tid == 0, TR_SETUP, 0);

    if (warp == WARP_COPY) {
        // ------------------------------------------------------------------ copies: a lane each, of a chunk or of the resident filters
        const int o0 = static_cast<int>(blockIdx.x % static_cast<unsigned>(g.tiles_o)) * g.TN;
        const size_t blk_stride = static_cast<size_t>(g.opad) * g.RS * 32;
        const unsigned blk_bytes = static_cast<unsigned>(g.TN * g.RS * 32), run = static_cast<unsigned>(g.HL) * 16u;
        const int8_t* wsrc = g.wgt + static_cast<size_t>(o0) * g.RS * 32;
        const bool resident = g.resident != 0;
        bool ok = true, waited = false;
        if (!g.early_b) { mm_pdl_wait(); waited = true; }
        if (resident) {
            if (lane == 0) mbar_expect_tx(wgt_full, blk_bytes * g.nunits);
            __syncwarp();
            for (int b = lane; b < g.nunits; b += 32) mm_bulk(op_smem + static_cast<size_t>(b) * blk_bytes, wsrc + b * blk_stride, blk_bytes, wgt_full);
        }
        // Filters prepared for other widths are converted as they arrive (mma_kernel.cuh, convert_filters); the first copies are made as if they were not.
        uint32_t mark;
        asm volatile("ld.global.b32 %0, [%1];" : "=r"(mark) : "l"(g.wgt + blk_stride * g.Cw - 4) : "memory");
        bool first = true, other = false;
        int is = 0;
        unsigned ps = 0;
        const int per_unit = g.halves * g.nplanes;
        for (int m = static_cast<int>(blockIdx.x / static_cast<unsigned>(g.tiles_o)); m < g.tiles_m && ok; m += g.step_m) {
            const unsigned char* src = g.src + static_cast<long long>(m) * g.PT * 2048;
            for (int c = 0; c < g.nchunks; ++c) {
                const int u0 = c * g.units, nu = min(g.units, g.nunits - u0);
                ok = mm_wait(&empty[is], ps ^ 1u);
                if (!ok) break;
                unsigned char* dst = op_smem + g.off_stage + static_cast<size_t>(is) * g.stage_bytes;
                const bool filters = !resident && !other;
                if (!resident && other) convert_filters<true>(g, dst + g.a_bytes, o0, u0, nu, lane);
                if (lane == 0) mbar_expect_tx(&full[is], static_cast<unsigned>(nu * per_unit) * run + (filters ? blk_bytes * nu : 0u));
                __syncwarp();
                if (filters)
                    for (int b = lane; b < nu; b += 32) mm_bulk(dst + g.a_bytes + static_cast<size_t>(b) * blk_bytes, wsrc + (u0 + b) * blk_stride, blk_bytes, &full[is]);
                if (!waited) { mm_pdl_wait(); waited = true; }
                for (int k = lane; k < nu * per_unit; k += 32) {
                    const int pl = g.nplanes == 1 ? 0 : k & 3, h = g.nplanes == 1 ? k : k >> 2;         // channel group of the chunk
                    // (of an odd number of groups the last one stands in for the missing one, whose filters are zero)
                    const int grp = min(u0 * g.halves + h, g.Cw - 1);
                    mm_bulk(dst + static_cast<size_t>(k) * run, src + grp * g.src_group + pl * g.src_plane, run, &full[is]);
                }
                if (first) {
                    first = false;
                    other = mark != MM_NIBBLE_MARK;
                    if (other) {
                        ok = mm_wait(resident ? wgt_full : &full[0], 0);
                        if (resident) convert_filters<true>(g, op_smem, o0, 0, g.nunits, lane);
                        else convert_filters<true>(g, dst + g.a_bytes, o0, u0, nu, lane);
                    }
                    __syncwarp();
                    if (lane == 0) mm_arrive(form_ok);
                }
                if (++is == g.nse) { is = 0; ps ^= 1u; }
            }
        }
        if (!ok && lane == 0) atomicOr(g.status, STATUS_TIMEOUT);
        __syncwarp();
    } else if (warp == WARP_MMA) {
        const OperIssue m{full, empty, full_acc, empty_acc, wgt_full, form_ok, smem0, tmem};
        if (g.R == 1) oper_issue<TAPS_1>(g, m);
        else if (g.R == 3 && g.stride == 1) oper_issue<TAPS_3S1>(g, m);
        else if (g.R == 3 && g.pad == 1) oper_issue<TAPS_3S2>(g, m);
        else oper_issue<TAPS_ANY>(g, m);
    } else {
        const int quad = warp & 3, set = (warp >> 2) & 1;
        const uint32_t lane_addr = static_cast<uint32_t>(quad * 32) << 16;
        // scale factors of 2 for every row, column and block
        if (warp < OP_EW) {
        for (int c = set * 8; c < MM_SF_COLS; c += 8 * (OP_EW / 4)) mm_st8(tmem + lane_addr + static_cast<uint32_t>(g.sf_col + c), 0x80808080u);
        mm_st_wait();
        mm_fence_before();
        __syncwarp();
        if (lane == 0)
            for (int s = 0; s < g.nacc; ++s) mm_arrive(&empty_acc[s]);
        }
        if (!g.early_b) mm_pdl_wait();
        MmaEpi e;
        e.smem = op_smem; e.full_acc = full_acc; e.empty_acc = empty_acc; e.fast_ok = fast_ok;
        e.acc = tmem + lane_addr; e.row0 = quad * 32 + lane; e.set = set;
        e.tid = tid; e.lane = lane; e.warp = warp; e.red_full = nullptr;
        // (pairs of row tiles where that leaves both warps of a lane quadrant some)
        const bool pair = g.PT > 1 && g.PT * (g.TN >> 5) >= 4;
        bool ok;
        if (g.residual) ok = pair ? oper_epilogue<true, 2, FULL>(g, e) : oper_epilogue<true, 1, FULL>(g, e);
        else ok = pair ? oper_epilogue<false, 2, FULL>(g, e) : oper_epilogue<false, 1, FULL>(g, e);
        if (!ok && lane == 0) atomicOr(g.status, STATUS_TIMEOUT);
    }
    mm_fence_before();
    __syncthreads();
    MM_TRACE(tid == 0, TR_END, 0);
    if (warp == WARP_MMA) {
        mm_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(g.tmem_cols) : "memory");
    }
}

}  // namespace bs
