// The layers a mixed-precision network keeps in floating point (paper, Section VII-D: a few quantisation-sensitive layers
// stay FP32, the rest is quantised): the first convolution with its max pooling, and the final average pooling + fully
// connected layer.  The paper gives no arithmetic for them beyond "FP32".  Fixed here, because a quantiser turns the stem's
// output into integer codes and every rounding matters: IEEE binary32; a convolution output is a chain of fused multiply-adds
// that starts at the bias and walks the taps channel-outermost, then row, then column, all ascending; the fully connected
// layer walks its inputs ascending; the average pool sums integer codes exactly and multiplies once.
#include "common.cuh"

namespace bs {

// ----------------------------------------------------------------------------- convolution, register-tiled
//
// CTA tile: TH x TW output pixels of one image x 64 filters; thread = 8 filters x 8 consecutive output columns.
// Weights of the 64 filters ([c][r][s][64], 16-byte vectors of four filters) and the input halo sit in shared memory.  For a
// fixed (c, r) a thread keeps the input row segment of its eight outputs in registers and walks the S columns: per column two
// 128-bit weight loads feed 64 fused multiply-adds (with four filters per thread the shared-memory pipe, not the FMA pipe, set
// the pace: 22 TFLOP/s).  A warp is 8 filter octets x 4 strips: its weight loads are 8 distinct vectors, its input loads four
// broadcasts.
// What bounds it: the FMA pipe, 64 fused multiply-adds a clock and SM sub-partition pair in theory, about 85 % of that measured on
// registers alone, one by one or in pairs; pairs leave issue slots for the loads.  Stem of 64 images of 224 x 224 (15.1 GFLOP): 440 us
// with single FMAs, 4-byte copies and 16-byte stores, 376 with pairs, 326 with 16-byte copies and 32-byte stores as well; without
// staging and stores the loop alone takes 282.
// Tile shapes of 32 strips of eight outputs: 16 x 16, 8 x 32 or 32 x 8, whichever covers the output with the fewest tiles.
constexpr int F32_STRIP = 8, F32_STRIPS = 32, F32_OT = 64, F32_THREADS = 256, F32_FPT = 8;

struct ConvF32Args {
    const float* x;
    const float* w;
    const float* bias;
    float* out;
    int N, C, H, W, O, R, stride, pad, relu, P, Q;
    int th, tw;                   // output tile: rows, columns (strips are numbered row-major over it)
    int in_h, pitch;              // staged input tile: rows, row pitch (floats, multiple of 4)
    int tiles_p, tiles_q, tiles_o;
    int sectors;                  // output strips start on 32-byte boundaries
};

// acc = (x, x) * w + acc on two filters at once: two IEEE fused multiply-adds in one instruction.
__device__ __forceinline__ void fma_pair(float2& acc, float2 x, float2 w)
{
    uint64_t d = (static_cast<uint64_t>(__float_as_uint(acc.y)) << 32) | __float_as_uint(acc.x);
    const uint64_t a = (static_cast<uint64_t>(__float_as_uint(x.y)) << 32) | __float_as_uint(x.x);
    const uint64_t b = (static_cast<uint64_t>(__float_as_uint(w.y)) << 32) | __float_as_uint(w.x);
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
    acc.x = __uint_as_float(static_cast<uint32_t>(d));
    acc.y = __uint_as_float(static_cast<uint32_t>(d >> 32));
}

// One output strip to global memory: eight floats, 32-byte aligned (one whole sector per thread; 16-byte pieces wrote every sector twice).
__device__ __forceinline__ void store_strip(float* dst, const float (&v)[F32_STRIP])
{
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]),
                 "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
}

// SHIFT >= 0: rows of x are 16-byte multiples and the halo is staged in 16-byte pieces from the boundary SHIFT floats before its
// first column (SHIFT = -pad mod 4; a piece lies inside the image or outside it as a whole).  SHIFT < 0: in single floats.
template <int S, int STRIDE, int SHIFT>
__global__ void __launch_bounds__(F32_THREADS, 2) conv2d_f32_tiled_kernel(const ConvF32Args g)
{
    extern __shared__ __align__(16) float f32_smem[];
    dependent_begin(g.out);
    constexpr int SH = SHIFT > 0 ? SHIFT : 0;
    constexpr int WIN = (F32_STRIP - 1) * STRIDE + S + SH;       // input columns one strip needs
    constexpr int WIN4 = (WIN + 3) / 4;
    float* s_w = f32_smem;                                       // [C][R][S][2][8][4]
    float* s_x0 = f32_smem + g.C * g.R * S * F32_OT;             // [2][C][in_h][pitch]: the halo of the next tile lands while this one is computed
    const int halo_floats = g.C * g.in_h * g.pitch;
    const int tid = threadIdx.x;
    const int to = blockIdx.y, o0 = to * F32_OT;

    // weights once per CTA: global [O][C][R][S] -> shared [c][r][s][o - o0] (zero beyond O).  A warp takes 8 consecutive taps (one
    // sector) of 4 filters.
    const int taps = g.C * g.R * S;
    for (int i = tid >> 5; i < (taps + 7) / 8 * (F32_OT / 4); i += F32_THREADS / 32) {
        // filter o = 8 * octet + k sits at [tap][k / 4][octet][k % 4]: the eight threads of a quarter warp, one octet each, read
        // 128 contiguous bytes with each of their two vector loads
        const int t = (i >> 4) * 8 + (tid & 7), o = (i & 15) * 4 + ((tid & 31) >> 3);
        if (t < taps)
            s_w[t * F32_OT + ((o & 7) >> 2) * 32 + (o >> 3) * 4 + (o & 3)] = (o0 + o < g.O) ? g.w[static_cast<size_t>(o0 + o) * taps + t] : 0.0f;
    }
    const int tiles = g.N * g.tiles_p * g.tiles_q;
    // Input halo of a tile, zero outside the image (a zero tap leaves the chain unchanged: fma(0, w, acc) == acc), fetched with
    // asynchronous copies (zero-filled where the source is outside), so the copies of tile k + 1 fly while tile k is computed.  A warp
    // takes whole rows; 4-byte copies with an index each cost 50 us on the stem above.
    auto stage = [&](int tile, float* dst) {
        constexpr int E = SHIFT >= 0 ? 4 : 1;                    // floats per copy
        int b = tile;
        const int tq = b % g.tiles_q; b /= g.tiles_q;
        const int tp = b % g.tiles_p; b /= g.tiles_p;
        const int n = b;
        const int y0 = tp * g.th * STRIDE - g.pad, x0 = tq * g.tw * STRIDE - g.pad - SH;
        const int rows = g.C * g.in_h, per_row = g.pitch / E;
        // lanes: as many rows at once as 32 lanes hold (per_row is at least 4 and 10 on the stem)
        const int span = per_row <= 4 ? 4 : per_row <= 8 ? 8 : per_row <= 16 ? 16 : 32;
        const int lane = tid & 31, col = lane & (span - 1), rstep = (F32_THREADS / 32) * (32 / span);
        int row = (tid >> 5) * (32 / span) + lane / span, y2 = row, c2 = 0;
        while (y2 >= g.in_h) { y2 -= g.in_h; ++c2; }
        for (; row < rows; row += rstep) {
            const int y = y0 + y2;
            const bool yok = y >= 0 && y < g.H;
            const float* src_row = g.x + ((static_cast<size_t>(n) * g.C + c2) * g.H + (yok ? y : 0)) * g.W;
            for (int k = col; k < per_row; k += span) {
                const int x = x0 + k * E;
                const bool ok = yok && x >= 0 && x < g.W;
                const float* src = ok ? src_row + x : g.x;
                const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst + row * g.pitch + k * E));
                if constexpr (E == 4) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
                else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(ok ? 4 : 0) : "memory");
            }
            y2 += rstep;
            while (y2 >= g.in_h) { y2 -= g.in_h; ++c2; }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (static_cast<int>(blockIdx.x) < tiles) stage(blockIdx.x, s_x0);
    int buf = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x, buf ^= 1) {
    int b = tile;
    const int tq = b % g.tiles_q; b /= g.tiles_q;
    const int tp = b % g.tiles_p; b /= g.tiles_p;
    const int n = b;
    const int p0 = tp * g.th, q0 = tq * g.tw;
    const float* s_x = s_x0 + buf * halo_floats;
    // the other buffer was read by the tile before this one: every thread is past that (barrier at the end of the loop body)
    if (tile + static_cast<int>(gridDim.x) < tiles) {
        stage(tile + gridDim.x, s_x0 + (buf ^ 1) * halo_floats);
        asm volatile("cp.async.wait_group 1;" ::: "memory");     // this tile's copies have landed; the next tile's may still fly
    } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();

    const int cq = tid & 7, strip = tid >> 3;                    // filter octet, strip
    const int sp = strip / (g.tw / F32_STRIP), sq = strip % (g.tw / F32_STRIP);
    float2 acc[F32_STRIP][F32_FPT / 2];
    {
        float bq[F32_FPT];
#pragma unroll
        for (int k = 0; k < F32_FPT; ++k) bq[k] = (g.bias && o0 + cq * F32_FPT + k < g.O) ? g.bias[o0 + cq * F32_FPT + k] : 0.0f;
#pragma unroll
        for (int j = 0; j < F32_STRIP; ++j)
#pragma unroll
            for (int k = 0; k < F32_FPT / 2; ++k) acc[j][k] = make_float2(bq[2 * k], bq[2 * k + 1]);  // the chain starts at the bias
    }
    for (int c = 0; c < g.C; ++c) {
        for (int r = 0; r < g.R; ++r) {
            const float* row = s_x + (c * g.in_h + sp * STRIDE + r) * g.pitch + sq * F32_STRIP * STRIDE;
            float xr[WIN4 * 4];
#pragma unroll
            for (int v = 0; v < WIN4; ++v) {
                const float4 t = *reinterpret_cast<const float4*>(row + 4 * v);
                xr[4 * v] = t.x; xr[4 * v + 1] = t.y; xr[4 * v + 2] = t.z; xr[4 * v + 3] = t.w;
            }
            const float* wrow = s_w + ((c * g.R + r) * S) * F32_OT + cq * 4;
#pragma unroll
            for (int s = 0; s < S; ++s) {
                const float4 wa = *reinterpret_cast<const float4*>(wrow + s * F32_OT);
                const float4 wb = *reinterpret_cast<const float4*>(wrow + s * F32_OT + 32);
#pragma unroll
                for (int j = 0; j < F32_STRIP; ++j) {
                    const float2 xv = make_float2(xr[j * STRIDE + s + SH], xr[j * STRIDE + s + SH]);
                    fma_pair(acc[j][0], xv, make_float2(wa.x, wa.y));
                    fma_pair(acc[j][1], xv, make_float2(wa.z, wa.w));
                    fma_pair(acc[j][2], xv, make_float2(wb.x, wb.y));
                    fma_pair(acc[j][3], xv, make_float2(wb.z, wb.w));
                }
            }
        }
    }
    const int p = p0 + sp, qb = q0 + sq * F32_STRIP;
#pragma unroll
    for (int k = 0; k < F32_FPT; ++k) {
        const int o = o0 + cq * F32_FPT + k;
        if (o >= g.O || p >= g.P) continue;
        float* dst = g.out + ((static_cast<size_t>(n) * g.O + o) * g.P + p) * g.Q + qb;
        float v[F32_STRIP];
#pragma unroll
        for (int j = 0; j < F32_STRIP; ++j) {
            const float a = (k & 1) ? acc[j][k / 2].y : acc[j][k / 2].x;
            v[j] = g.relu ? fmaxf(a, 0.0f) : a;
        }
        if (qb + F32_STRIP <= g.Q && g.sectors) {
            store_strip(dst, v);
        } else if (qb + F32_STRIP <= g.Q && (g.Q & 3) == 0) {
            reinterpret_cast<float4*>(dst)[0] = make_float4(v[0], v[1], v[2], v[3]);
            reinterpret_cast<float4*>(dst)[1] = make_float4(v[4], v[5], v[6], v[7]);
        } else {
#pragma unroll
            for (int j = 0; j < F32_STRIP; ++j)
                if (qb + j < g.Q) dst[j] = v[j];
        }
    }
    __syncthreads();                                             // every thread is done reading this tile's halo buffer
    }   // tiles
}

// Any other shape: one thread per output, the same chain in the same order (slow; the stem shapes take the tiled kernel).
__global__ void conv2d_f32_direct_kernel(const float* __restrict__ x, const float* __restrict__ w, const float* __restrict__ bias,
                                         float* __restrict__ out, int N, int C, int H, int W, int O, int R, int S, int stride, int pad,
                                         int relu, int P, int Q)
{
    const long long total = static_cast<long long>(N) * O * P * Q;
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += static_cast<long long>(gridDim.x) * blockDim.x) {
        long long t = i;
        const int q = static_cast<int>(t % Q); t /= Q;
        const int p = static_cast<int>(t % P); t /= P;
        const int o = static_cast<int>(t % O);
        const int n = static_cast<int>(t / O);
        float acc = bias ? bias[o] : 0.0f;
        for (int c = 0; c < C; ++c)
            for (int r = 0; r < R; ++r)
                for (int s = 0; s < S; ++s) {
                    const int y = p * stride - pad + r, xx = q * stride - pad + s;
                    if (y < 0 || y >= H || xx < 0 || xx >= W) continue;
                    acc = fmaf(x[((static_cast<size_t>(n) * C + c) * H + y) * W + xx], w[((static_cast<size_t>(o) * C + c) * R + r) * S + s], acc);
                }
        out[i] = relu ? fmaxf(acc, 0.0f) : acc;
    }
}

// ----------------------------------------------------------------------------- pooling and the classifier

__global__ void maxpool2d_f32_kernel(const float* __restrict__ x, float* __restrict__ out, long long planes, int H, int W, int k, int stride,
                                     int pad, int P, int Q)
{
    const long long total = planes * P * Q;
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += static_cast<long long>(gridDim.x) * blockDim.x) {
        const int q = static_cast<int>(i % Q);
        const int p = static_cast<int>((i / Q) % P);
        const long long pl = i / (static_cast<long long>(P) * Q);
        const float* src = x + pl * H * W;
        float m = -INFINITY;
        for (int r = 0; r < k; ++r) {
            const int y = p * stride - pad + r;
            if (y < 0 || y >= H) continue;
            for (int s = 0; s < k; ++s) {
                const int xx = q * stride - pad + s;
                if (xx < 0 || xx >= W) continue;
                m = fmaxf(m, src[static_cast<size_t>(y) * W + xx]);
            }
        }
        out[i] = m;
    }
}

// 3x3 window, stride 2, pad 1 on rows of even width (the stem's pooling): a thread produces four consecutive outputs from three rows of
// eight inputs, read as 128-bit vectors where W is a multiple of 8 (VEC) and as 64-bit ones otherwise, plus the column to their left.
// The maximum does not depend on the order of its operands, so this is the same result as the generic kernel.  Bound by HBM: 64 x 64
// planes of 112 x 112, 257 MB, take 40 us (6.4 TB/s); 16 x 64 planes of 100 x 100, 30 -> 14 us against the generic kernel.
template <bool VEC>
__global__ void __launch_bounds__(128) maxpool3x3s2p1_f32_kernel(const float* __restrict__ x_in, float* __restrict__ out, unsigned planes, int H, int W, int P, int Q)
{
    const float* x = dependent_begin(x_in);
    const unsigned q4n = static_cast<unsigned>(Q + 3) >> 2, per_plane = static_cast<unsigned>(P) * q4n;
    // grid.x: blocks of 128 quadruples of one plane; grid.y strides over the planes
    const unsigned i = blockIdx.x * 128u + threadIdx.x;
    if (i >= per_plane) return;
    const int p = static_cast<int>(i / q4n), q4 = static_cast<int>(i - static_cast<unsigned>(p) * q4n);
    for (unsigned k = blockIdx.y; k < planes; k += gridDim.y) {
        const size_t pl = k;
        const float* src = x + pl * H * W;
        float m[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const int y = 2 * p - 1 + r;
            if (y < 0 || y >= H) continue;
            const float* row = src + static_cast<size_t>(y) * W + 8 * q4;
            float v[8];
            if constexpr (VEC) {
                const float4 a = *reinterpret_cast<const float4*>(row), b = *reinterpret_cast<const float4*>(row + 4);
                v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
            } else {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float2 a = 8 * q4 + 2 * u < W ? *reinterpret_cast<const float2*>(row + 2 * u) : make_float2(-INFINITY, -INFINITY);
                    v[2 * u] = a.x; v[2 * u + 1] = a.y;
                }
            }
            const float left = q4 > 0 ? row[-1] : -INFINITY;
            m[0] = fmaxf(m[0], fmaxf(left, fmaxf(v[0], v[1])));
            m[1] = fmaxf(m[1], fmaxf(v[1], fmaxf(v[2], v[3])));
            m[2] = fmaxf(m[2], fmaxf(v[3], fmaxf(v[4], v[5])));
            m[3] = fmaxf(m[3], fmaxf(v[5], fmaxf(v[6], v[7])));
        }
        float* dst = out + (pl * P + p) * Q + 4 * q4;
        if constexpr (VEC) {
            *reinterpret_cast<float4*>(dst) = make_float4(m[0], m[1], m[2], m[3]);
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (4 * q4 + u < Q) dst[u] = m[u];
        }
    }
}

// Global average pool of packed activation codes [N][H][W][Cw][bits] -> float [N][C]: exact integer sum, one multiplication.
// A warp is one channel word of one image, lane = channel; the plane words of eight pixels are in flight at once (one after the
// other the loads' latency was all the time it took).
template <int BITS>
__global__ void avgpool_codes_kernel(const uint32_t* __restrict__ packed, float* __restrict__ out, int N, int C, int HW, int Cw, int sign, float inv)
{
    const int unit = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (unit >= N * Cw) return;
    const int n = unit / Cw, cw = unit - n * Cw, c = cw * 32 + lane;
    const uint32_t* src = packed + (static_cast<size_t>(n) * HW * Cw + cw) * BITS;
    const size_t pitch = static_cast<size_t>(Cw) * BITS;
    int sum = 0;
    for (int p0 = 0; p0 < HW; p0 += 8) {
        uint32_t w[8][BITS];
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int j = 0; j < BITS; ++j) w[u][j] = p0 + u < HW ? src[(p0 + u) * pitch + j] : 0u;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            unsigned pat = 0;
#pragma unroll
            for (int j = 0; j < BITS; ++j) pat |= ((w[u][j] >> lane) & 1u) << j;
            if (p0 + u < HW) sum += pattern_value(pat, BITS, sign);
        }
    }
    if (c < C) out[static_cast<size_t>(n) * C + c] = static_cast<float>(sum) * inv;
}

// out[n][j] = bias[j] + sum_k x[n][k] w[j][k], a chain of fused multiply-adds over ascending k: 4 cycles a step, 512 steps take
// 1.1 us whatever the batch.  Block: 32 outputs j (lane) x 16 rows n (four per warp, so a weight read from shared memory serves
// four chains and the inputs are broadcasts, four k per 128-bit load).  The operands pass through a ring of FC_STAGES chunks of
// FC_KC k filled by asynchronous copies, which keeps three chunks in flight; the chain crosses the chunks in order.  Rows of the
// weight chunk are 16 bytes longer than the chunk: eight lanes of a 128-bit load hit different banks.
// VEC: K is a multiple of 4 and the rows can be copied in 16-byte pieces, else in 4-byte ones.
constexpr int FC_KC = 64, FC_STAGES = 4, FC_J = 32, FC_N = 16, FC_THREADS = 128;
constexpr int FC_WPITCH = FC_KC + 4, FC_STAGE = FC_J * FC_WPITCH + FC_N * FC_KC;

template <bool VEC>
__global__ void __launch_bounds__(FC_THREADS) fc_f32_kernel(const float* __restrict__ x, const float* __restrict__ w, const float* __restrict__ bias,
                                                             float* __restrict__ out, int N, int K, int J)
{
    extern __shared__ __align__(16) float fc_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int j0 = blockIdx.x * FC_J, n0 = blockIdx.y * FC_N, j = j0 + lane;
    const int chunks = (K + FC_KC - 1) / FC_KC;
    // a chunk's 32 weight rows and 16 input rows; what lies outside the matrices is filled with zeros and never used
    auto fetch = [&](int chunk) {
        float* s_w = fc_smem + (chunk % FC_STAGES) * FC_STAGE;
        float* s_x = s_w + FC_J * FC_WPITCH;
        constexpr int E = VEC ? 4 : 1, PER = FC_KC / E;
        for (int i = threadIdx.x; i < (FC_J + FC_N) * PER; i += FC_THREADS) {
            const int r = i / PER, kk = (i % PER) * E, k = chunk * FC_KC + kk;
            const bool is_w = r < FC_J;
            const int row = is_w ? j0 + r : n0 + r - FC_J;
            const bool ok = row < (is_w ? J : N) && k < K;
            const float* src = (is_w ? w : x) + (ok ? static_cast<size_t>(row) * K + k : 0);
            const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(is_w ? s_w + r * FC_WPITCH + kk : s_x + (r - FC_J) * FC_KC + kk));
            if constexpr (VEC) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
            else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(ok ? 4 : 0) : "memory");
        }
    };
#pragma unroll
    for (int c = 0; c < FC_STAGES - 1; ++c) {
        if (c < chunks) fetch(c);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    float acc[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] = (bias && j < J) ? bias[j] : 0.0f;
    for (int c = 0; c < chunks; ++c) {
        asm volatile("cp.async.wait_group %0;" ::"n"(FC_STAGES - 2) : "memory");
        __syncthreads();                       // chunk c has landed, and every thread is done with the one before it
        if (c + FC_STAGES - 1 < chunks) fetch(c + FC_STAGES - 1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const float* s_w = fc_smem + (c % FC_STAGES) * FC_STAGE + lane * FC_WPITCH;
        const float* s_x = fc_smem + (c % FC_STAGES) * FC_STAGE + FC_J * FC_WPITCH + warp * 4 * FC_KC;
        const int kn = K - c * FC_KC < FC_KC ? K - c * FC_KC : FC_KC;
        if (kn == FC_KC) {
#pragma unroll 4
            for (int kk = 0; kk < FC_KC; kk += 4) {
                const float4 v = *reinterpret_cast<const float4*>(s_w + kk);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float4 u = *reinterpret_cast<const float4*>(s_x + i * FC_KC + kk);
                    acc[i] = fmaf(u.w, v.w, fmaf(u.z, v.z, fmaf(u.y, v.y, fmaf(u.x, v.x, acc[i]))));
                }
            }
        } else {
            for (int kk = 0; kk < kn; ++kk)
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i] = fmaf(s_x[i * FC_KC + kk], s_w[kk], acc[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int n = n0 + warp * 4 + i;
        if (j < J && n < N) out[static_cast<size_t>(n) * J + j] = acc[i];
    }
}

template <int S, int STRIDE, int SHIFT>
static int launch_conv_tiled(const ConvF32Args& g, size_t smem, cudaStream_t st)
{
    auto kern = conv2d_f32_tiled_kernel<S, STRIDE, SHIFT>;
    if (smem > 48 * 1024 && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess) {
        cudaGetLastError();
        return BS_ERR_CUDA;
    }
    const long long tiles = static_cast<long long>(g.N) * g.tiles_p * g.tiles_q;
    if (tiles > 0x7fffffffLL || g.tiles_o > 65535) return BS_ERR_UNSUPPORTED;
    int sms = device_sm_count();
    if (sms <= 0) return BS_ERR_CUDA;
    long long per_o = static_cast<long long>(sms) * 2 / g.tiles_o;         // two CTAs per SM (registers), persistent over the tiles
    if (per_o < 1) per_o = 1;
    if (per_o > tiles) per_o = tiles;
    return launch_dependent(kern, dim3(static_cast<unsigned>(per_o), static_cast<unsigned>(g.tiles_o)), dim3(F32_THREADS), smem, st, g);
}

}  // namespace bs

extern "C" int bs_conv2d_f32(const float* x, const float* w, const float* bias, int N, int C, int H, int W, int O, int R, int S, int stride,
                             int pad, int relu, float* out, void* stream)
{
    if (!x || !w || !out || N <= 0 || C <= 0 || H <= 0 || W <= 0 || O <= 0 || R <= 0 || S <= 0 || stride < 1 || pad < 0) return BS_ERR_INVALID_ARG;
    if (H + 2 * pad < R || W + 2 * pad < S) return BS_ERR_INVALID_ARG;
    if (!bs::aligned16(x) || !bs::aligned16(w) || !bs::aligned16(out) || (bias && (reinterpret_cast<uintptr_t>(bias) & 3u))) return BS_ERR_ALIGNMENT;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    bs::ConvF32Args g{};
    g.x = x; g.w = w; g.bias = bias; g.out = out;
    g.N = N; g.C = C; g.H = H; g.W = W; g.O = O; g.R = R; g.stride = stride; g.pad = pad; g.relu = relu;
    g.P = (H + 2 * pad - R) / stride + 1;
    g.Q = (W + 2 * pad - S) / stride + 1;
    const bool tiled = (S == 7 && stride == 2) || (S == 3 && stride == 1) || (S == 3 && stride == 2) || (S == 1 && stride == 1);
    if (tiled) {
        long long best = -1;
        for (const int tw : {16, 32, 8}) {
            const int th = bs::F32_STRIPS * bs::F32_STRIP / tw;
            const long long t = static_cast<long long>(bs::ceil_div(g.P, th)) * bs::ceil_div(g.Q, tw);
            if (best < 0 || t < best) { best = t; g.th = th; g.tw = tw; }
        }
        // 16-byte staging where rows allow it, for the padding its kernels are built for ("same" padding of the window)
        g.sectors = g.Q % 8 == 0 && (reinterpret_cast<uintptr_t>(out) & 31u) == 0;
        const bool wide = W % 4 == 0 && pad == S / 2;
        const int shift = wide ? (4 - pad % 4) % 4 : 0;
        g.in_h = (g.th - 1) * stride + R;
        // every strip reads whole 16-byte vectors: the last one may run a few floats past the halo
        const int win4 = ((bs::F32_STRIP - 1) * stride + S + shift + 3) / 4 * 4;
        g.pitch = (g.tw / bs::F32_STRIP - 1) * bs::F32_STRIP * stride + win4;
        g.tiles_p = bs::ceil_div(g.P, g.th); g.tiles_q = bs::ceil_div(g.Q, g.tw); g.tiles_o = bs::ceil_div(O, bs::F32_OT);
        const size_t smem = (static_cast<size_t>(C) * R * S * bs::F32_OT + 2 * static_cast<size_t>(C) * g.in_h * g.pitch) * 4;
        if (smem <= 200 * 1024) {
            if (S == 7) return wide ? bs::launch_conv_tiled<7, 2, 1>(g, smem, st) : bs::launch_conv_tiled<7, 2, -1>(g, smem, st);
            if (S == 3 && stride == 1) return wide ? bs::launch_conv_tiled<3, 1, 3>(g, smem, st) : bs::launch_conv_tiled<3, 1, -1>(g, smem, st);
            if (S == 3) return wide ? bs::launch_conv_tiled<3, 2, 3>(g, smem, st) : bs::launch_conv_tiled<3, 2, -1>(g, smem, st);
            return wide ? bs::launch_conv_tiled<1, 1, 0>(g, smem, st) : bs::launch_conv_tiled<1, 1, -1>(g, smem, st);
        }
    }
    const long long total = static_cast<long long>(N) * O * g.P * g.Q;
    long long blocks = (total + 255) / 256;
    if (blocks > 148 * 32) blocks = 148 * 32;
    bs::conv2d_f32_direct_kernel<<<static_cast<unsigned>(blocks), 256, 0, st>>>(x, w, bias, out, N, C, H, W, O, R, S, stride, pad, relu, g.P, g.Q);
    return cudaGetLastError() == cudaSuccess ? BS_OK : BS_ERR_CUDA;
}

extern "C" int bs_maxpool2d_f32(const float* x, int N, int C, int H, int W, int k, int stride, int pad, float* out, void* stream)
{
    if (!x || !out || N <= 0 || C <= 0 || H <= 0 || W <= 0 || k <= 0 || stride < 1 || pad < 0 || 2 * pad > k) return BS_ERR_INVALID_ARG;
    if (H + 2 * pad < k || W + 2 * pad < k) return BS_ERR_INVALID_ARG;
    const int P = (H + 2 * pad - k) / stride + 1, Q = (W + 2 * pad - k) / stride + 1;
    const long long planes = static_cast<long long>(N) * C, total = planes * P * Q;
    if (k == 3 && stride == 2 && pad == 1 && W % 2 == 0 && Q * 2 == W && planes < (1LL << 31) && bs::aligned16(x) && bs::aligned16(out)) {
        const long long per_plane = static_cast<long long>(P) * ((Q + 3) / 4);
        const dim3 grid(static_cast<unsigned>((per_plane + 127) / 128), static_cast<unsigned>(planes < 65535 ? planes : 65535));
        if (per_plane < (1LL << 31)) {
            return bs::launch_dependent(W % 8 == 0 ? bs::maxpool3x3s2p1_f32_kernel<true> : bs::maxpool3x3s2p1_f32_kernel<false>, grid, dim3(128), 0,
                                        static_cast<cudaStream_t>(stream), x, out, static_cast<unsigned>(planes), H, W, P, Q);
        }
    }
    long long blocks = (total + 255) / 256;
    if (blocks > 148 * 64) blocks = 148 * 64;
    bs::maxpool2d_f32_kernel<<<static_cast<unsigned>(blocks), 256, 0, static_cast<cudaStream_t>(stream)>>>(x, out, planes, H, W, k, stride, pad, P, Q);
    return cudaGetLastError() == cudaSuccess ? BS_OK : BS_ERR_CUDA;
}

extern "C" int bs_avgpool_codes_f32(const uint32_t* packed, int N, int C, int H, int W, int a_bits, bs_sign_t a_sign, float inv, float* out,
                                    void* stream)
{
    if (!packed || !out || N <= 0 || C <= 0 || H <= 0 || W <= 0 || !bs::bits_ok(a_bits, a_sign)) return BS_ERR_INVALID_ARG;
    if (static_cast<long long>(N) * C > 0x7fffffffLL || static_cast<long long>(H) * W * ((1 << a_bits)) >= (1LL << 24)) return BS_ERR_UNSUPPORTED;
    const int Cw = (C + 31) / 32, blocks = (N * Cw + 3) / 4;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const auto kern = a_bits == 1 ? bs::avgpool_codes_kernel<1> : a_bits == 2 ? bs::avgpool_codes_kernel<2> : a_bits == 3 ? bs::avgpool_codes_kernel<3> : bs::avgpool_codes_kernel<4>;
    kern<<<static_cast<unsigned>(blocks), 128, 0, st>>>(packed, out, N, C, H * W, Cw, a_sign, inv);
    return cudaGetLastError() == cudaSuccess ? BS_OK : BS_ERR_CUDA;
}

extern "C" int bs_fc_f32(const float* x, const float* w, const float* bias, int N, int K, int J, float* out, void* stream)
{
    if (!x || !w || !out || N <= 0 || K <= 0 || J <= 0) return BS_ERR_INVALID_ARG;
    const dim3 grid(static_cast<unsigned>((J + bs::FC_J - 1) / bs::FC_J), static_cast<unsigned>((N + bs::FC_N - 1) / bs::FC_N));
    if (grid.y > 65535) return BS_ERR_UNSUPPORTED;
    constexpr int smem = bs::FC_STAGES * bs::FC_STAGE * 4;
    static_assert(smem <= 227 * 1024, "ring of the fully connected layer");
    const bool vec = K % 4 == 0 && bs::aligned16(x) && bs::aligned16(w);
    const auto kern = vec ? bs::fc_f32_kernel<true> : bs::fc_f32_kernel<false>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) { cudaGetLastError(); return BS_ERR_CUDA; }
    // plain launches here and for the average pool: begun early the two took 23 us instead of 15
    kern<<<grid, bs::FC_THREADS, smem, static_cast<cudaStream_t>(stream)>>>(x, w, bias, out, N, K, J);
    return cudaGetLastError() == cudaSuccess ? BS_OK : BS_ERR_CUDA;
}
