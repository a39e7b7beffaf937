// Entry points of the tensor-core formulation: validation, filter preparation, layers and chains of layers (kernel: mma_conv.cu).
#include "common.cuh"
#include "mma_conv.h"
#include "oper_conv.h"

namespace bs {

// One thread per 16-byte vector of the prepared filter layout [C/32][O/8][tap][2][8 filters][16 channels], the core matrices of
// the B operand block by block; nibbles: [ceil(C/64)][O/8][tap][2][8 filters][32 channels], sign and magnitude.  Within a group of 32 filters
// the rows, and within a block of 32 channels the bytes, stand in the orders of mma_conv.h; nibble j of word m is channel 4 j + m.
__global__ void tc_prepare_weights_kernel(const uint32_t* __restrict__ packed, int8_t* __restrict__ out, long long nvec, int O, int RS, int Cw,
                                          int WB, int sign, int opad8, bool nibbles, long long last)
{
    const long long idx = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (idx >= nvec) return;
    const FilterVector f = filter_vector(idx, opad8, RS);
    const int o = f.o, tap = f.tap, half = f.half, blk = f.step;
    uint32_t vals[4] = {0, 0, 0, 0};
    if (nibbles) {
        const int cw = blk * 2 + half;
        if (o < O && cw < Cw) {
            const uint32_t* w = packed + ((static_cast<size_t>(o) * RS + tap) * Cw + cw) * WB;
            for (int ch = 0; ch < 32; ++ch) {
                unsigned pat = 0;
                for (int i = 0; i < WB; ++i) pat |= ((w[i] >> ch) & 1u) << i;
                const int v = pattern_value(pat, WB, sign);
                vals[ch & 3] |= static_cast<uint32_t>(v < 0 ? 8 - v : v) << (4 * (ch >> 2));
            }
        }
    } else if (o < O) {
        const uint32_t* w = packed + ((static_cast<size_t>(o) * RS + tap) * Cw + blk) * WB;
        for (int b = 0; b < 16; ++b) {
            const int ch = mma_channel_of_byte(half * 16 + b);
            unsigned pat = 0;
            for (int i = 0; i < WB; ++i) pat |= ((w[i] >> ch) & 1u) << i;
            const unsigned byte = static_cast<unsigned>(pattern_value(pat, WB, sign)) & 0xFFu;
            vals[b >> 2] |= byte << (8 * (b & 3));
        }
    }
    const uint4 v = make_uint4(vals[0], vals[1], vals[2], vals[3]);
    if (nibbles) put_nibbles(reinterpret_cast<uint4*>(out), idx, nvec, last, v);
    else reinterpret_cast<uint4*>(out)[idx] = v;
}

static int tc_max_abs(int bits, int sign)
{
    if (sign == BS_BIPOLAR) return 1;
    if (sign == BS_SIGNED) return 1 << (bits - 1);
    return (1 << bits) - 1;
}

// Validation shared by the support query and the launch.  Returns BS_OK when the tensor-core path can run `p`.
static int tc_validate_shape(const bs_conv_params* p)
{
    if (!p) return BS_ERR_INVALID_ARG;
    if (p->N <= 0 || p->C <= 0 || p->H <= 0 || p->W <= 0 || p->O <= 0 || p->R <= 0 || p->S <= 0) return BS_ERR_INVALID_ARG;
    if (!bits_ok(p->a_bits, p->a_sign) || !bits_ok(p->w_bits, p->w_sign)) return BS_ERR_INVALID_ARG;
    if (p->stride < 1 || p->pad < 0) return BS_ERR_INVALID_ARG;
    if (p->i32_layout != BS_NCHW && p->i32_layout != BS_NHWC) return BS_ERR_INVALID_ARG;
    if (p->R != p->S || (p->R != 1 && p->R != 3 && p->R != 5 && p->R != 7)) return BS_ERR_UNSUPPORTED;
    if (p->stride > 2 || p->pad >= p->R) return BS_ERR_UNSUPPORTED;
    if (p->a_sign == BS_BIPOLAR && p->pad != 0) return BS_ERR_UNSUPPORTED;
    if (p->H + 2 * p->pad < p->R || p->W + 2 * p->pad < p->S) return BS_ERR_INVALID_ARG;
    const long long kred = static_cast<long long>(p->C) * p->R * p->S;
    if (kred * tc_max_abs(p->a_bits, p->a_sign) * tc_max_abs(p->w_bits, p->w_sign) >= (1LL << 31)) return BS_ERR_UNSUPPORTED;
    return BS_OK;
}

// What can be run with prepared filters: channels that fill their words (the prepared tiles have no ragged block), and packed pixel
// records of 16-byte multiples, or of 8-byte multiples on rows that are 16-byte multiples (a contract of the entry points; the
// kernels themselves take any record).
static int tc_validate(const bs_conv_params* p)
{
    if (!p) return BS_ERR_INVALID_ARG;
    bs_conv_params q = *p;
    if (p->w_sign == BS_SIGNED_NIBBLES) q.w_sign = BS_SIGNED;
    const int rc = tc_validate_shape(&q);
    if (rc != BS_OK) return rc;
    if (p->C % 32 != 0 || (p->w_sign == BS_SIGNED_NIBBLES && !mma_nibbles(p->C, p->R * p->S, p->a_bits, p->w_bits, p->w_sign))) return BS_ERR_UNSUPPORTED;
    const int rec = p->C / 32 * p->a_bits;
    if (rec % 4 != 0) {
        if (rec % 2 != 0 || (p->W * rec) % 4 != 0) return BS_ERR_UNSUPPORTED;
        if (p->R == 1 && p->stride == 1 && p->pad == 0 && (static_cast<long long>(p->N) * p->H * p->W) % 2 != 0) return BS_ERR_UNSUPPORTED;
    }
    return BS_OK;
}

// Output side of the validation (pointers, code formats, channel slices).
static int tc_validate_outputs(const uint32_t* act, const void* wgt, const bs_conv_params* p, const int32_t* out_i32, const uint32_t* out_packed)
{
    if (!act || !wgt || (!out_i32 && !out_packed)) return BS_ERR_INVALID_ARG;
    if (!aligned16(act) || !aligned16(wgt) || (out_i32 && !aligned16(out_i32)) || (out_packed && !aligned16(out_packed))) return BS_ERR_ALIGNMENT;
    if (out_packed) {
        if (!p->scale || !p->bias) return BS_ERR_INVALID_ARG;
        if (!bits_ok(p->out_bits, p->out_sign)) return BS_ERR_INVALID_ARG;
        if (p->out_c_offset < 0 || p->out_c_total < p->out_c_offset + p->O) return BS_ERR_INVALID_ARG;
        if (p->out_c_offset % 32 != 0) return BS_ERR_UNSUPPORTED;
        if (p->O % 32 != 0 && p->out_c_offset + p->O != p->out_c_total) return BS_ERR_UNSUPPORTED;
        if (p->residual) {
            if (!bits_ok(p->res_bits, p->res_sign)) return BS_ERR_INVALID_ARG;
            if (p->res_c_offset < 0 || p->res_c_total < p->res_c_offset + p->O) return BS_ERR_INVALID_ARG;
            if (p->res_c_offset % 32 != 0) return BS_ERR_UNSUPPORTED;
            if (!aligned16(p->residual)) return BS_ERR_ALIGNMENT;
        }
    }
    return BS_OK;
}

static int tc_conv_impl(const uint32_t* act, const int8_t* wgt, const bs_conv_params* p, int32_t* out_i32, uint32_t* out_packed,
                        cudaStream_t st, bool chained)
{
    int rc = tc_validate(p);
    if (rc == BS_OK) rc = tc_validate_outputs(act, wgt, p, out_i32, out_packed);
    return rc == BS_OK ? mma_conv_run(act, wgt, nullptr, p, out_i32, out_packed, st, chained, false) : rc;
}

constexpr int TC_CHAIN_MAX = 4;

// Whether the layers can run as one chain: 2..TC_CHAIN_MAX layers of the same geometry (batch, image, channels = filters, kernel,
// stride 1, output as large as the input), the same activation and weight formats, and whole packed outputs whose width is the
// next layer's activation width.
static bool tc_chain_ok(int n, const bs_conv_params* params)
{
    if (n < 2 || n > TC_CHAIN_MAX || !params) return false;
    const bs_conv_params* p0 = &params[0];
    for (int l = 0; l < n; ++l) {
        const bs_conv_params* p = &params[l];
        if (tc_validate(p) != BS_OK || !bits_ok(p->out_bits, p->out_sign)) return false;
        if (p->stride != 1 || p->pad != (p->R - 1) / 2 || p->O != p->C) return false;
        if (p->out_c_offset != 0 || p->out_c_total != p->O) return false;
        if (p->residual && (!bits_ok(p->res_bits, p->res_sign) || p->res_c_offset != 0 || p->res_c_total != p->O)) return false;
        if (l == 0) continue;
        if (p->N != p0->N || p->C != p0->C || p->H != p0->H || p->W != p0->W || p->R != p0->R || p->S != p0->S || p->a_bits != p0->a_bits ||
            p->a_sign != p0->a_sign || p->w_bits != p0->w_bits || p->w_sign != p0->w_sign)
            return false;
        if (params[l - 1].out_bits != p->a_bits || params[l - 1].out_sign != p->a_sign) return false;
    }
    return mma_conv_run(nullptr, reinterpret_cast<const int8_t*>(16), nullptr, p0, nullptr, nullptr, nullptr, false, true) == BS_OK;
}

// The layers of a chain are launches of their own and use no workspace.  The call still asks for one, of the size callers were always told: a
// word for every 16 x 8 output tile of every layer.
static long long tc_chain_tiles(const bs_conv_params* p)
{
    if (p->R == 1) return ceil_div_ll(static_cast<long long>(p->N) * p->H * p->W, 128);
    const int rows = p->H + p->R - 1;                    // row groups of an image in a stack of small images, halo included
    const int stacked = p->H <= 16 ? (16 - p->H) / rows + 1 : 1;
    return static_cast<long long>(ceil_div(p->W, 8)) * (p->H <= 16 ? 1 : ceil_div(p->H, 16)) * ceil_div(p->N, stacked < p->N ? stacked : p->N);
}

static size_t tc_chain_ws_bytes(int n, const bs_conv_params* p) { return (static_cast<size_t>(n) * tc_chain_tiles(p) + 4) * sizeof(unsigned); }

static int tc_chain_impl(int n, const uint32_t* const* act, const int8_t* const* wgt, const bs_conv_params* params,
                         uint32_t* const* out, void* workspace, size_t workspace_bytes, cudaStream_t st, bool chained)
{
    if (!act || !wgt || !params || !out || !workspace) return BS_ERR_INVALID_ARG;
    if (n < 2 || n > TC_CHAIN_MAX) return BS_ERR_UNSUPPORTED;
    for (int l = 0; l < n; ++l)
        if (!act[l] || !wgt[l] || !out[l]) return BS_ERR_INVALID_ARG;
    if (!tc_chain_ok(n, params)) return BS_ERR_UNSUPPORTED;
    // a layer may read (activations, residual) what an EARLIER layer of the chain wrote, or tensors final before the launch
    for (int l = 0; l < n; ++l)
        for (int k = l; k < n; ++k)
            if (act[l] == out[k] || (params[l].residual && params[l].residual == out[k])) return BS_ERR_UNSUPPORTED;
    if (workspace_bytes < tc_chain_ws_bytes(n, params)) return BS_ERR_INVALID_ARG;
    if (!aligned16(workspace)) return BS_ERR_ALIGNMENT;
    for (int l = 0; l < n; ++l) {
        const int rc = tc_validate_outputs(act[l], wgt[l], &params[l], nullptr, out[l]);
        if (rc != BS_OK) return rc;
    }
    // The layers follow each other as programmatic dependent launches: a layer's set-up and filter fetch run while the layer before
    // it finishes.  (One grid for all layers, its tiles waiting on per-tile counters, saved launches but paid for the counters, the
    // fences and the switch of filters in the middle of the pipeline: 0.326 against 0.290 ms on a residual stack of batch 64.)
    for (int l = 0; l < n; ++l) {
        // the first layer's filters are only known to be final early when the caller says so, the others' as soon as the call is made
        const int rc = mma_conv_run(act[l], wgt[l], nullptr, &params[l], nullptr, out[l], st, chained, false);
        if (rc != BS_OK) return rc;
    }
    return BS_OK;
}

}  // namespace bs

extern "C" size_t bs_tc_weights_bytes(int O, int C, int R, int S)
{
    if (O <= 0 || C <= 0 || R <= 0 || S <= 0 || C % 32 != 0) return 0;
    return static_cast<size_t>((O + 127) / 128 * 128) * R * S * C;
}

// Layers of these widths read so much from the front of the prepared tensor, and its last 16 bytes.
extern "C" size_t bs_tc_weights_read_bytes(int O, int C, int R, int S, int w_bits, int a_bits)
{
    const size_t all = bs_tc_weights_bytes(O, C, R, S);
    if (all == 0 || !bs::bits_ok(w_bits, BS_UNSIGNED) || !bs::bits_ok(a_bits, BS_UNSIGNED)) return 0;
    return bs::mma_nibbles(C, R * S, a_bits, w_bits, BS_UNSIGNED) ? all / (C / 32) * ((C / 32 + 1) / 2) : all;
}

extern "C" int bs_tc_prepare_weights(const uint32_t* wgt_packed, int O, int C, int R, int S, int w_bits, bs_sign_t w_sign,
                                     int a_bits, int8_t* out, void* stream)
{
    if (!wgt_packed || !out || O <= 0 || C <= 0 || R <= 0 || S <= 0) return BS_ERR_INVALID_ARG;
    const bs_sign_t sign = w_sign == BS_SIGNED_NIBBLES ? BS_SIGNED : w_sign;
    if (!bs::bits_ok(w_bits, sign) || a_bits < 1 || a_bits > 4) return BS_ERR_INVALID_ARG;
    if (!bs::aligned16(wgt_packed) || !bs::aligned16(out)) return BS_ERR_ALIGNMENT;
    if (C % 32 != 0) return BS_ERR_UNSUPPORTED;
    const int opad8 = (O + 127) / 128 * 16;
    const bool nibbles = bs::mma_nibbles(C, R * S, a_bits, w_bits, w_sign);
    if (w_sign == BS_SIGNED_NIBBLES && !nibbles) return BS_ERR_UNSUPPORTED;
    const long long nvec = static_cast<long long>(nibbles ? (C / 32 + 1) / 2 : C / 32) * opad8 * R * S * 2 * 8;
    const long long blocks = (nvec + 255) / 256;
    if (blocks > 0x7fffffffLL) return BS_ERR_UNSUPPORTED;
    bs::tc_prepare_weights_kernel<<<static_cast<unsigned>(blocks), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        wgt_packed, out, nvec, O, R * S, C / 32, w_bits, sign, opad8, nibbles,
        static_cast<long long>(C / 32) * opad8 * R * S * 2 * 8 - 1);
    return cudaGetLastError() == cudaSuccess ? BS_OK : BS_ERR_CUDA;
}

extern "C" int bs_tc_supported(const bs_conv_params* p)
{
    if (bs::tc_validate(p) != BS_OK) return 0;
    // the answer of the planner itself; the epilogue fields do not change what fits, so the query plans for raw accumulators
    return bs::mma_conv_run(nullptr, reinterpret_cast<const int8_t*>(16), nullptr, p, nullptr, nullptr, nullptr, false, true) == BS_OK ? 1 : 0;
}

extern "C" int bitserial_conv2d_tc(const uint32_t* act_packed, const int8_t* wgt_tc, const bs_conv_params* p, int32_t* out_i32,
                                   uint32_t* out_packed, void* stream)
{
    return bs::tc_conv_impl(act_packed, wgt_tc, p, out_i32, out_packed, static_cast<cudaStream_t>(stream), false);
}

extern "C" size_t bs_tc_chain_workspace_bytes(const bs_conv_params* layers, int nlayers)
{
    return bs::tc_chain_ok(nlayers, layers) ? bs::tc_chain_ws_bytes(nlayers, layers) : 0;
}

extern "C" int bitserial_conv2d_tc_chain(int nlayers, const uint32_t* const* act_packed, const int8_t* const* wgt_tc,
                                         const bs_conv_params* layers, uint32_t* const* out_packed, void* workspace,
                                         size_t workspace_bytes, int chained, void* stream)
{
    return bs::tc_chain_impl(nlayers, act_packed, wgt_tc, layers, out_packed, workspace, workspace_bytes,
                             static_cast<cudaStream_t>(stream), chained != 0);
}

extern "C" int bitserial_conv2d_tc_chained(const uint32_t* act_packed, const int8_t* wgt_tc, const bs_conv_params* p,
                                           int32_t* out_i32, uint32_t* out_packed, void* stream)
{
    return bs::tc_conv_impl(act_packed, wgt_tc, p, out_i32, out_packed, static_cast<cudaStream_t>(stream), true);
}

extern "C" int bitserial_gemm_tc(const uint32_t* a_packed, const int8_t* w_tc, int M, int N, int K, int a_bits, bs_sign_t a_sign,
                                 int w_bits, bs_sign_t w_sign, const float* scale, const float* bias, int relu, int out_bits,
                                 bs_sign_t out_sign, int32_t* out_i32, uint32_t* out_packed, void* stream)
{
    if (M <= 0 || N <= 0 || K <= 0) return BS_ERR_INVALID_ARG;
    bs_conv_params p{};
    p.N = 1; p.C = K; p.H = 1; p.W = M; p.O = N; p.R = 1; p.S = 1; p.stride = 1; p.pad = 0;
    p.a_bits = a_bits; p.a_sign = a_sign; p.w_bits = w_bits; p.w_sign = w_sign;
    p.scale = scale; p.bias = bias; p.relu = relu; p.out_bits = out_bits; p.out_sign = out_sign;
    p.out_c_offset = 0; p.out_c_total = N; p.i32_layout = BS_NHWC;
    return bs::tc_conv_impl(a_packed, w_tc, &p, out_i32, out_packed, static_cast<cudaStream_t>(stream), false);
}

static int bs_sequence_check(const bs_sequence_layer* layers, int nlayers)
{
    if (!layers || nlayers <= 0) return BS_ERR_INVALID_ARG;
    for (int l = 0; l < nlayers; ++l) {
        const bs_sequence_layer& s = layers[l];
        if (!s.wgt_tc && !s.wgt_packed) return BS_ERR_INVALID_ARG;
        int rc = s.wgt_tc ? bs::tc_validate(&s.p) : bs::tc_validate_shape(&s.p);
        if (rc == BS_OK) rc = bs::tc_validate_outputs(s.act_packed, s.wgt_tc ? static_cast<const void*>(s.wgt_tc) : s.wgt_packed, &s.p, nullptr, s.out_packed);
        if (rc != BS_OK) return rc;
    }
    return BS_OK;
}

extern "C" size_t bs_sequence_workspace_bytes(const bs_sequence_layer* layers, int nlayers)
{
    return bs_sequence_check(layers, nlayers) == BS_OK ? bs::oper_workspace_bytes(layers, nlayers) : 0;
}

extern "C" int bs_sequence_layer_plan(const bs_sequence_layer* layers, int nlayers, int layer, bs_layer_plan* out)
{
    if (!out || layer < 0 || layer >= nlayers) return BS_ERR_INVALID_ARG;
    const int rc = bs_sequence_check(layers, nlayers);
    return rc == BS_OK ? bs::oper_layer_plan(layers, nlayers, layer, out) : rc;
}

extern "C" int bs_sequence_create_ws(const bs_sequence_layer* layers, int nlayers, void* side_stream, void* workspace, size_t workspace_bytes, bs_sequence** out)
{
    if (!out) return BS_ERR_INVALID_ARG;
    const int rc = bs_sequence_check(layers, nlayers);
    if (rc != BS_OK) return rc;
    for (int l = 0; l < nlayers; ++l)
        if (layers[l].aside && !side_stream) return BS_ERR_INVALID_ARG;
    if (workspace && !bs::aligned16(workspace)) return BS_ERR_ALIGNMENT;
    return bs::mma_sequence_create(layers, nlayers, static_cast<cudaStream_t>(side_stream), workspace, workspace_bytes, reinterpret_cast<bs::Sequence**>(out));
}

extern "C" int bs_sequence_create(const bs_sequence_layer* layers, int nlayers, void* side_stream, bs_sequence** out)
{
    return bs_sequence_create_ws(layers, nlayers, side_stream, nullptr, 0, out);
}

extern "C" int bs_sequence_launches(const bs_sequence* sequence)
{
    return sequence ? bs::mma_sequence_launches(reinterpret_cast<const bs::Sequence*>(sequence)) : 0;
}

extern "C" int bs_sequence_run(bs_sequence* sequence, void* stream) { return bs_sequence_run_ready(sequence, nullptr, stream); }

extern "C" const bs_operand_tensor* bs_sequence_input(const bs_sequence* sequence, const uint32_t* packed)
{
    return sequence ? reinterpret_cast<const bs_operand_tensor*>(bs::mma_sequence_input(reinterpret_cast<const bs::Sequence*>(sequence), packed)) : nullptr;
}

extern "C" int bs_sequence_run_ready(bs_sequence* sequence, const bs_operand_tensor* ready, void* stream)
{
    return sequence ? bs::mma_sequence_run(reinterpret_cast<bs::Sequence*>(sequence), reinterpret_cast<const bs::OperTensor*>(ready), static_cast<cudaStream_t>(stream))
                    : BS_ERR_INVALID_ARG;
}

extern "C" void bs_sequence_destroy(bs_sequence* sequence) { bs::mma_sequence_destroy(reinterpret_cast<bs::Sequence*>(sequence)); }
