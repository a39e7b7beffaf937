// Host side of the tensor-core convolution: plan of a layer and launch (kernel: mma_kernel.cuh).
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <unordered_map>
#include <vector>

#include "mma_kernel.cuh"
#include "oper_conv.h"

namespace bs {

// ----------------------------------------------------------------------------- plan

namespace {

constexpr int MM_SMEM_MAX = 224 * 1024;

int up(int v, int m) { return (v + m - 1) / m * m; }

int max_abs_of(int bits, int sign) { return sign == BS_BIPOLAR ? 1 : (sign == BS_UNSIGNED ? (1 << bits) - 1 : 1 << (bits - 1)); }

struct Cand {
    int TN, PT, units, cfg, cps, ns, resident, groups, split, nse, nsb, nacc, f4;
    size_t smem;
    double cost;
};

// Shared-memory layout of a candidate; false when it does not fit.  g carries the problem, the candidate the tiling.
bool mma_layout(MmaArgs& g, Cand& c, int A, int WB, bool int_rows, int sms)
{
    const bool packed_b = WB > 0;
    const int st = g.stride, XT = c.cfg ? 256 : 128, EW = c.cfg ? 8 : 4;
    const int rmax = st == 1 ? g.R - 1 - g.pad : (g.R - 1 - g.pad) >> 1;
    const int Wp = (g.W + st - 1) / st, Hp = (g.H + st - 1) / st;
    g.rmin = st == 1 ? -g.pad : (-g.pad) >> 1;
    g.smin = g.rmin;
    g.flat = g.R == 1 && st == 1 && g.pad == 0;
    g.nplanes = g.R > 1 && st == 2 ? 4 : 1;
    g.strip_q = ceil_div(g.Q, c.ns);
    if (c.ns == 1) {
        g.pitch = Wp - g.smin > g.Q + rmax ? Wp - g.smin : g.Q + rmax;
        g.xoff = 0;
        if (g.R == 1) g.pitch = g.Q;
    } else {
        g.pitch = g.strip_q + rmax - g.smin;
        g.xoff = g.smin;
    }
    const int PH = g.R == 1 ? g.P : (Hp - g.rmin > g.P + rmax ? Hp - g.rmin : g.P + rmax);
    g.hstart = g.rmin * g.pitch + (c.ns == 1 ? g.smin : 0);
    const int BM = 128 * c.PT;
    g.HL = BM + (rmax - g.rmin) * g.pitch + (rmax - g.smin);
    g.NI = g.HL * g.nplanes;
    g.img_rows = PH;
    const long long per_img = static_cast<long long>(PH) * g.pitch;
    const long long total = static_cast<long long>(g.N) * c.ns * per_img;
    if (total + per_img + 4096 + g.HL > 0x7fffffffLL || g.NI > 4096) return false;
    // the kernel counts input pixels (stride 2: up to four times the positions) and the words of a packed filter tile in 32 bits
    if (static_cast<long long>(g.N) * g.H * g.W > 0x7fffffffLL || (packed_b && static_cast<long long>(c.TN) * g.RS * g.Cw * WB > 0x7fffffffLL)) return false;
    g.total = static_cast<int>(total);
    g.d_img = make_div(static_cast<int>(per_img));
    g.d_pitch = make_div(g.pitch);
    g.d_strips = make_div(c.ns);
    g.TN = c.TN; g.PT = c.PT; g.units = c.units;
    g.nunits = (g.Cw + 1) / 2;
    g.nblk = g.f4 ? g.nunits : g.Cw;
    const int bpu = g.f4 ? 1 : 2;                          // K steps of a unit
    g.nchunks = ceil_div(g.nunits, c.units);
    g.tiles_m = static_cast<int>(ceil_div_ll(total, BM));
    g.tiles_o = ceil_div(g.O, c.TN);
    g.d_rs = make_div(g.RS);
    // An item split over a cluster: every CTA streams its chunks, at least two of them (with one, the sums cost what it saves).  No more CTAs than two thirds of the SMs: clusters need SMs of one
    // GPC that are free at the same time, and 128 CTAs in clusters of four already ran 20 to 50 % longer than without the split.
    g.split = c.split;
    g.split_log = c.split == 1 ? 0 : c.split == 2 ? 1 : c.split == 4 ? 2 : 3;
    if (c.split > 1 && (c.resident || c.cps != 1 || g.nchunks < 2 * c.split || static_cast<long long>(g.tiles_m) * g.tiles_o * c.split * 3 > 2 * sms)) return false;
    const int red_bytes = (c.split - 1) * 128 * c.PT * c.TN * 4;
    g.groups = c.groups;
    const int GT = XT / c.groups;                          // threads of an expander group
    g.nslots = ceil_div(g.NI * c.units, GT);
    g.bslots = ceil_div(c.TN * g.RS * c.units, GT);
    auto piece = [&](int bits) { return (2 * bits) % 4 == 0 && (g.Cw * bits) % 4 == 0 ? 16 : ((g.Cw * bits) % 2 == 0 ? 8 : 4); };
    g.psz = piece(A);
    g.bpsz = piece(WB > 0 ? WB : 1);
    // boxes of [row][units]: rows of 16-byte multiples in memory, box rows of 16 .. 128 bytes
    g.rowA = c.units * 8 * A;
    g.rowB = c.units * 8 * WB;
    const bool fb = packed_b && !c.resident;
    g.tma = g.flat && (g.Cw * A) % 4 == 0 && g.rowA % 16 == 0 && g.rowA <= 128 && (!fb || ((g.Cw * WB) % 4 == 0 && g.rowB % 16 == 0 && g.rowB <= 128));
    g.nsp = g.tma && c.groups == 1 ? 3 : 2 * c.groups;
    auto swizzle = [](int row) { return row == 32 ? 1 : row == 64 ? 3 : row == 128 ? 7 : 0; };
    g.swzA = swizzle(g.rowA);
    g.swzB = swizzle(g.rowB);
    g.one_word = g.f4 && g.Cw == 1 && !g.tma;
    g.e_bytes = up((g.one_word ? 1 : 2 * bpu) * c.units * g.NI * 16, 128);
    g.b_bytes = c.units * bpu * c.TN * g.RS * 32;
    g.stg_bytes = g.tma ? up(BM * g.rowA, 1024) : g.nslots * GT * (g.one_word ? 4 : 8) * A;
    g.bstg_bytes = !fb ? 0 : g.tma ? up(c.TN * g.rowB, 1024) : g.bslots * GT * 8 * WB;
    const int rel_bytes = g.flat ? 0 : up(g.NI * 4 * (1 + (c.units == 1 ? g.nsp + c.groups : 0)), 16);      // relative rows; located pixels of each group, one table more than stages
    const int pix_bytes = rel_bytes + (fb && !g.tma && c.units == 1 ? up(c.TN * g.RS * 4, 16) : 0);
    const int cap = c.cfg ? 222 * 1024 : 111 * 1024;
    const int tab = c.TN * (g.f4 && A == 3 && g.a_kind == 0 ? 12 : 8) + 64;          // scales, biases, residual multipliers, sums of filters
    const int fixed = tab + 320 + red_bytes + (g.tma ? 1024 : 0) + (int_rows ? EW * 4096 : 0) + 256 + pix_bytes;
    const long long filters = c.resident ? static_cast<long long>(g.nblk) * c.TN * g.RS * 32 : 0;
    const long long rest = fixed + static_cast<long long>(g.nsp) * (g.stg_bytes + g.bstg_bytes) + filters;
    c.nsb = 0;
    long long used = 0;
    int nse = 4;
    if (c.resident) {
        for (; nse >= 2; --nse) {
            used = rest + static_cast<long long>(nse) * g.e_bytes;
            if (used <= cap) break;
        }
        if (nse < 2) return false;
    } else if (packed_b) {
        for (; nse >= 2; --nse) {
            used = rest + static_cast<long long>(nse) * (g.e_bytes + g.b_bytes);
            if (used <= cap) break;
        }
        if (nse < 2) return false;
    } else {
        bool fit = false;
        for (int n = 4; n >= 1 && !fit; --n) {
            used = rest + static_cast<long long>(n) * (g.e_bytes + g.b_bytes);
            if (used <= cap) { nse = n; c.nsb = n; fit = true; }
        }
        if (!fit) return false;
    }
    if (nse < c.groups) return false;
    c.nse = nse;
    g.nse = nse; g.nsb = c.resident ? 0 : (packed_b ? nse : c.nsb);
    const int sf = g.f4 ? MM_SF_COLS : 0, cols = 512 / (c.cfg ? 1 : 2) - sf;
    if (2 * c.PT * c.TN <= cols) c.nacc = 2;
    else if (c.PT * c.TN <= cols) c.nacc = 1;
    else return false;
    g.nacc = c.nacc;
    int tc = 32;
    g.sf_col = c.nacc * c.PT * c.TN;
    while (tc < g.sf_col + sf) tc *= 2;
    g.tmem_cols = tc;
    long long off = c.resident ? filters : static_cast<long long>(g.nsb) * g.b_bytes;
    g.off_e = static_cast<int>(off);                off += static_cast<long long>(nse) * g.e_bytes;
    if (g.tma) off = (off + 1023) / 1024 * 1024;
    g.off_stg = static_cast<int>(off);              off += static_cast<long long>(g.nsp) * g.stg_bytes;
    g.off_bstg = static_cast<int>(off);             off += static_cast<long long>(g.nsp) * g.bstg_bytes;
    g.off_pix = static_cast<int>(off);              g.off_brow = static_cast<int>(off) + rel_bytes;
    off += pix_bytes;
    off = (off + 127) / 128 * 128;
    g.off_out = static_cast<int>(off);              if (int_rows) off += EW * 4096;
    g.off_tab = static_cast<int>(off);              off += tab;
    off = (off + 15) / 16 * 16;
    g.off_bar = static_cast<int>(off);              off += 320;
    g.off_red = static_cast<int>(off);              off += red_bytes;
    g.bulk_b = packed_b && c.resident && static_cast<long long>(c.TN) * g.RS * g.Cw * WB * 4 <= static_cast<long long>(nse) * g.e_bytes &&
               (static_cast<long long>(g.O % c.TN) * g.RS * g.Cw * WB) % 4 == 0;
    c.smem = static_cast<size_t>(off);
    return off <= cap + 512;
}

// Time model of a candidate in SM cycles: the pipeline of one CTA (expansion, MMAs, epilogue; a stage's hand-off included) over
// its items, plus what nothing overlaps at both ends.  The constants are fitted to timed plans (B200 at 1.95 GHz): int8 to about 2500 of
// 45 layers and products (1 to 300 pixels wide, 32 to 4608 channels, batches 1 to 64), nibbles to 17000 of 77; then what only packed
// filters and int32 outputs have (filt_*, resident_once, e_i32, e_nchw, rows*) to 60000 plans of 670 calls on their own, three quarters of
// them, judged on the rest: the plan with the lowest modelled time is on average 3.8 % slower than the fastest there on either form, 4.3 and
// 4.9 % before (a flat 1900 cycles for resident filters of less than an item per SM, int32 in rows of pixels at the rate of odd rows of filters).
struct MmaFit {
    double mma_chunk;                       // cycles per chunk beside its MMAs
    double unit, one_word, flat, staged;    // expansion, instructions per warp and 64-channel unit of 32 rows: arithmetic, of 32 channels only, copies by TMA, by thread
    double filt_flat, filt_staged;          // packed filters streamed, instructions per 32 rows and unit
    double x_cpi, x_chunk, x_group, x_once; // cycles per such instruction, per chunk; share by which a further group overlaps; once
    double e_res, e_codes, e_i32, e_nchw, e_cpi, e_once;        // epilogue, instructions per block of 32 x 32 outputs (int32 in rows of filters or of pixels); cycles per instruction; per item
    double e_pair;                          // of e_res and e_codes where two row tiles share a pass
    double rows, rows_odd;                  // bytes per cycle of int32 rows, of rows that are not multiples of 16 bytes
    double split;                           // cycles of a split item beside its sums
    double l2;                              // bytes per cycle of streamed prepared filters
    double ipc, two_first, start, filt_resident, resident_once, streamed, one_stage, half;   // filt_resident, resident_once: resident packed filters, cycles per channel word of 32 rows, per launch
};
constexpr MmaFit FIT_INT8 = {148, 102, 102, 1, 41, 20, 59, 5.34, 629, 0.83, 628, 215, 138, 94, 113, 4.59, 997, 1, 17.2, 12.8, 2200, 68.7, 3.08, 1.19, 4215, 102, 910, 1.07, 1.11, 0.93};
constexpr MmaFit FIT_NIBBLES = {262, 63, 31, 1, 92.5, 77.8, 123, 5.49, 457, 0.889, 705, 247, 114, 263, 122, 4.01, 982, 0.931, 19.2, 15, 4236, 98.3, 1.45, 1.226, 3484, 205, 1540, 1.076, 0.961, 0.934};

double mma_cost(const MmaArgs& g, const Cand& c, int A, int WB, bool packed_out, int sms)
{
    const MmaFit& k = g.f4 ? FIT_NIBBLES : FIT_INT8;
    const bool packed_b = WB > 0;
    const double mma = c.TN == 32 ? 42 : c.TN == 64 ? 49 : c.TN == 128 ? 65 : 129;      // cycles per MMA of 128 x TN x (32 int8 or 64 nibbles)
    const int W = c.cfg ? 8 : 4;                                   // expander warps, epilogue warps
    const int nchunks = ceil_div(g.nchunks, c.split);              // of one CTA
    const double share = static_cast<double>(nchunks) / g.nchunks;
    const double t_m = share * c.PT * g.RS * g.nblk * mma + k.mma_chunk * nchunks;
    const int row_groups = ceil_div(g.NI, 32);
    double xi = share * row_groups * g.nunits * ((g.one_word ? k.one_word : A <= 2 ? k.unit : k.unit + 9.0) + (g.tma ? k.flat : k.staged));
    if (!c.resident && packed_b) xi += share * c.TN * g.RS / 32.0 * g.nunits * (WB <= 2 ? (g.tma ? k.filt_flat : k.filt_staged) : 69.0);
    const double units_of_work = static_cast<double>(row_groups) * c.units * c.groups / W;       // per warp of a group and chunk
    const double chunk = xi / nchunks * c.groups / W * (ceil(units_of_work) / units_of_work) * k.x_cpi + k.x_chunk;
    const double t_x = chunk * nchunks / (1.0 + (c.groups - 1) * k.x_group) + k.x_once;
    const double block = packed_out ? (g.has_residual ? k.e_res : k.e_codes) * (c.PT > 1 ? k.e_pair : 1.0) : g.i32_nhwc ? k.e_i32 : k.e_nchw, rows = g.i32_nhwc && g.O % 4 ? k.rows_odd : k.rows;
    double t_e = ceil_div(c.PT * (c.TN / 32), W / 4) * block * k.e_cpi + k.e_once;
    if (!packed_out && c.PT * 128.0 * c.TN * 4 / rows > t_e) t_e = c.PT * 128.0 * c.TN * 4 / rows;
    // sums through shared memory of the cluster
    if (c.split > 1) t_e += k.split + ceil_div(c.PT * (c.TN / 32), W / 4) * 200.0 * (c.split - 1);
    const double t_b = (!c.resident && !packed_b) ? share * c.TN * g.RS * g.nblk * 32 / k.l2 : 0.0;       // L2 -> shared memory
    const long long items = static_cast<long long>(g.tiles_m) * g.tiles_o * c.split;
    long long ctas = static_cast<long long>(sms) * c.cps;
    if (c.resident) ctas = ctas / g.tiles_o * g.tiles_o;
    if (ctas < 1) return 1e18;
    if (ctas > items) ctas = items;
    const double per_cta = static_cast<double>(ceil_div_ll(items, ctas)), active = static_cast<double>(ceil_div_ll(ctas, sms));
    const double issue = (xi + c.PT * 4.0 * (c.TN / 32) * block) / k.ipc;
    const double t_mb = t_m > t_b ? t_m : t_b;
    double step = c.nacc == 2 ? (t_mb > t_e ? t_mb : t_e) : t_mb + t_e;
    if (t_x > step) step = t_x;
    if (active * t_mb > step) step = active * t_mb;
    if (active * issue > step) step = active * issue;
    const double rest_x = t_x > chunk ? t_x - chunk : 0.0;
    double first = chunk + (t_mb > rest_x ? t_mb : rest_x) + t_e;
    if (active > 1.0) first *= k.two_first;
    double t = k.start + first + (per_cta - 1.0) * step;
    if (c.resident && packed_b) t += c.TN * g.RS * (g.f4 ? 2 * g.nblk : g.Cw) / 32.0 * k.filt_resident / (2 * W) * 4.0;
    // Resident packed filters of a call on its own also hold up the first pixel until every warp has expanded its share, where streamed
    // ones come with it (behind a chained layer that happens while the other still runs).
    if (c.resident && packed_b && !g.early_b) t += k.resident_once;
    if (!c.resident && !packed_b) t *= k.streamed;
    if (c.nse < 2) t *= k.one_stage;
    if (!c.cfg) t *= k.half;
    return t;
}

}  // namespace

// Everything about a layer that does not depend on its pointers: filled arguments, kernel, grid.
struct MmaPlan {
    MmaArgs g;
    MmaKernel kern;
    unsigned grid, block;
    int smem;
    int rc;                 // BS_OK, or why there is no plan
};

enum : int { MM_PREPARED = 1, MM_I32 = 2, MM_CODES = 4, MM_RESIDUAL = 8, MM_CHAINED = 16, MM_QUERY = 32, MM_ALONE = 64 };

static int make_plan(MmaPlan& plan, const bs_conv_params* p, int flags, int sms)
{
    const bool out_i32 = flags & MM_I32, out_packed = flags & MM_CODES, residual = flags & MM_RESIDUAL, packed_b = !(flags & MM_PREPARED);
    // the callers have validated sizes, bit widths, pointers and output slices; what this path refuses is said here
    if (p->stride > 2 || p->R > 7) return BS_ERR_UNSUPPORTED;
    if (p->a_sign == BS_BIPOLAR && p->w_sign == BS_BIPOLAR && p->C % 32 != 0) return BS_ERR_UNSUPPORTED;
    if (residual && p->res_c_offset % 32 != 0) return BS_ERR_UNSUPPORTED;
    MmaArgs& g = plan.g;
    const int A = p->a_bits;
    g.has_residual = residual;
    g.res_scale = p->res_scale;
    g.N = p->N; g.H = p->H; g.W = p->W; g.O = p->O; g.R = p->R; g.RS = p->R * p->S; g.stride = p->stride; g.pad = p->pad;
    g.P = (p->H + 2 * p->pad - p->R) / p->stride + 1;
    g.Q = (p->W + 2 * p->pad - p->S) / p->stride + 1;
    g.Cw = ceil_div(p->C, 32);
    auto kind = [](int sign) { return sign == BS_UNSIGNED ? 0 : sign == BS_BIPOLAR ? 2 : 1; };
    g.a_kind = kind(p->a_sign); g.w_kind = kind(p->w_sign);
    g.relu = p->relu; g.out_bits = p->out_bits; g.out_sign = p->out_sign;
    g.out_cw_off = p->out_c_offset / 32; g.out_cw_total = ceil_div(p->out_c_total > 0 ? p->out_c_total : 1, 32);
    g.res_bits = p->res_bits; g.res_sign = p->res_sign; g.res_c_off = p->res_c_offset;
    g.res_cw_total = ceil_div(p->res_c_total > 0 ? p->res_c_total : 1, 32);
    g.i32_nhwc = p->i32_layout == BS_NHWC;
    g.opad = up(p->O, 128);
    // Nibbles, but int8 for packed filters where the reduction is so short that nibbles save few MMAs or none (up to 32 channels leave half of a
    // K step empty) and the way out decides: int8 sums need no conversion to int32.  Time on nibbles over time on int8, the
    // plans chosen for 220 layers: int32 in rows of pixels, 1x1: 32 channels 1.07, 64 and 96 1.05, 128 1.03, 160 and 192 1.02, to 288 1.00,
    // more 0.96 (14 x 19 x 72 x 70, 125 filters: 12.1 -> 10.2 us); larger windows, up to 32 channels, 2048 outputs per SM and more: 3x3 1.01, 5x5 1.10, fewer
    // outputs 0.98 and 0.97; codes of 5x5 windows over up to 32 channels 1.12 and 0.89 on these sides, of 3x3 windows 0.96 and 0.94.
    const bool short_k = g.Cw == 1 && static_cast<double>(g.N) * g.P * g.Q * g.O >= 2048.0 * sms;
    const bool pixel_rows = out_i32 && !out_packed && !g.i32_nhwc;
    g.f4 = (packed_b ? mma_nibbles_packed(p->C, g.RS, p->a_bits, p->w_bits, p->w_sign) : mma_nibbles(p->C, g.RS, p->a_bits, p->w_bits, p->w_sign)) &&
           !(packed_b && (pixel_rows ? short_k || (g.R == 1 && g.Cw <= 6) : short_k && g.R >= 5 && !out_i32));
    // Unsigned activations of three bits need the filters' sums, which only resident filters give: such plans on nibbles against all on int8, by their
    // modelled time, with 6 % for int8.  Of 135 layers with larger windows, timed on both forms, 6 go to nibbles, which take 0.36 to 0.83 of int8's time.
    // Without the 6 % 14 would, the others 0.67 to 0.92, but of 90 more layers one then loses (59 x 37 x 68 x 68, 448 filters, stride 2: 50.7 -> 55.0 us),
    // and with 11 % for nibbles 39 would, four of them slower.  1x1 stays on int8: what the 6 % leave of 169 products and layers takes 0.82 to 1.19
    // of int8's time (111 x 3428 x 2688: 11.7 -> 14.0 us; 7 x 239 x 88 x 88, 64 filters: 7.6 -> 8.4), and the model does not tell them apart.
    if (A == 3 && p->a_sign == BS_UNSIGNED && g.R == 1) g.f4 = 0;
    const bool offset = g.f4 && A == 3 && p->a_sign == BS_UNSIGNED;
    // Signed activations of three bits, filters of three bits under narrower ones: nibbles for larger windows, which take 0.88 of int8's time over 348
    // layers of the former, 0.89 over 177 of the latter, and up to 1.2 in one of 25, which the model does not tell from the others.  1x1: both forms
    // by their modelled time, with 10 % for nibbles.  316 calls timed on both: 0.93 of int8's time; on nibbles alone 7 lose more than 3 %, large products a
    // quarter (2049 x 2620 x 4182: 92.6 -> 117.7 us); without the 10 % 55 lose more than 3 % against nibbles, with them 16, at most 12 %.
    const bool either = g.f4 && g.R == 1 && (A == 3 || p->w_bits == 3);
    const double bound = static_cast<double>(p->C) * g.RS * max_abs_of(p->a_bits, p->a_sign) * max_abs_of(p->w_bits, p->w_sign);
    g.acc_bound = static_cast<float>(bound);
    g.preset = out_packed && !out_i32 && bound < 4.0e6 && p->out_sign != BS_BIPOLAR &&
               (!residual || (p->res_sign == BS_UNSIGNED && fabsf(p->res_scale) < 3.9f && (p->res_scale == 0.0f || fabsf(p->res_scale) > 1e-18f)));
    {
        int qmin, qmax;
        code_limits(p->out_bits > 0 ? p->out_bits : 1, p->out_sign, qmin, qmax);
        const bool lo0 = qmin == 0 || p->relu;
        // the forms with a residual read its words and a table of multipliers that is written only where there is one
        if (!lo0) g.epi = residual ? 5 : 4;
        else if (p->out_bits <= 2 && (!residual || p->res_bits <= 2)) g.epi = residual ? 1 : 0;
        else g.epi = residual ? 3 : 2;
    }
    g.early_b = flags & MM_CHAINED ? 1 : 0;
    const bool int_rows = out_i32 && g.i32_nhwc && p->R == 1 && p->stride == 1 && p->pad == 0;

    Cand best{};
    best.cost = 1e30;
    bool found = false;
    auto consider = [&](Cand c) {
        MmaArgs t = g;
        if (!mma_layout(t, c, A, packed_b ? p->w_bits : 0, int_rows, sms)) return;
        c.cost = mma_cost(t, c, A, packed_b ? p->w_bits : 0, out_packed, sms);
        c.f4 = g.f4;
        if (g.f4) c.cost *= offset ? 1.06 : either ? 0.9 : 1.0;
        if (c.cost < best.cost) { best = c; found = true; }
    };
    int ns_list[12], nns = 0;
    if (g.R == 1) ns_list[nns++] = 1;
    else {
        static const int widths[] = {1 << 30, 112, 84, 64, 48, 40, 32, 24, 20, 16, 12, 8};      // outputs per strip row, roughly
        for (int w : widths) {
            const int ns = w > g.Q ? 1 : ceil_div(g.Q, w);
            if (nns == 0 || ns_list[nns - 1] != ns) ns_list[nns++] = ns;
        }
    }
#ifdef BS_TUNING
    int ov[8] = {0, 0, 0, -1, 0, -1, 0, 0};    // TN, PT, units, config, strips, resident, groups, split; 0 / -1: free
    if (const char* e = getenv("BS_MM")) sscanf(e, "%d,%d,%d,%d,%d,%d,%d,%d", ov, ov + 1, ov + 2, ov + 3, ov + 4, ov + 5, ov + 6, ov + 7);
#endif
    for (int form = 0; form < (offset || either ? 2 : 1); ++form, g.f4 = 0)
    for (int TN = 32; TN <= 256; TN *= 2) {
        if (TN > 32 && TN / 2 >= up(p->O, 32)) continue;
        if (TN == 256 && !packed_b && g.opad % 256 != 0) continue;
        for (int PT = 1; PT <= 4; PT *= 2)
            for (int cfg = 0; cfg < 3; ++cfg)
                for (int k = 0; k < nns; ++k)
                    for (int units = 1; units <= (g.R == 1 ? 4 : 1); units *= 2) {
                        if (units > 1 && units > (g.Cw + 1) / 2) continue;
                        for (int v = 0; v < 18; ++v) {
                            const int res = v & 1, groups = 1 << ((v >> 1) % 3), split = 1 << (v / 6);
                            if ((groups > 2 && cfg != 1) || (offset && form == 0 && !res)) continue;
                            // Splits only for calls on their own: between the layers of a stack the change to another kernel costs what
                            // the split gains (18- and 50-layer stacks of batch 1 to 17: 2 % faster to 3 % slower).
                            // 32 filters wide: wider tiles expand more filters per CTA, and 32 without a split then beats them
                            // (3734 x 70 x 2944: 13.7 us; 128 wide and split: 19.9; 3000 x 64 x 4096: 32 wide 13.9, split 11.1).
                            if (split > 1 && (!(flags & MM_ALONE) || res || cfg != 1 || PT > 1 || TN > 32)) continue;
#ifdef BS_TUNING
                            if ((ov[0] && TN != ov[0]) || (ov[1] && PT != ov[1]) || (ov[2] && units != ov[2]) || (ov[3] >= 0 && cfg != ov[3]) ||
                                (ov[4] && ns_list[k] != ov[4]) || (ov[5] >= 0 && res != ov[5]) || (ov[6] && groups != ov[6]) || (ov[7] && split != ov[7]))
                                continue;
#endif
                            Cand c{};
                            c.TN = TN; c.PT = PT; c.units = units; c.cfg = cfg == 1; c.cps = cfg == 0 ? 2 : 1; c.ns = ns_list[k]; c.resident = res; c.groups = groups; c.split = split;
                            consider(c);
                        }
                    }
    }
    if (!found) return BS_ERR_UNSUPPORTED;
    g.f4 = best.f4;
    if (!mma_layout(g, best, A, packed_b ? p->w_bits : 0, int_rows, sms)) return BS_ERR_UNSUPPORTED;
#ifdef BS_TUNING
    if (getenv("BS_MM_VERBOSE"))
        fprintf(stderr, "mma plan: N%d C%d %dx%d O%d k%d s%d A%d W%d %s -> TN %d PT %d units %d cfg %d x %d strips %d resident %d groups %d split %d nse %d nsb %d units %d nacc %d HL %d NI %d tiles %d x %d smem %zu cost %.0f\n",
                p->N, p->C, p->H, p->W, p->O, p->R, p->stride, A, p->w_bits, packed_b ? "packed" : "prepared", best.TN, best.PT, best.units, best.cfg, best.cps, best.ns, best.resident, best.groups, best.split,
                best.nse, g.nsb, g.nunits, g.nacc, g.HL, g.NI, g.tiles_m, g.tiles_o, best.smem, best.cost);
#endif
    if (flags & MM_QUERY) return BS_OK;
    g.status = status_device_ptr();
    if (!g.status) return BS_ERR_CUDA;
    // int32 += int8 x int8, or float += e2m1 x e2m1 with ue8m0 scale factors; TN columns, 128 rows
    g.idesc = (g.f4 ? (1u << 7) | (1u << 10) | (1u << 23) : (2u << 4) | (1u << 7) | (1u << 10)) | (static_cast<unsigned>(g.TN >> 3) << 17) | (static_cast<unsigned>(128 >> 4) << 24);
    const int cps = best.cps;
    const long long items = static_cast<long long>(g.tiles_m) * g.tiles_o;
    long long grid = static_cast<long long>(sms) * cps;
    if (best.resident) grid = grid / g.tiles_o * g.tiles_o;
    if (best.split > 1) grid = items * best.split;
    else if (grid > items) grid = items;
    const int wb = packed_b ? p->w_bits : 0;
    const bool half = !best.cfg, split = best.split > 1;
    plan.kern = g.f4 ? (A == 1 ? mma_kernel_f1(wb, half, split) : A == 2 ? mma_kernel_f2(wb, half, split) : mma_kernel_f3(wb, half, split, offset)) : A == 1 ? mma_kernel_a1(wb, half, split) : A == 2 ? mma_kernel_a2(wb, half, split) : A == 3 ? mma_kernel_a3(wb, half, split) : mma_kernel_a4(wb, half, split);
    plan.grid = static_cast<unsigned>(grid);
    plan.block = best.cfg ? MmaShape<false>::THREADS : MmaShape<true>::THREADS;
    plan.smem = static_cast<int>(best.smem);
    // the limit is a property of the kernel, not of the launch: set to the largest any plan uses
    if (cudaFuncSetAttribute(plan.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, MM_SMEM_MAX) != cudaSuccess) {
        cudaGetLastError();
        return BS_ERR_CUDA;
    }
    return BS_OK;
}

// Plans by shape, format and device: a program calls the same few layers again and again, and a search costs tens of
// microseconds.  At most MAX_PLANS are kept (about 600 bytes each); when full the table starts over.
namespace {
struct PlanKey {
    int v[28];
    bool operator==(const PlanKey& o) const { return memcmp(v, o.v, sizeof v) == 0; }
};
struct PlanHash {
    size_t operator()(const PlanKey& k) const
    {
        uint64_t h = 1469598103934665603ull;
        for (int x : k.v) h = (h ^ static_cast<uint32_t>(x)) * 1099511628211ull;
        return static_cast<size_t>(h ^ (h >> 29));
    }
};
constexpr size_t MAX_PLANS = 4096;
}  // namespace

static int find_plan(MmaPlan& out, const bs_conv_params* p, int flags)
{
    int dev = -1;
    int sms = device_sm_count();
    if (sms <= 0) {
        if (!(flags & MM_QUERY)) return BS_ERR_CUDA;
        sms = 148;                      // a support query without a device plans for a full B200
    } else if (cudaGetDevice(&dev) != cudaSuccess) {
        return BS_ERR_CUDA;
    }
    // What a caller leaves in fields that its outputs do not depend on reaches neither the key nor the plan: without codes the epilogue's,
    // without a residual the residual's.
    bs_conv_params q = *p;
    if (!(flags & MM_CODES)) q.relu = q.out_bits = q.out_sign = q.out_c_offset = q.out_c_total = 0;
    if (!(flags & MM_RESIDUAL)) {
        q.res_bits = q.res_sign = q.res_c_offset = q.res_c_total = 0;
        q.res_scale = 0.0f;
    }
    int scale_bits = 0;
    memcpy(&scale_bits, &q.res_scale, 4);
    const PlanKey key = {{q.N, q.C, q.H, q.W, q.O, q.R, q.S, q.stride, q.pad, q.a_bits, q.a_sign, q.w_bits, q.w_sign, q.relu, q.out_bits, q.out_sign,
                          q.out_c_offset, q.out_c_total, q.res_bits, q.res_sign, q.res_c_offset, q.res_c_total, scale_bits, q.i32_layout, flags, dev, sms, 0}};
    static std::unordered_map<PlanKey, MmaPlan, PlanHash> plans;
    static std::mutex mu;
    {
        std::lock_guard<std::mutex> lock(mu);
#ifdef BS_TUNING
        plans.clear();
#endif
        auto it = plans.find(key);
        if (it != plans.end()) { out = it->second; return out.rc; }
    }
    MmaPlan plan{};
    plan.rc = make_plan(plan, &q, flags, sms);
    if (plan.rc == BS_OK || plan.rc == BS_ERR_UNSUPPORTED) {
        std::lock_guard<std::mutex> lock(mu);
        if (plans.size() >= MAX_PLANS) plans.clear();
        plans.emplace(key, plan);
    }
    out = plan;
    return plan.rc;
}

// Tensor map of a row-major matrix of `rows` rows of `words` words, fetched in boxes of box_rows rows x row_bytes bytes.
static bool encode_rows(CUtensorMap* tm, const uint32_t* base, int rows, int words, int row_bytes, int box_rows)
{
    typedef CUresult (*Fn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                           CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    static Fn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* q = nullptr;
        cudaDriverEntryPointQueryResult r;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &q, cudaEnableDefault, &r) == cudaSuccess && r == cudaDriverEntryPointSuccess) fn = reinterpret_cast<Fn>(q);
    });
    if (!fn) return false;
    const cuuint64_t dims[2] = {static_cast<cuuint64_t>(words), static_cast<cuuint64_t>(rows)};
    const cuuint64_t strides[1] = {static_cast<cuuint64_t>(words) * 4};
    const cuuint32_t box[2] = {static_cast<cuuint32_t>(row_bytes / 4), static_cast<cuuint32_t>(box_rows)}, es[2] = {1, 1};
    const CUtensorMapSwizzle sw = row_bytes == 32 ? CU_TENSOR_MAP_SWIZZLE_32B : row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B :
                                  row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE;
    return fn(tm, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<uint32_t*>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
              CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Plan of a layer with its pointers filled in.
static int bind_plan(MmaPlan& plan, const uint32_t* act, const int8_t* wgt, const uint32_t* wgt_packed, const bs_conv_params* p, int32_t* out_i32,
                     uint32_t* out_packed, bool chained, bool plan_only, bool alone)
{
    const int flags = (wgt ? MM_PREPARED : 0) | (out_i32 ? MM_I32 : 0) | (out_packed ? MM_CODES : 0) | (out_packed && p->residual ? MM_RESIDUAL : 0) |
                      (chained ? MM_CHAINED : 0) | (plan_only ? MM_QUERY : 0) | (alone && !chained ? MM_ALONE : 0);
    const int rc = find_plan(plan, p, flags);
    if (rc != BS_OK || plan_only) return rc;
    MmaArgs& g = plan.g;
    g.act = act; g.wgt = wgt; g.wgt_packed = wgt_packed; g.out_i32 = out_i32; g.out_packed = out_packed;
    g.scale = p->scale; g.bias = p->bias;
    g.residual = out_packed ? p->residual : nullptr;
    if (g.tma) {
        if (!encode_rows(&g.tmA, act, g.total, g.Cw * p->a_bits, g.rowA, 128 * g.PT < 256 ? 128 * g.PT : 256)) return BS_ERR_CUDA;
        if (!wgt && g.nsb > 0 && !encode_rows(&g.tmB, wgt_packed, g.O, g.Cw * p->w_bits, g.rowB, g.TN)) return BS_ERR_CUDA;
    }
    return BS_OK;
}

// Every launch may start while the kernel before it drains (barriers, tensor memory, filter fetch when the caller allows); the
// kernel waits for that kernel itself before it reads or writes anything the stream orders.
static int launch_plan(const MmaPlan& plan, cudaStream_t st)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(plan.grid);
    cfg.blockDim = dim3(plan.block);
    cfg.dynamicSmemBytes = static_cast<size_t>(plan.smem);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = static_cast<unsigned>(plan.g.split);
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = plan.g.split > 1 ? 2 : 1;
    if (cudaLaunchKernelEx(&cfg, plan.kern, plan.g) != cudaSuccess) {
        cudaGetLastError();
        return BS_ERR_CUDA;
    }
    return BS_OK;
}

int mma_conv_run(const uint32_t* act, const int8_t* wgt, const uint32_t* wgt_packed, const bs_conv_params* p, int32_t* out_i32,
                 uint32_t* out_packed, cudaStream_t st, bool chained, bool plan_only)
{
    MmaPlan plan;
    const int rc = bind_plan(plan, act, wgt, wgt_packed, p, out_i32, out_packed, chained, plan_only, true);
    return rc != BS_OK || plan_only ? rc : launch_plan(plan, st);
}

// A bound sequence of layers: plans, pointers and tensor maps as of its creation, the events of its forks and joins.
struct Sequence {
    struct Step {
        MmaPlan plan;
        cudaEvent_t fork, done;     // set for a step that runs beside its successors
        int join[4];                // steps beside which this one must have finished, -1: none
    };
    std::vector<Step> steps;
    cudaStream_t side;
    OperSequence* oper;             // the layers on operand tensors, or null: as planned in the steps
    ~Sequence()
    {
        if (oper) oper_destroy(oper);
        for (Step& s : steps) {
            if (s.fork) cudaEventDestroy(s.fork);
            if (s.done) cudaEventDestroy(s.done);
        }
    }
};

int mma_sequence_create(const bs_sequence_layer* layers, int n, cudaStream_t side, void* workspace, size_t bytes, Sequence** out)
{
    Sequence* q = new (std::nothrow) Sequence;
    if (!q) return BS_ERR_CUDA;
    q->side = side;
    q->oper = workspace ? oper_create(layers, n, workspace, bytes) : nullptr;
    q->steps.resize(static_cast<size_t>(n));
    for (Sequence::Step& s : q->steps) s.fork = s.done = nullptr;
    for (int i = 0; i < n; ++i) {
        const bs_sequence_layer& l = layers[i];
        Sequence::Step& s = q->steps[i];
        // a layer beside its successors starts from an event, not from the kernel before it: no early filter fetch
        int rc = q->oper ? BS_OK : bind_plan(s.plan, l.act_packed, l.wgt_tc, l.wgt_packed, &l.p, nullptr, l.out_packed, l.chained && !l.aside, false, false);
        for (int k = 0; k < 4; ++k) {
            s.join[k] = l.join[k];
            if (l.join[k] >= i) rc = BS_ERR_INVALID_ARG;
        }
        if (rc == BS_OK && l.aside &&
            (cudaEventCreateWithFlags(&s.fork, cudaEventDisableTiming) != cudaSuccess || cudaEventCreateWithFlags(&s.done, cudaEventDisableTiming) != cudaSuccess)) {
            cudaGetLastError();
            rc = BS_ERR_CUDA;
        }
        if (rc != BS_OK) { delete q; return rc; }
    }
    *out = q;
    return BS_OK;
}

int mma_sequence_launches(const Sequence* q) { return static_cast<int>(q->steps.size()) + (q->oper ? oper_imports(q->oper) : 0); }

const OperTensor* mma_sequence_input(const Sequence* q, const uint32_t* packed) { return q->oper ? oper_input(q->oper, packed) : nullptr; }

int mma_sequence_run(Sequence* q, const OperTensor* ready, cudaStream_t st)
{
    if (q->oper) {
        const int rc = oper_begin(q->oper, ready, st);
        if (rc != BS_OK) return rc;
    }
    for (size_t i = 0; i < q->steps.size(); ++i) {
        Sequence::Step& s = q->steps[i];
        cudaStream_t on = st;
        for (int k = 0; k < 4 && s.join[k] >= 0; ++k)
            if (cudaStreamWaitEvent(st, q->steps[s.join[k]].done, 0) != cudaSuccess) { cudaGetLastError(); return BS_ERR_CUDA; }
        if (s.fork) {
            if (cudaEventRecord(s.fork, st) != cudaSuccess || cudaStreamWaitEvent(q->side, s.fork, 0) != cudaSuccess) { cudaGetLastError(); return BS_ERR_CUDA; }
            on = q->side;
        }
        const int rc = q->oper ? oper_layer(q->oper, static_cast<int>(i), on) : launch_plan(s.plan, on);
        if (rc != BS_OK) return rc;
        if (s.done && cudaEventRecord(s.done, on) != cudaSuccess) { cudaGetLastError(); return BS_ERR_CUDA; }
    }
    return BS_OK;
}

void mma_sequence_destroy(Sequence* q) { delete q; }

}  // namespace bs
