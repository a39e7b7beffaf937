// Host side of the layers on operand tensors: which sequences take them, where the tensors lie, plans and launches (kernel: oper_kernel.cuh).
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "oper_conv.h"
#include "oper_kernel.cuh"

namespace bs {

// ----------------------------------------------------------------------------- packed codes -> operand tensors

// A lane per pixel and channel word: a warp reads the words of 32 pixels (whole sectors over its channel words, which a block shares) and writes runs
// of 512 bytes.
static __global__ void __launch_bounds__(256) oper_import_kernel(const __grid_constant__ OperTensor g)
{
    const uint32_t* src = dependent_begin(g.packed);
    const int lane = threadIdx.x & 31, warps = static_cast<int>(gridDim.x) * 8, pixels = g.N * g.d_img.d, runs = (pixels + 31) / 32;
    for (long long w = blockIdx.x * 8 + (threadIdx.x >> 5); w < static_cast<long long>(runs) * g.Cw; w += warps) {
        const int run = static_cast<int>(w / g.Cw), cw = static_cast<int>(w - static_cast<long long>(run) * g.Cw), pix = run * 32 + lane;
        if (pix >= pixels) continue;
        const uint32_t* p = src + (static_cast<size_t>(pix) * g.Cw + cw) * g.bits;
        uint32_t e, d;
        if (g.bits == 2) {
            const uint2 t = *reinterpret_cast<const uint2*>(p);
            oper_pairs(t.x, t.y, e, d);
        } else {
            oper_pairs(p[0], 0u, e, d);
        }
        const int n = fdiv(pix, g.d_img), rem = pix - n * g.d_img.d, y = fdiv(rem, g.d_row), x = rem - y * g.W;
        oper_put(g.dst1, g.dst2, cw, oper_at1(g.dst1, n, y, x), oper_at2(g.dst2, n, y, x), e, d);
    }
}

// ----------------------------------------------------------------------------- packed filters -> prepared ones, of several layers in a launch

constexpr int OP_FILTERS = 16;              // layers whose filters a pass prepares, at most

struct FilterSet {
    struct Layer {
        const uint32_t* packed;             // [O][R*S][Cw][bits]
        uint4* out;                         // as bs_tc_prepare_weights lays out nibbles, [C/64][O/8][tap][2][8 filters], the mark in the last vector
        int O, RS, Cw, bits, kind, groups, vecs;        // groups of eight filters, vectors written
        long long last;
    } layer[OP_FILTERS];
};

static __global__ void __launch_bounds__(256) oper_filters_kernel(const __grid_constant__ FilterSet set)
{
    const FilterSet::Layer& f = set.layer[blockIdx.y];
    const uint32_t* packed = dependent_begin(f.packed);
    for (int idx = blockIdx.x * 256 + threadIdx.x; idx < f.vecs; idx += gridDim.x * 256) {
        const FilterVector at = filter_vector(static_cast<unsigned>(idx), f.groups, f.RS);
        const int cw = at.step * 2 + at.half;
        uint32_t v[4] = {0, 0, 0, 0};
        if (at.o < f.O && cw < f.Cw) {
            const uint32_t* p = packed + ((static_cast<size_t>(at.o) * f.RS + at.tap) * f.Cw + cw) * f.bits;
            uint32_t w[2] = {p[0], f.bits > 1 ? p[1] : 0u};
            if (f.bits == 1) expand_nibbles<1>(w, f.kind, v);
            else expand_nibbles<2>(w, f.kind, v);
        }
        put_nibbles(f.out, idx, f.vecs, f.last, make_uint4(v[0], v[1], v[2], v[3]));
    }
}

// ----------------------------------------------------------------------------- tensors of a sequence

namespace {

constexpr int OP_SMEM_MAX = 224 * 1024, OP_MAX_ROWS = 1024;         // of a CTA that has an SM to itself; half of it otherwise

int up(int v, int m) { return (v + m - 1) / m * m; }

// One form of a tensor: for readers of stride 1, or of stride 2 with a plane per parity.
struct Form {
    bool used;
    int pitch, rows;                // positions of a row, rows of an image
    long long positions;            // of a plane
    size_t offset, group, plane;    // bytes
};

struct Tensor {
    const uint32_t* ptr;
    int N, H, W, Cw, bits;
    Form form[2];
    std::vector<char> written;      // channel words that a layer has written so far
    bool import, read;
    size_t bytes() const { return static_cast<size_t>(N) * H * W * Cw * bits * 4; }
};

struct Shape { int rmin, rmax, P, Q; };        // first and last row (and column) shift of a tap in positions

Shape shape_of(const bs_conv_params& p)
{
    Shape s;
    s.rmin = p.stride == 1 ? -p.pad : -((p.pad + 1) >> 1);
    s.rmax = p.stride == 1 ? p.R - 1 - p.pad : (p.R - 1 - p.pad) >> 1;
    s.P = (p.H + 2 * p.pad - p.R) / p.stride + 1;
    s.Q = (p.W + 2 * p.pad - p.S) / p.stride + 1;
    return s;
}

struct Layout {
    std::vector<Tensor> tensors;
    std::vector<int> src, dst;      // of each layer
    std::vector<size_t> filters;    // where its filters are prepared in front of the layers, 0: they came prepared
    size_t bytes;
};

int tensor_index(Layout& l, const uint32_t* ptr, int N, int H, int W, int Cw, int bits)
{
    for (size_t i = 0; i < l.tensors.size(); ++i) {
        const Tensor& t = l.tensors[i];
        if (t.ptr == ptr) return t.N == N && t.H == H && t.W == W && t.Cw == Cw && t.bits == bits ? static_cast<int>(i) : -1;
    }
    Tensor t{};
    t.ptr = ptr; t.N = N; t.H = H; t.W = W; t.Cw = Cw; t.bits = bits;
    t.written.assign(static_cast<size_t>(Cw), 0);
    l.tensors.push_back(t);
    return static_cast<int>(l.tensors.size()) - 1;
}

// What the layers read and write, and where the operand tensors lie in the workspace.  false: a layer does not qualify, tensors overlap, or one is
// used with two shapes.
bool lay_out(const bs_sequence_layer* layers, int n, Layout& l)
{
    // Layers whose records the prepared-filter entry points refuse come with packed filters; one launch prepares them in every pass, where each such
    // layer gains a microsecond or more.
    int unprepared = 0;
    for (int i = 0; i < n; ++i) unprepared += !layers[i].wgt_tc;
    if (unprepared > n / 3 || unprepared > OP_FILTERS) return false;
    for (int i = 0; i < n; ++i) {
        const bs_conv_params& p = layers[i].p;
        if (!layers[i].out_packed || !layers[i].act_packed || p.C % 32 != 0) return false;
        if (p.a_sign != BS_UNSIGNED || p.out_sign != BS_UNSIGNED || p.out_bits > 2 || p.out_bits < 1) return false;
        if (!mma_nibbles(p.C, p.R * p.S, p.a_bits, p.w_bits, p.w_sign) || p.stride > 2 || p.R != p.S) return false;
        if (p.residual && (p.res_sign != BS_UNSIGNED || p.res_bits > 2 || !(fabsf(p.res_scale) < 3.9f) || (p.res_scale != 0.0f && fabsf(p.res_scale) <= 1e-18f))) return false;
        const Shape s = shape_of(p);
        const int src = tensor_index(l, layers[i].act_packed, p.N, p.H, p.W, p.C / 32, p.a_bits);
        const int dst = tensor_index(l, layers[i].out_packed, p.N, s.P, s.Q, ceil_div(p.out_c_total, 32), p.out_bits);
        if (src < 0 || dst < 0 || src == dst) return false;
        l.src.push_back(src);
        l.dst.push_back(dst);
        Tensor& t = l.tensors[src];
        t.read = true;
        for (char w : t.written)
            if (!w) t.import = true;           // (its contents before the first layer are what the missing words hold)
        Form& f = t.form[p.stride - 1];
        const int h = ceil_div(p.H, p.stride), w = ceil_div(p.W, p.stride);
        auto most = [](int& v, int x) { if (x > v) v = x; };
        f.used = true;
        most(f.pitch, w - s.rmin);
        most(f.pitch, s.Q + s.rmax);
        most(f.rows, h - s.rmin);
        most(f.rows, s.P + s.rmax);
        Tensor& o = l.tensors[dst];
        for (int k = 0; k < ceil_div(p.O, 32); ++k) o.written[p.out_c_offset / 32 + k] = 1;
    }
    for (const Tensor& a : l.tensors)
        for (const Tensor& b : l.tensors) {
            const char *pa = reinterpret_cast<const char*>(a.ptr), *pb = reinterpret_cast<const char*>(b.ptr);
            if (&a != &b && pa < pb + b.bytes() && pb < pa + a.bytes()) return false;
        }
    // Room in front for the taps above the first row and behind for those and the rest of the last tile; what is read there and between the
    // images is zero or belongs to no output.
    size_t off = 0;
    for (Tensor& t : l.tensors)
        for (int k = 0; k < 2; ++k) {
            Form& f = t.form[k];
            if (!f.used) continue;
            f.positions = static_cast<long long>(t.N) * f.rows * f.pitch;
            if (4 * (f.positions + 8) + 8LL * f.pitch + OP_MAX_ROWS > 0x7fffffffLL || static_cast<long long>(t.N) * t.H * t.W > 0x7fffffffLL) return false;
            const size_t edge = (static_cast<size_t>(8) * f.pitch + 8) * 16;
            f.plane = (static_cast<size_t>(f.positions) * 16 + 127) / 128 * 128;
            f.group = f.plane * (k ? 4 : 1);
            f.offset = (off + edge + 255) / 256 * 256;
            off = f.offset + f.group * static_cast<size_t>(t.Cw) + edge + static_cast<size_t>(OP_MAX_ROWS) * 16;
        }
    for (int i = 0; i < n; ++i) {
        const bs_conv_params& p = layers[i].p;
        l.filters.push_back(0);
        if (layers[i].wgt_tc) continue;
        l.filters.back() = (off + 255) / 256 * 256;
        off = l.filters.back() + bs_tc_weights_bytes(p.O, p.C, p.R, p.S);
    }
    l.bytes = off;
    return true;
}

OperDst dst_of(const Tensor& t, int k, unsigned char* ws, int word)
{
    OperDst d{};
    const Form& f = t.form[k];
    if (!f.used) return d;
    d.base = ws + f.offset + static_cast<size_t>(word) * f.group;
    d.group = static_cast<long long>(f.group);
    d.plane = static_cast<int>(f.plane / 16);
    d.pitch = f.pitch;
    d.img = f.rows * f.pitch;
    return d;
}

struct Cand { int TN, PT, units, cps, full, resident, nse, nacc; size_t smem; long long grid; double cost; };

// Shared memory of a candidate; false when it does not fit.
bool layout_cand(OperArgs& g, Cand& c, int sms)
{
    const int smem_max = c.full ? OP_SMEM_MAX : OP_SMEM_MAX / 2;
    const int rmax = g.stride == 1 ? g.R - 1 - g.pad : (g.R - 1 - g.pad) >> 1, BM = 128 * c.PT;
    g.TN = c.TN; g.PT = c.PT; g.units = c.units; g.resident = c.resident;
    g.HL = BM + (rmax - g.rmin) * g.pitch + (rmax - g.smin);
    g.NI = g.HL * g.nplanes;
    if (g.NI > 0x3FFF) return false;                       // field of the operand descriptor
    g.nchunks = ceil_div(g.nunits, c.units);
    g.tiles_m = ceil_div(g.total, BM);
    g.tiles_o = ceil_div(g.O, c.TN);
    if (g.tiles_o > sms) return false;
    const long long run = static_cast<long long>(g.NI) * 16 * g.halves;
    const long long blk = static_cast<long long>(c.TN) * g.RS * 32, filters = c.resident ? blk * g.nunits : 0;
    if (filters > smem_max || blk > smem_max || run * c.units > smem_max) return false;
    g.a_bytes = up(static_cast<int>(run) * c.units, 128);
    g.stage_bytes = g.a_bytes + (c.resident ? 0 : static_cast<int>(blk) * c.units);
    const int fixed = up(c.TN * 8 + 64, 128) + 256;
    const long long room = smem_max - fixed - filters;
    int most = static_cast<int>(room > 0 ? room / g.stage_bytes : 0);
    const int slots = sms * c.cps / g.tiles_o, waves = ceil_div(g.tiles_m, slots);
    if (most > OP_STAGES) most = OP_STAGES;
    if (most > waves * g.nchunks) most = waves * g.nchunks;        // (less shared memory for the next launch to wait for)
    if (most < 1) return false;
    c.nse = g.nse = most;
    const int cols = (c.full ? 512 : 256) - MM_SF_COLS;
    if (c.PT * c.TN > cols) return false;
    c.nacc = cols / (c.PT * c.TN);
    if (c.nacc > 4) c.nacc = 4;
    if (c.nacc > waves) c.nacc = waves;
    // (with one buffer a team of epilogue warps could take the end of its last item for that of its next: the other team's lies between)
    if (c.full && c.nacc < 2) return false;
    g.nacc = c.nacc;
    g.sf_col = c.nacc * c.PT * c.TN;
    int tc = 32;
    while (tc < g.sf_col + MM_SF_COLS) tc *= 2;
    g.tmem_cols = tc;
    g.off_stage = static_cast<int>(filters);
    g.off_tab = g.off_stage + c.nse * g.stage_bytes;
    g.off_bar = g.off_tab + up(c.TN * 8 + 64, 128);
    c.smem = static_cast<size_t>(g.off_bar) + 256;
    // the same number of waves on no more CTAs than it takes
    g.step_m = ceil_div(g.tiles_m, waves);
    c.grid = static_cast<long long>(g.step_m) * g.tiles_o;
    return true;
}

// Time model of a candidate in SM cycles: a CTA's items one after the other (ring of stages, MMAs, epilogue), and what the CTAs of an SM share.  Fitted
// to about 4000 timed plans of 135 layers (1 to 64 images, 7 to 300 pixels wide, 32 to 2048 channels, chained launches, B200 at 1.92 GHz):
// the plan with the lowest modelled time is on average 1.3 % (6 % with the constants first guessed) slower than the fastest.
struct OperFit {
    double start, full_start;       // of a launch; more where a CTA takes a whole SM and cannot begin beside the launch before
    double lat, rate, fill;         // a chunk's copies: cycles, bytes per cycle of one chunk; share of the first one that nothing hides
    double issue, m32, m64, m128;   // cycles per MMA: between two of one CTA, of the tensor core for 32, 64, 128 filters
    double chunk;                   // cycles per chunk beside its MMAs
    double e_codes, e_res, e_pair;  // two blocks of 32 x 32 outputs side by side, with a residual; factor where row tiles share the scales
    double e_once, teams;           // per item; share of an epilogue's time that two teams take
    double s_codes, s_res, l2;      // of the SM: a quarter block, with a residual; bytes per cycle
};
constexpr OperFit OPER_FIT = {1256, 1888, 278, 177, 1.42, 48.6, 42, 20.6, 26.6, 443, 920, 1548, 0.904, 1568, 0.447, 77.6, 33.1, 103.7};

double cost_of(const OperArgs& g, const Cand& c, int sms)
{
    const OperFit& k = OPER_FIT;
    const double mma = c.TN == 32 ? k.m32 : c.TN == 64 ? k.m64 : k.m128, n = static_cast<double>(c.PT) * g.RS * g.nunits;
    const double t_m = n * (mma > k.issue ? mma : k.issue) + k.chunk * g.nchunks;
    const int blocks = c.PT * (c.TN / 32), waves = ceil_div(g.tiles_m, g.step_m);
    const double pair = c.PT > 1 && blocks >= 4 ? k.e_pair : 1.0;
    const double t_e = ceil_div(blocks, 2) * (g.residual ? k.e_res : k.e_codes) * pair + k.e_once;
    const double active = static_cast<double>(ceil_div_ll(c.grid, sms));
    const double bytes = (static_cast<double>(g.NI) * 16 * g.halves + (c.resident ? 0.0 : c.TN * g.RS * 32.0)) * g.nunits;
    const double load = k.lat + bytes / g.nchunks / k.rate;
    const double ring = g.nchunks * (load + t_m / g.nchunks) / c.nse;
    const double t_mb = t_m > ring ? t_m : ring;
    auto most = [](double a, double b) { return a > b ? a : b; };
    const double shared_m = most(active * n * mma, active * bytes / k.l2), shared_e = active * blocks * 4.0 * (g.residual ? k.s_res : k.s_codes) * pair;
    const double e_rate = c.full ? t_e * k.teams : t_e;
    const double step = most(most(c.nacc > 1 ? most(t_mb, e_rate) : t_mb + t_e, shared_m), shared_e);
    return k.start + (c.full ? k.full_start : 0.0) + load * k.fill + most(t_mb, shared_m) + most(t_e, shared_e) + (waves - 1) * step;
}

}  // namespace

struct OperSequence {
    struct Step { OperArgs g; unsigned grid; int smem, full; };
    struct Import { OperTensor g; unsigned grid; };
    std::vector<Step> steps;
    std::vector<Import> imports;
    FilterSet filters;
    int nfilters, filter_blocks;
};

// Arguments of layer i but its tiling.
static bool fill(OperArgs& g, const bs_sequence_layer& l, const Layout& lay, int i, unsigned char* ws)
{
    const bs_conv_params& p = l.p;
    const Shape s = shape_of(p);
    const Tensor &in = lay.tensors[lay.src[i]], &out = lay.tensors[lay.dst[i]];
    const Form& f = in.form[p.stride - 1];
    g.N = p.N; g.O = p.O; g.R = p.R; g.RS = p.R * p.S; g.P = s.P; g.Q = s.Q; g.stride = p.stride; g.pad = p.pad; g.Cw = p.C / 32;
    g.opad = up(p.O, 128);
    g.rmin = g.smin = s.rmin;
    g.pitch = f.pitch;
    g.total = static_cast<int>(f.positions);
    g.nplanes = p.stride == 2 && p.R > 1 ? 4 : 1;
    g.d_img = make_div(f.rows * f.pitch);
    g.d_pitch = make_div(f.pitch);
    g.nunits = (g.Cw + 1) / 2;
    g.halves = g.Cw == 1 ? 1 : 2;
    g.src = ws + f.offset + (static_cast<long long>(s.rmin) * f.pitch + s.rmin) * 16;
    g.src_group = static_cast<long long>(f.group);
    g.src_plane = static_cast<long long>(f.plane);
    g.wgt = l.wgt_tc ? l.wgt_tc : reinterpret_cast<int8_t*>(ws + lay.filters[i]);
    g.out_packed = l.out_packed;
    const int word = p.out_c_offset / 32;
    g.dst1 = dst_of(out, 0, ws, word);
    g.dst2 = dst_of(out, 1, ws, word);
    if ((out.form[0].used || out.form[1].used) && p.O % 32 != 0) return false;
    g.scale = p.scale; g.bias = p.bias; g.residual = p.residual; g.res_scale = p.res_scale;
    g.acc_bound = static_cast<float>(static_cast<double>(p.C) * g.RS * ((1 << p.a_bits) - 1) * (p.w_sign == BS_BIPOLAR ? 1 : p.w_sign == BS_UNSIGNED ? (1 << p.w_bits) - 1 : 1 << (p.w_bits - 1)));
    g.relu = p.relu; g.out_bits = p.out_bits; g.out_sign = p.out_sign;
    g.out_cw_off = word; g.out_cw_total = out.Cw;
    g.res_bits = p.res_bits; g.res_sign = p.res_sign; g.res_c_off = p.res_c_offset;
    g.res_cw_total = ceil_div(p.res_c_total > 0 ? p.res_c_total : 1, 32);
    g.early_b = l.chained && !l.aside && l.wgt_tc;
    g.status = status_device_ptr();
    return true;
}

static bool plan_layer(OperSequence::Step& s, int sms)
{
    Cand best{};
    best.cost = 1e30;
    bool found = false;
#ifdef BS_TUNING
    int ov[6] = {0, 0, 0, 0, -1, 0};        // TN, PT, units, CTAs per SM, resident
    if (const char* e = s.g.O > 32 || s.g.R > 1 || getenv("BS_OP_ALL") ? getenv("BS_OP") : nullptr) sscanf(e, "%d,%d,%d,%d,%d", ov, ov + 1, ov + 2, ov + 3, ov + 4);
#endif
    for (int TN = 32; TN <= 128; TN *= 2) {
        if (TN > 32 && TN / 2 >= up(s.g.O, 32)) continue;
        for (int PT = 1; PT <= 4; PT *= 2)
            for (int units = 1; units <= 4; units *= 2) {
                if (units > 1 && (units > s.g.nunits || s.g.R > 1)) continue;
                for (int v = 0; v < 6; ++v) {
                    Cand c{};
                    c.TN = TN; c.PT = PT; c.units = units; c.resident = v & 1; c.full = v >> 1 == 2; c.cps = c.full ? 1 : 1 + (v >> 1);
#ifdef BS_TUNING
                    if ((ov[0] && TN != ov[0]) || (ov[1] && PT != ov[1]) || (ov[2] && units != ov[2]) || (ov[3] && c.cps + 2 * c.full != ov[3]) || (ov[4] >= 0 && c.resident != ov[4])) continue;
#endif
                    OperArgs t = s.g;
                    if (!layout_cand(t, c, sms)) continue;
                    c.cost = cost_of(t, c, sms);
                    if (c.cost < best.cost) { best = c; found = true; }
                }
            }
    }
    if (!found || !layout_cand(s.g, best, sms)) return false;
#ifdef BS_TUNING
    if (getenv("BS_OP_VERBOSE"))
        fprintf(stderr, "oper plan: N%d C%d %dx%d O%d k%d s%d res%d -> TN %d PT %d units %d cps %d full %d resident %d stages %d nacc %d HL %d tiles %d x %d grid %lld smem %zu cost %.0f\n", s.g.N, s.g.Cw * 32,
                s.g.P, s.g.Q, s.g.O, s.g.R, s.g.stride, s.g.residual ? 1 : 0, best.TN, best.PT, best.units, best.cps, best.full, best.resident, best.nse, best.nacc, s.g.HL, s.g.tiles_m, s.g.tiles_o, best.grid, best.smem, best.cost);
#endif
    // float += e2m1 x e2m1 with ue8m0 scale factors; TN columns, 128 rows
    s.g.idesc = (1u << 7) | (1u << 10) | (1u << 23) | (static_cast<unsigned>(s.g.TN >> 3) << 17) | (static_cast<unsigned>(128 >> 4) << 24);
    s.grid = static_cast<unsigned>(best.grid);
    s.smem = static_cast<int>(best.smem);
    s.full = best.full;
    return true;
}

static bool build(const bs_sequence_layer* layers, int n, unsigned char* ws, OperSequence& q, size_t& bytes)
{
    Layout lay{};
    if (!lay_out(layers, n, lay)) return false;
    int sms = device_sm_count();
    if (sms <= 0) sms = 148;
    q.steps.resize(static_cast<size_t>(n));
    q.nfilters = q.filter_blocks = 0;
    for (int i = 0; i < n; ++i) {
        memset(static_cast<void*>(&q.steps[i]), 0, sizeof q.steps[i]);
        if (!fill(q.steps[i].g, layers[i], lay, i, ws) || !plan_layer(q.steps[i], sms)) return false;
        const bs_conv_params& p = layers[i].p;
        if (!layers[i].wgt_tc) {
            FilterSet::Layer& f = q.filters.layer[q.nfilters++];
            const int groups = up(p.O, 128) / 8, RS = p.R * p.S, Cw = p.C / 32;
            const long long vecs = static_cast<long long>((Cw + 1) / 2) * groups * RS * 16;
            if (vecs > 0x7fffff00LL) return false;
            f = {layers[i].wgt_packed, reinterpret_cast<uint4*>(ws + lay.filters[i]), p.O, RS, Cw, p.w_bits, p.w_sign == BS_SIGNED ? 1 : p.w_sign == BS_BIPOLAR ? 2 : 0, groups,
                 static_cast<int>(vecs), static_cast<long long>(Cw) * groups * RS * 16 - 1};
            const int blocks = static_cast<int>((vecs + 255) / 256);
            if (blocks > q.filter_blocks) q.filter_blocks = blocks < 4 * sms ? blocks : 4 * sms;
        }
    }
    for (const Tensor& t : lay.tensors) {
        if (!t.read || !t.import) continue;
        OperSequence::Import m{};
        m.g.packed = t.ptr;
        m.g.dst1 = dst_of(t, 0, ws, 0);
        m.g.dst2 = dst_of(t, 1, ws, 0);
        m.g.N = t.N; m.g.H = t.H; m.g.W = t.W; m.g.Cw = t.Cw; m.g.bits = t.bits;
        m.g.d_img = make_div(t.H * t.W);
        m.g.d_row = make_div(t.W);
        const long long blocks = (ceil_div_ll(static_cast<long long>(t.N) * t.H * t.W, 32) * t.Cw + 7) / 8;
        m.grid = static_cast<unsigned>(blocks < 8LL * sms ? blocks : 8LL * sms);
        q.imports.push_back(m);
    }
    bytes = lay.bytes;
    return true;
}

size_t oper_workspace_bytes(const bs_sequence_layer* layers, int n)
{
    OperSequence q;
    size_t bytes = 0;
    return build(layers, n, nullptr, q, bytes) ? bytes : 0;
}

int oper_layer_plan(const bs_sequence_layer* layers, int n, int i, bs_layer_plan* out)
{
    OperSequence q;
    size_t bytes = 0;
    if (!build(layers, n, nullptr, q, bytes)) return BS_ERR_UNSUPPORTED;
    const OperSequence::Step& s = q.steps[static_cast<size_t>(i)];
    *out = {s.g.TN, s.g.PT, s.g.units, s.g.resident, s.g.nse, s.g.nacc, s.full ? 2 : 1, static_cast<int>(s.grid), ceil_div(s.g.tiles_m, s.g.step_m)};
    return BS_OK;
}

OperSequence* oper_create(const bs_sequence_layer* layers, int n, void* workspace, size_t bytes)
{
    OperSequence* q = new (std::nothrow) OperSequence;
    size_t need = 0;
    if (q && workspace && build(layers, n, static_cast<unsigned char*>(workspace), *q, need) && need <= bytes && status_device_ptr() &&
        cudaFuncSetAttribute(bitserial_oper_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, OP_SMEM_MAX / 2) == cudaSuccess &&
        cudaFuncSetAttribute(bitserial_oper_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, OP_SMEM_MAX) == cudaSuccess)
        return q;
    cudaGetLastError();
    delete q;
    return nullptr;
}

int oper_imports(const OperSequence* q) { return static_cast<int>(q->imports.size()) + (q->nfilters > 0); }

const OperTensor* oper_input(const OperSequence* q, const uint32_t* packed)
{
    for (const OperSequence::Import& m : q->imports)
        if (m.g.packed == packed) return &m.g;
    return nullptr;
}

int oper_begin(const OperSequence* q, const OperTensor* ready, cudaStream_t st)
{
    if (q->nfilters > 0) {
        const int rc = launch_dependent(oper_filters_kernel, dim3(static_cast<unsigned>(q->filter_blocks), static_cast<unsigned>(q->nfilters)), dim3(256), 0, st, q->filters);
        if (rc != BS_OK) return rc;
    }
    for (const OperSequence::Import& m : q->imports) {
        if (&m.g == ready) continue;
        const int rc = launch_dependent(oper_import_kernel, dim3(m.grid), dim3(256), 0, st, m.g);
        if (rc != BS_OK) return rc;
    }
    return BS_OK;
}

int oper_layer(const OperSequence* q, int i, cudaStream_t st)
{
    const OperSequence::Step& s = q->steps[static_cast<size_t>(i)];
    return launch_dependent(s.full ? bitserial_oper_kernel<true> : bitserial_oper_kernel<false>, dim3(s.grid), dim3(oper_threads(s.full)), static_cast<size_t>(s.smem), st, s.g);
}

void oper_destroy(OperSequence* q) { delete q; }

}  // namespace bs

#ifdef BS_TRACE
// Trace builds: as bs_tc_trace_read, of the layers on operand tensors.
extern "C" int bs_oper_trace_read(long long* out, int clear)
{
    if (cudaDeviceSynchronize() != cudaSuccess) return BS_ERR_CUDA;
    if (cudaMemcpyFromSymbol(out, bs::g_mm_trace, sizeof(bs::g_mm_trace)) != cudaSuccess) return BS_ERR_CUDA;
    if (clear) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, bs::g_mm_trace) != cudaSuccess || cudaMemset(p, 0, sizeof(bs::g_mm_trace)) != cudaSuccess) return BS_ERR_CUDA;
    }
    return BS_OK;
}
#endif
