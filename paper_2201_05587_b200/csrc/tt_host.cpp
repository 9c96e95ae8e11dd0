// Host logic of libtt: workloads, kernel classes, schedule records, the transfer /
// legalisation / validity layer, the selector.  Nothing here touches the device.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>
#include <new>
#include "tt_internal.h"

using namespace tt;

namespace {

uint64_t fnv1a(const void* data, size_t n, uint64_t h = 1469598103934665603ull) {
    const unsigned char* p = static_cast<const unsigned char*>(data);
    for (size_t i = 0; i < n; ++i) { h ^= p[i]; h *= 1099511628211ull; }
    return h;
}

int round_up(int v, int m) { return (v + m - 1) / m * m; }
long long round_up64(long long v, long long m) { return (v + m - 1) / m * m; }
int pow2_ceil(int v) { int p = 1; while (p < v) p <<= 1; return p; }
int pow2_floor(int v) { int p = 1; while (p * 2 <= v) p <<= 1; return p; }

int family_of(tt_op op) {
    switch (op) {
        case TT_OP_CONV2D: case TT_OP_DENSE: case TT_OP_BATCH_MATMUL: return TT_FAMILY_GEMM_TC;
        case TT_OP_DWCONV2D: return TT_FAMILY_DW_SIMT;
        case TT_OP_SOFTMAX: return TT_FAMILY_ROW_SIMT;
    }
    return -1;
}

bool conv_like(tt_op op) { return op == TT_OP_CONV2D || op == TT_OP_DWCONV2D; }

}  // namespace

namespace tt {

uint64_t class_hash(int op, const tt_shapes& s) {
    // A kernel class is the sequence of operators, regardless of data sizes (Section 4.2).
    int32_t v[5] = {op, s.has_bias != 0, s.act, s.has_residual != 0, op == TT_OP_BATCH_MATMUL ? (s.trans_b != 0) : 0};
    return fnv1a(v, sizeof v);
}

size_t tensor_elems(const tt_workload* w, int which) {
    const tt_shapes& s = w->sh;
    switch (w->op) {
        case TT_OP_CONV2D:
            switch (which) {
                case 0: return (size_t)s.n * s.c * s.h * s.w;
                case 1: return (size_t)s.k * s.c * s.r * s.s;
                case 2: return s.has_bias ? (size_t)s.k : 0;
                case 3: return s.has_residual ? (size_t)s.n * s.k * w->P * w->Q : 0;
                default: return (size_t)s.n * s.k * w->P * w->Q;
            }
        case TT_OP_DWCONV2D:
            switch (which) {
                case 0: return (size_t)s.n * s.c * s.h * s.w;
                case 1: return (size_t)s.c * s.r * s.s;
                case 2: return s.has_bias ? (size_t)s.c : 0;
                case 3: return 0;
                default: return (size_t)s.n * s.c * w->P * w->Q;
            }
        case TT_OP_DENSE:
        case TT_OP_BATCH_MATMUL:
            switch (which) {
                case 0: return (size_t)s.batch * s.m * s.kk;
                case 1: return (size_t)s.batch * s.nn * s.kk;
                case 2: return s.has_bias ? (size_t)s.nn : 0;
                case 3: return s.has_residual ? (size_t)s.batch * s.m * s.nn : 0;
                default: return (size_t)s.batch * s.m * s.nn;
            }
        case TT_OP_SOFTMAX:
            return (which == 0 || which == 4) ? (size_t)s.batch * s.m * s.nn : 0;
    }
    return 0;
}

// ---- legalisation -------------------------------------------------------------------------------------------

// conv2d with k_order = 1: the reduction walks blocks of 32 channels and, inside a block, tap by tap (tt_conv.cu).  Filters
// are re-packed into that order by a kernel of its own, once per weight pointer, which single images of other layouts
// would not earn back: the order exists for stride-1 convolutions with 16-byte image rows and, for any stride and row length,
// from two images on.
static bool tap_major_possible(const tt_workload* w) {
    const tt_shapes& s = w->sh;
    return w->op == TT_OP_CONV2D && s.r * s.s <= 64 && (long long)w->P * w->Q > 1 && s.stride_h * s.stride_w <= kPmMaxPlanes &&
           s.r < 100 && s.s < 100 && s.pad_h < 100 && s.pad_w < 100 && ((s.stride_h == 1 && s.stride_w == 1 && (s.w % 4) == 0) || s.n >= 2);
}

namespace {
int floor_div(int a, int b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }
// One axis of the padded-linear numbering: per parity class the first tap, its shift, the number of taps; the positions that a
// row (or an image) takes so that taps which reach past its end find zeros.
struct TapAxis { int first[16], shift[16], count[16], lo, hi, pitch; };
TapAxis tap_axis(int taps, int stride, int pad, int extent, int outputs) {
    TapAxis t{};
    t.lo = floor_div(-pad, stride); t.hi = floor_div(taps - 1 - pad, stride);
    for (int a = 0; a < stride; ++a)
        for (int r = 0; r < taps; ++r) {
            if (r - pad - stride * floor_div(r - pad, stride) != a) continue;
            if (t.count[a]++ == 0) { t.first[a] = r; t.shift[a] = floor_div(r - pad, stride); }
        }
    const int data = (extent + stride - 1) / stride;
    t.pitch = std::max(data + std::max(0, -t.lo), outputs + std::max(0, t.hi));
    return t;
}
unsigned magic_of(int d) { return d == 1 ? 0xffffffffu : (unsigned)(0x100000000ull / (unsigned)d); }
}  // namespace

static tt_status legalise_conv_tapmajor(const tt_workload* w, const tt_schedule_record* rec, int mode, Plan* plan) {
    tt_apply_info& I = plan->info;
    const tt_shapes& s = w->sh;
    const bool strict = mode == TT_MODE_STRICT;
    tt_schedule_record L = *rec;
    int changed = 0;
    const int RS = s.r * s.s, CB = (s.c + 31) / 32;
    const TapAxis ty = tap_axis(s.r, s.stride_h, s.pad_h, s.h, w->P), tx = tap_axis(s.s, s.stride_w, s.pad_w, s.w, w->Q);
    const long long image = (long long)ty.pitch * tx.pitch;
    const int M = s.k;
    // padded-linear positions up to the last output
    const long long Nl = (s.n - 1) * image + (long long)(w->P - 1) * tx.pitch + w->Q, Kl = (long long)CB * RS * 32;
    if (Nl > 0x3fffffffLL || Kl > 0x3fffffffLL) return TT_ERR_RESOURCE;
    const int N = (int)Nl, K = (int)Kl;
    // fixed by the mode: filters on the 128 rows, no split-K, one accumulator per tile; a reduction tile is `tps` taps of one
    // 32-channel block (tile_k = 32 * tps, tps a divisor of the tap count, tile_k <= 128)
    int tps = 1;
    for (int d = 1; d <= 4; ++d) if (RS % d == 0 && 32 * d <= rec->tile_k) tps = d;
    const int tk = 32 * tps;
    if (strict && (rec->mma_m_axis == 2 || rec->tile_k != tk || rec->split_k != 1)) return TT_ERR_INVALID_SCHEDULE;
    L.mma_m_axis = 1; L.tile_m = kHwTileM; L.tile_k = tk; L.split_k = 1; L.acc_split = 1; L.slab_tiles = 0; L.k_order = 1;
    // (one kernel serves both forms: its CTAs always walk)
    const bool persistent = rec->persistent == 1;
    L.persistent = 1; L.ctas_per_sm = 1;
    if (rec->ctas_per_sm == 2) { if (strict) return TT_ERR_INVALID_SCHEDULE; changed |= TT_CHG_FORM; }
    L.precision = 0;                                      // (no error-compensated products for convolutions)
    if (rec->precision != 0) { if (strict) return TT_ERR_INVALID_SCHEDULE; changed |= TT_CHG_FORM; }
    if (rec->tile_m != kHwTileM) changed |= TT_CHG_TILE_M;
    if (rec->split_k != 1) changed |= TT_CHG_SPLIT_K;
    int tn = std::min(256, std::max(16, round_up(rec->tile_n, 16)));
    tn = std::min(tn, round_up(N, 16));
    const int k_tiles = CB * RS / tps;
    // (the walking kernel's filter pipeline runs on across tiles: no point in clamping it to one tile's reduction)
    const int st = persistent ? std::min(kMaxStages, rec->stages) : std::min(std::min(kMaxStages, rec->stages), k_tiles);
    if (strict && (tn != rec->tile_n || st != rec->stages || (changed & ~TT_CHG_TILE_M))) return TT_ERR_INVALID_SCHEDULE;
    const int tiles_m = (M + kHwTileM - 1) / kHwTileM;
    // How the tiles are laid over the SMs is this rule's choice unless the record is to
    // run as written (strict mode); the legal record says what it chose (tile_n, cta_group).
    // Where the record's tiles fill more than half of the SMs, columns are dealt evenly over the rounds that its tile needs: 121
    // tiles of 224 columns become 141 of 192; a tile with which they take fewer rounds replaces it where that is a tenth cheaper.
    // Where they fill less, CTAs share a tile's channel blocks as a cluster: as many as save the most cycles, as long as all
    // clusters are resident at once (20 clusters of 7 are not: 320 -> 200 at 9 x 9, batch 6, 64 columns: 17.0 us, in clusters of 5
    // 9.3); the widest tile replaces the record's where that is cheaper.
    // Cycles: a tap takes what its columns take the tensor core, 2 each, or what shared memory has to move in 128-byte lines, its
    // filters in and out, 256, its columns, about 32 for the slab; the read-out 30 a column; the exchange in a cluster 750 and 25 for every
    // column that a CTA leaves to others.  Least squares over 27 layers under 15 widths and 8 clusters each give 29, 753 and 22 (and the
    // taps' cycles a factor of 1.01).  3x3 64 -> 64 at 56 x 56, batch 4, 192 columns: 11.3 us alone, 10.1 in pairs; 1x1 64 -> 128 at
    // 14 x 14, batch 8, 96 columns: 5.1 and 5.5; 1x1 512 -> 64 there, 256 columns: 29.9 and 11.6 in eights; 3x3 512 -> 512 at 7 x 7,
    // batch 32: 22.7 with 128 columns in pairs, 22.2 with 256 in fours.
    // Those layers under 7 records each: 1.81 times faster than as written without clusters in the geometric mean, 1.18 times the best of
    // all widths and clusters; one pair slower than as written (by 4 %).
    const auto tiles_of = [&](int n) { return (long long)tiles_m * ((N + n - 1) / n); };
    struct Share { long long cycles; int ctas; };
    const auto share_of = [&](int n) {
        const long long tap = std::max(2 * n, n + 288);
        Share best{CB * RS * tap + 30 * n, 1};
        for (int k = 2; k <= std::min(8, CB); ++k) {
            if (tiles_of(n) > kResidentClusters[k]) continue;
            const long long cycles = (CB + k - 1) / k * RS * tap + 30 * n + 750 + 25 * n * (k - 1) / k;
            if (cycles < best.cycles) best = Share{cycles, k};
        }
        return best;
    };
    const auto cost_of = [&](int n) { return (tiles_of(n) + kSms - 1) / kSms * share_of(n).cycles; };
    const auto dealt = [&](long long rounds) {           // the columns of a tile when all of them take `rounds` rounds
        const long long columns = rounds * kSms / tiles_m;
        return columns >= 1 ? std::max<long long>(16, round_up64((N + columns - 1) / columns, 16)) : 0x7fffffffLL;
    };
    int split = std::max(1, rec->cta_group);
    if (strict) {
        // (the CTAs of a cluster take one tile: all tiles have to be resident at once)
        if (split > std::min(8, CB) || (split > 1 && tiles_of(tn) * split > kSms)) return TT_ERR_INVALID_SCHEDULE;
    } else {
        if (tiles_of(tn) * 2 > kSms) {
            const long long rounds = (tiles_of(tn) + kSms - 1) / kSms;
            tn = (int)std::min<long long>(tn, dealt(rounds));
            for (long long r = 1; r < rounds && r <= 4; ++r) {
                if (dealt(r) > 256) continue;
                if (cost_of((int)dealt(r)) * 10 < cost_of(tn) * 9) tn = (int)dealt(r);
                break;
            }
        }
        const int widest = std::min(256, round_up(N, 16));
        if (tiles_of(tn) * 2 <= kSms && cost_of(widest) < cost_of(tn)) tn = widest;
        split = tiles_of(tn) * 2 > kSms ? 1 : share_of(tn).ctas;
    }
    L.tile_n = tn; L.cta_group = split;
    if (tn != rec->tile_n) changed |= TT_CHG_TILE_N;
    if (split != std::max(1, rec->cta_group)) changed |= TT_CHG_CLUSTER;
    const int tiles_n = (N + tn - 1) / tn;
    const long long tiles = (long long)tiles_m * tiles_n;
    if (tiles > 0x7fffffffLL) return TT_ERR_RESOURCE;
    // shared memory: filter stages | one or two slabs | staging blocks of the read-out (twelve warps' where all tiles are
    // resident, over the idle pipeline).  A barrier is passed for up to three taps, whose issue then
    // hides its latency; the record's stages times its taps per reduction tile say how many taps' filters are in flight.  Records
    // that ask for the same run the same, so the legal one names them in one way: reduction tiles of one tap.
    const int shift_min = ty.lo * tx.pitch + tx.lo, shift_max = std::max(0, ty.hi) * tx.pitch + std::max(0, tx.hi);
    const int lines = tn + shift_max - std::min(shift_min, 0);
    const long long slab = (long long)lines * 128;
    const long long epi = 4ll * kPmEpiBlockBytes;
    const long long tail = 12ll * kPmEpiBlockBytes;
    const int plane_taps = *std::max_element(ty.count, ty.count + 16) * *std::max_element(tx.count, tx.count + 16);   // of the largest parity class
    const int want = std::min(kMaxStages, st * tps);
    int q = plane_taps == 4 ? 2 : std::min(3, plane_taps), depth = std::max(2, (want + q - 1) / q);
    int bufs = (CB > 1 || plane_taps < RS || tiles > kSms) ? 2 : 1;
    auto total = [&] { return std::max(round_up64((long long)depth * q * kPmTapBytes + bufs * slab, 1024) + epi, round_up64(tail, 1024)) + 1024; };
    while (total() > kDynSmemLimit) {
        if (depth > 2) --depth;
        else if (q > 1) --q;
        else if (bufs > 1) --bufs;
        else if (depth > 1) --depth;
        else break;
    }
    if (strict) {
        if (depth * q < want) return TT_ERR_RESOURCE;
    } else {
        L.tile_k = 32; L.stages = std::min(kMaxStages, depth * q);
        if (rec->tile_k != L.tile_k) changed |= TT_CHG_TILE_K;
        if (rec->stages != L.stages) changed |= TT_CHG_STAGES;
    }
    const long long smem = total();
    const int tmem_cols = std::max(32, pow2_ceil(tiles > kSms ? tn + round_up(tn, 32) : round_up(tn, 32)));
    I = tt_apply_info{};
    I.legal = L; I.changed = changed;
    I.grid_x = (int)std::min<long long>(tiles, kSms / split); I.grid_y = split; I.grid_z = 1;
    I.threads = 448;
    I.smem_bytes = (int)std::min<long long>(std::max<long long>(smem, 116 * 1024), 0x7fffffff);     // one CTA per SM
    I.tmem_cols = tmem_cols;
    I.workspace_bytes = (int64_t)M * K * 4;              // the re-packed filters
    I.exchange_kib = (int32_t)(split > 1 ? tiles * split * ((tn + 31) / 32) * 16 : 0);   // 4 KiB per CTA, 32 columns and lane quadrant
    I.launches = 2;
    if (smem > kDynSmemLimit) return TT_ERR_RESOURCE;
    plan->swap_ab = false;
    plan->gm = M; plan->gn = N; plan->gk = K; plan->gbatch = 1;
    plan->partial_bytes = 0;
    plan->repack = true;
    plan->a_tensor = 1; plan->b_tensor = 0;
    plan->g = GemmArgs{};
    GemmArgs& g = plan->g;                               // what the filters' tensor map is made from
    g.M = M; g.N = N; g.K = K; g.batch = 1; g.atom_k = 32; g.a_mode = OPM_TMA; g.b_mode = -1; g.a_rs = K; g.a_ks = 1;
    ConvPmArgs& c = plan->pm;
    c = ConvPmArgs{};
    c.M = M; c.C = s.c; c.H = s.h; c.W = s.w; c.R = s.r; c.S = s.s; c.P = w->P; c.Q = w->Q; c.images = s.n;
    c.sh = s.stride_h; c.sw = s.stride_w; c.act = s.act;
    c.blocks = CB;
    c.wp = tx.pitch; c.image_pitch = (int)image;
    c.magic_wp = magic_of(c.wp); c.magic_image = magic_of(c.image_pitch);
    c.shift_min = std::min(shift_min, 0); c.slab_lines = lines;
    for (int a = 0; a < s.stride_h; ++a) for (int b = 0; b < s.stride_w; ++b)
        if (ty.count[a] > 0 && tx.count[b] > 0)
            c.planes[c.n_planes++] = ConvPlane{(signed char)a, (signed char)b, (signed char)ty.shift[a], (signed char)tx.shift[b],
                                               (unsigned char)ty.count[a], (unsigned char)tx.count[b], (unsigned char)ty.first[a], (unsigned char)tx.first[b]};
    c.tile_n = tn; c.tiles_m = tiles_m; c.tiles_n = tiles_n; c.total_tiles = (int)tiles; c.raster = L.raster; c.split = split;
    c.stages = depth; c.taps_per_stage = q; c.slab_bufs = bufs;
    c.slab_off = (unsigned)(depth * q * kPmTapBytes); c.slab_bytes = (unsigned)slab;
    c.epi_off = (unsigned)round_up64((long long)depth * q * kPmTapBytes + bufs * slab, 1024);
    c.idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((unsigned)(tn >> 3) << 17) | ((unsigned)(kHwTileM >> 4) << 24);
    c.tmem_cols = (unsigned)tmem_cols;
    return TT_OK;
}

// What a plan may do beside what its record says, as long as there is room for it.
struct PlanOptions {
    bool boxes;                                          // ragged rows come by TMA, in boxes of groups of four
    bool fewer_splits;                                   // splits that are not resident at once are fewer
};

static tt_status plan_gemm(const tt_workload* w, const tt_schedule_record* rec, int mode, PlanOptions may, Plan* plan) {
    // nonsense is refused whatever the kernel and the reduction order
    if (rec->tile_m <= 0 || rec->tile_n <= 0 || rec->tile_k <= 0 || rec->stages <= 0 || rec->split_k <= 0 ||
        rec->raster < 0 || rec->raster > 1 || rec->mma_m_axis < 0 || rec->mma_m_axis > 2 || rec->persistent < 0 ||
        rec->persistent > 1 || rec->cta_group < 0 || rec->cta_group > (rec->k_order == 1 ? 8 : 2) || rec->ctas_per_sm < 0 || rec->ctas_per_sm > 2 ||
        rec->acc_split < 0 || rec->k_order < 0 || rec->k_order > 1 || rec->warp_layout != 0 || rec->precision < 0 || rec->precision > 1 ||
        (w->op == TT_OP_CONV2D && rec->slab_tiles < 0))
        return TT_ERR_INVALID_SCHEDULE;
    if (rec->k_order == 1) {
        if (tap_major_possible(w)) {
            // (rows so wide that the taps' slab of positions exceeds shared memory are walked in the stored order)
            const tt_status st = legalise_conv_tapmajor(w, rec, mode, plan);
            if (st != TT_ERR_RESOURCE || mode == TT_MODE_STRICT) return st;
        }
        if (mode == TT_MODE_STRICT) return TT_ERR_INVALID_SCHEDULE;       // no such reduction order on this kernel
    }
    tt_apply_info& I = plan->info;
    tt_schedule_record L = *rec;
    int changed = 0;
    const bool strict = mode == TT_MODE_STRICT;
    // Which output axis becomes the accumulator's 128 rows.  Left to the library (0), the shorter-than-a-tile
    // axis goes to the MMA's N side, where 16..256 columns are legal.
    tt_shapes s = w->sh;                                  // a copy: a pointwise convolution is re-viewed below
    int P = w->P, Q = w->Q;
    bool swap = rec->mma_m_axis == 2;
    if (rec->mma_m_axis == 0) swap = w->view.gm <= 64 && w->view.gn > w->view.gm;
    L.mma_m_axis = swap ? 2 : 1;
    L.k_order = 0;
    if (rec->k_order != 0) changed |= TT_CHG_KORDER;    // reformulated: the stored channel-major order
    plan->repack = false;
    plan->swap_ab = swap;
    plan->gm = swap ? w->view.gn : w->view.gm;
    plan->gn = swap ? w->view.gm : w->view.gn;
    const int M = plan->gm, N = plan->gn, K = plan->gk, B = plan->gbatch;
    // A split factor larger than the loop itself is invalid code when nothing may be reformulated (Section 4.2).
    if (strict && (rec->tile_m > round_up(M, 32) || rec->tile_n > round_up(N, 16) || rec->tile_k > round_up(K, 8)))
        return TT_ERR_INVALID_SCHEDULE;
    // tile_m: the accumulator always spans 128 tensor-memory lanes; smaller logical tiles leave rows idle.
    L.tile_m = kHwTileM;
    if (L.tile_m != rec->tile_m) changed |= TT_CHG_TILE_M;
    // tile_n: legal MMA N for M = 128 is a multiple of 16 in [16, 256]; no wider than the padded extent.
    int tn = std::min(256, std::max(16, round_up(rec->tile_n, 16)));
    tn = std::min(tn, round_up(N, 16));
    if (tn != rec->tile_n) changed |= TT_CHG_TILE_N;
    L.tile_n = tn;
    // tile_k: power of two in [8, 128] (one to four 128-byte swizzle atoms, or one 32/64-byte atom).
    int tk = std::min(128, std::max(8, pow2_floor(rec->tile_k)));
    tk = std::min(tk, std::max(8, pow2_ceil(K)));
    if (tk != rec->tile_k) changed |= TT_CHG_TILE_K;
    L.tile_k = tk;
    int st = std::min(kMaxStages, rec->stages);
    if (st != rec->stages) changed |= TT_CHG_STAGES;
    L.stages = st;
    const int k_tiles = (K + tk - 1) / tk;
    // The persistent form: both operands must be reachable by TMA -- K-major with 16-byte rows, or row-contiguous (the
    // image of a pointwise convolution, the second operand of an NN batch_matmul) with 16-byte row pitch.
    // Error-compensated products need both operands as K-major TMA tiles (their remainders are worked out in place, tile by
    // tile) and exist in the one-tile form only: dense and batch_matmul NT with 16-byte rows.
    bool x3 = rec->precision == 1;
    if (x3 && !((w->op == TT_OP_DENSE || (w->op == TT_OP_BATCH_MATMUL && w->sh.trans_b)) && (K % 4) == 0)) {
        if (strict) return TT_ERR_INVALID_SCHEDULE;
        x3 = false; changed |= TT_CHG_FORM;
    }
    L.precision = x3 ? 1 : 0;
    bool persistent = rec->persistent == 1;
    if (persistent && x3) { if (strict) return TT_ERR_INVALID_SCHEDULE; persistent = false; changed |= TT_CHG_FORM; }
    {
        const tt_shapes& o = w->sh;
        bool can = (K % 4) == 0;
        if (w->op == TT_OP_CONV2D)
            can = can && o.r == 1 && o.s == 1 && o.stride_h == 1 && o.stride_w == 1 && o.pad_h == 0 && o.pad_w == 0 &&
                  ((long long)o.h * o.w) % 4 == 0;
        else if (w->op == TT_OP_BATCH_MATMUL && !o.trans_b)
            can = can && (o.nn % 4) == 0;
        if (persistent && !can) { if (strict) return TT_ERR_INVALID_SCHEDULE; persistent = false; changed |= TT_CHG_FORM; }
    }
    // An operand whose row index is the contiguous one, in 16-byte steps: TMA boxes that the tensor core reads MN-major.
    const bool mn_operand = w->op == TT_OP_CONV2D
        ? w->sh.r == 1 && w->sh.s == 1 && w->sh.stride_h == 1 && w->sh.stride_w == 1 && w->sh.pad_h == 0 && w->sh.pad_w == 0 && ((long long)w->sh.h * w->sh.w) % 4 == 0
        : w->op == TT_OP_BATCH_MATMUL && !w->sh.trans_b && w->sh.nn % 4 == 0;
    int cg = rec->cta_group == 2 ? 2 : 1;
    if (cg == 2 && (!persistent || mn_operand || tn < 32)) { if (strict) return TT_ERR_INVALID_SCHEDULE; cg = 1; changed |= TT_CHG_FORM; }
    if (rec->cta_group > 2) changed |= TT_CHG_FORM;       // (a cluster of the tap-major order, which is not this kernel's)
    L.persistent = persistent ? 1 : 0;
    L.cta_group = cg;
    if (persistent && !strict) {
        // Columns are dealt evenly over the rounds of the SMs that the record's tile needs, as long as those are few: 152 tiles of 256
        // columns are one full round and four tiles more, 240 of 160 are two rounds of little more than half the work (2419 x 1976 over 888:
        // 36.0 -> 30.8 us, by pairs of CTAs 24.9 -> 22.3; 2000 x 1600 over 2000 from 128 columns 41.8 -> 39.4).  Tiles narrower than 128
        // columns move more operand bytes for each of their products, and a last round of few tiles is over soon: those records stay as
        // they are below an eighth of a round (785 x 1160 over 384, 64 columns by pairs, 76 pairs' tiles: 14.3 us, 16.4 with 32; 3147 x 1352
        // over 1592, 128 columns 54.6, 62.3 with 96).  150 records of other sizes: 1.043 times faster than as written in the geometric
        // mean, six slower by more than 2 %; 1.041 and twenty without that line.
        const int per = kHwTileM * cg, step = cg == 2 || tn % 32 == 0 ? 32 : 16;
        const long long rows = (long long)((M + per - 1) / per) * B, units = kSms / cg;
        const long long tiles = rows * ((N + tn - 1) / tn), rounds = (tiles + units - 1) / units, columns = rounds * units / rows;
        if (rounds >= 2 && rounds <= 4) {
            const int even = round_up((int)((N + columns - 1) / columns), step);
            const bool worth = even >= 128 || (tiles - (rounds - 1) * units) * 8 >= units;
            if (even < tn && worth) { tn = even; changed |= TT_CHG_TILE_N; L.tile_n = tn; }
        }
    }
    int sk = persistent ? 1 : rec->split_k;
    if (sk > k_tiles) {
        if (strict) return TT_ERR_INVALID_SCHEDULE;
        sk = k_tiles;
    }
    if (may.fewer_splits && !strict && !persistent && !x3 && sk >= 2 && sk <= 8 && rec->ctas_per_sm != 2) {
        // The splits of a tile are a cluster, and a cluster keeps to one group of SMs: where the record's splits of all tiles are not
        // resident at once, fewer of them may take fewer rounds.  36 tiles of 64 columns in fours, of which 33 are resident, take two
        // rounds of a quarter of the reduction, in threes one round of a third (533 x 464 over 4096: 28.7 -> 20.5 us; as written in eighths 32.8;
        // 494 tiles in fours 119 -> 53, 608 in sevens 256 -> 52).  Cycles: 8 of the reduction take 64 to
        // issue or what the columns take, a round 3000 for its ends and 1000 for the exchange; the line is drawn at 0.85.
        const long long tiles = (long long)((M + kHwTileM - 1) / kHwTileM) * ((N + tn - 1) / tn) * B;
        const auto cost = [&](int n) {
            const long long rounds = (tiles + kResidentClusters[n] - 1) / kResidentClusters[n];
            return rounds * ((long long)((k_tiles + n - 1) / n) * (tk / 8) * std::max(64, tn) + (n > 1 ? 4000 : 3000));
        };
        int best = sk;
        if (tiles > kResidentClusters[sk])
            for (int n = sk - 1; n >= 1; --n) if (cost(n) * 20 < cost(sk) * 17 && cost(n) < cost(best)) best = n;
        sk = best;
    }
    const int per_split = (k_tiles + sk - 1) / sk;
    sk = (k_tiles + per_split - 1) / per_split;          // every split owns at least one reduction tile
    if (sk != rec->split_k) changed |= TT_CHG_SPLIT_K;
    L.split_k = sk;
    // accumulators: a power of two, all of them inside the 512 columns of tensor memory, none left without a step
    int nacc = (persistent || x3) ? 1 : std::min(8, pow2_floor(std::max(1, rec->acc_split)));
    while (nacc > 1 && (nacc * tn > 512 || (long long)nacc > (long long)per_split * (tk / 8))) nacc >>= 1;
    if (nacc != std::max(1, rec->acc_split)) { if (strict) return TT_ERR_INVALID_SCHEDULE; changed |= TT_CHG_ACC; }
    L.acc_split = nacc;
    // buffers beyond the reduction tiles of one CTA would never be filled
    // (the persistent form's pipeline runs on across tiles: there the depth is bounded by shared memory alone)
    if (!persistent && st > per_split) { st = per_split; changed |= TT_CHG_STAGES; L.stages = st; }
    if (strict && (changed & ~TT_CHG_TILE_M)) return TT_ERR_INVALID_SCHEDULE;

    const int atom_k = std::min(tk, 32), n_atoms = tk / atom_k, row_bytes = atom_k * 4;
    const unsigned a_stage = (unsigned)n_atoms * kHwTileM * row_bytes;
    // an MN-major operand B takes whole boxes of 32 rows
    const unsigned b_stage = swap || !mn_operand ? (unsigned)n_atoms * (tn / cg) * row_bytes : (unsigned)round_up(tn, 32) * tk * 4;
    if (persistent) {
        // ---- the persistent form: its own shared-memory plan, grid and arguments ----
        const tt_shapes& o = w->sh;
        const bool conv1 = w->op == TT_OP_CONV2D, nn = w->op == TT_OP_BATCH_MATMUL && !o.trans_b;
        // logical operands U (rows i of the output) and V (columns j): which of them is row-contiguous
        const bool u_mn = false, v_mn = conv1 || nn;
        const bool a_mn = swap ? v_mn : u_mn, b_mn = swap ? u_mn : v_mn;
        // How many stages: the record's, or, with a row-contiguous operand (whose boxes come from memory one after the other),
        // what the record field slab_tiles asks for; 0 = as many as fit, at most 8.
        const bool mn = a_mn || b_mn;
        if (mn && rec->slab_tiles < 0) return TT_ERR_INVALID_SCHEDULE;
        const long long stage = (long long)a_stage + b_stage;
        // Read-out staging: eight warps with three (a residual passes through them) or two 32 x 32 blocks each, fewer where
        // the record's stages need the room; never less than four warps with one block (5 KB, the width the unaligned
        // read-out's transposition takes).
        struct { int warps, bufs; } epi[] = {{8, 3}, {8, 2}, {4, 3}, {4, 2}, {8, 1}, {4, 1}};
        auto warp_bytes = [](int bufs) { return bufs == 1 ? 5120ll : bufs * 4096ll; };
        const bool res = w->sh.has_residual != 0;
        int ew = 4, eb = 1;
        auto total = [&](int stages, int warps, int bufs) { return round_up64(stages * stage, 1024) + warps * warp_bytes(bufs) + 1024; };
        while (!strict && st > 1 && total(st, 4, 1) > kDynSmemLimit) { --st; changed |= TT_CHG_STAGES; }
        // (from here on only what fits is asked for: a request for more must not cost the read-out its buffers)
        int want = !mn ? st : (rec->slab_tiles == 0 ? kMaxStages : std::min(kMaxStages, std::max(st, rec->slab_tiles)));
        while (rec->slab_tiles != 0 && want > st && total(want, 4, 1) > kDynSmemLimit) {
            if (strict) return TT_ERR_INVALID_SCHEDULE;
            --want;
        }
        // with a free depth the read-out's ring comes first, as long as three stages (or the record's) stay in flight
        const int keep = rec->slab_tiles == 0 && mn ? std::max(st, 3) : std::max(want, st);
        for (const auto& o : epi) {
            if (!res && o.bufs == 3) continue;
            if (total(keep, o.warps, o.bufs) <= kDynSmemLimit || (o.warps == 4 && o.bufs == 1)) { ew = o.warps; eb = o.bufs; break; }
        }
        int depth = std::max(want, st);
        while (depth > st && total(depth, ew, eb) > kDynSmemLimit) --depth;
        const long long smem_p = total(depth, ew, eb);
        if (!mn && rec->slab_tiles != 0) changed |= TT_CHG_SLAB;
        L.stages = st; L.split_k = 1; L.acc_split = 1; L.slab_tiles = (mn && rec->slab_tiles != 0) ? depth : 0; L.ctas_per_sm = 1;
        if (!strict && L.slab_tiles != rec->slab_tiles) changed |= TT_CHG_SLAB;
        if (rec->ctas_per_sm == 2) { if (strict) return TT_ERR_INVALID_SCHEDULE; changed |= TT_CHG_FORM; }
        if (strict && (changed & ~TT_CHG_TILE_M)) return TT_ERR_INVALID_SCHEDULE;
        const int rows_m = kHwTileM * cg;
        const int tiles_m = (M + rows_m - 1) / rows_m, tiles_n = (N + tn - 1) / tn;
        const long long units = (long long)tiles_m * tiles_n * B;
        if (units > 0x7fffffffLL) return TT_ERR_RESOURCE;
        I = tt_apply_info{};
        I.legal = L; I.changed = changed;
        I.grid_x = (int)std::min<long long>(units, kSms / cg) * cg; I.grid_y = 1; I.grid_z = 1;   // the launcher clamps to the device's SM count
        I.threads = kGemmThreads;
        // one CTA per SM: ask for more than half of an SM's shared memory
        I.smem_bytes = (int)std::max<long long>(smem_p, 116 * 1024);
        I.tmem_cols = std::max(32, pow2_ceil(tn + round_up(tn, 32)));     // (the read-out takes whole blocks of 32 columns)
        I.workspace_bytes = 0; I.launches = 1;
        plan->partial_bytes = 0;
        if (smem_p > kDynSmemLimit) return TT_ERR_RESOURCE;
        GemmArgs& g = plan->g;
        g = GemmArgs{};
        g.M = M; g.N = N; g.K = K; g.batch = B;
        g.tile_n = tn; g.tile_k = tk; g.stages = depth;
        g.k_tiles = k_tiles; g.k_tiles_per_split = k_tiles; g.split_k = 1;
        g.tiles_m = tiles_m; g.tiles_n = tiles_n; g.raster = L.raster;
        g.atom_k = atom_k; g.n_atoms = n_atoms; g.row_bytes = row_bytes;
        g.swz_mask = row_bytes == 128 ? 7 : (row_bytes == 64 ? 3 : 1);
        g.a_stage_bytes = a_stage; g.b_stage_bytes = b_stage;
        g.tmem_cols = (unsigned)I.tmem_cols; g.n_acc = 1; g.cluster = 0;
        g.idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((unsigned)(tn >> 3) << 17) | ((unsigned)(rows_m >> 4) << 24) |
                  (a_mn ? 1u << 15 : 0u) | (b_mn ? 1u << 16 : 0u);          // (an MN-major operand is read transposed)
        g.persistent = 1; g.cta_group = cg; g.total_tiles = (int)units;
        g.a_mn = a_mn; g.b_mn = b_mn; g.b_rows_cta = tn / cg;
        g.epi_off = (unsigned)round_up64(depth * stage, 1024);
        g.epi_warps = ew; g.epi_bufs = eb; g.epi_warp_bytes = (unsigned)warp_bytes(eb);
        struct Opnd { int mode; long long rs, ks, bs; int batched; } U{}, V{};
        long long y_is, y_js, y_bs;
        int bias_on;
        if (conv1) {
            const long long hw = (long long)o.h * o.w;
            U = {OPM_TMA, K, 1, 0, 0};                              // filters [k][c]
            V = {OPM_TMA_MN, 1, hw, (long long)o.c * hw, 1};        // image: pixel index contiguous, channels hw apart
            y_is = hw; y_js = 1; y_bs = (long long)o.k * hw; bias_on = 1;
        } else if (w->op == TT_OP_DENSE) {
            U = {OPM_TMA, K, 1, 0, 0};
            V = {OPM_TMA, K, 1, 0, 0};
            y_is = o.nn; y_js = 1; y_bs = 0; bias_on = 2;
        } else {
            U = {OPM_TMA, K, 1, (long long)o.m * K, 1};
            if (o.trans_b) V = {OPM_TMA, K, 1, (long long)o.nn * K, 1};
            else V = {OPM_TMA_MN, 1, o.nn, (long long)o.nn * K, 1};
            y_is = o.nn; y_js = 1; y_bs = (long long)o.m * o.nn; bias_on = 2;
        }
        const int u_tensor = conv1 ? 1 : 0;
        plan->a_tensor = swap ? 1 - u_tensor : u_tensor;
        plan->b_tensor = 1 - plan->a_tensor;
        const Opnd& A = swap ? V : U;
        const Opnd& Bo = swap ? U : V;
        g.a_mode = A.mode; g.a_rs = A.rs; g.a_ks = A.ks; g.a_bs = A.bs; g.a_tma_batched = A.batched;
        g.b_mode = Bo.mode; g.b_rs = Bo.rs; g.b_ks = Bo.ks; g.b_bs = Bo.bs; g.b_tma_batched = Bo.batched;
        g.y_ms = swap ? y_js : y_is; g.y_ns = swap ? y_is : y_js; g.y_bs = y_bs;
        g.bias_mode = o.has_bias ? (swap ? 3 - bias_on : bias_on) : 0;
        g.act = o.act;
        g.tx_bytes = a_stage + b_stage;
        g.vec_store = (g.y_ns == 1 && g.y_ms % 4 == 0 && g.y_bs % 4 == 0) ? 1 : 0;
        // TMA read-out: 16-byte rows, whole 32-column blocks (a narrower last block would write its neighbour's columns), and
        // two ring blocks per warp for the last tile, whose read-out nothing hides, so that one fills while the other is sent
        g.epi_late = ew == 4 && !res && depth * stage >= 8ll * kLateRingBytes;
        g.y_tma_batched = y_bs != 0;
        g.epi_tma = g.vec_store && tn % 32 == 0 && g.y_ms != 1 && (eb >= 2 || g.epi_late);
        g.res_tma = res && eb >= 2 && (g.epi_tma || (g.y_ms == 1 && g.y_ns % 4 == 0 && g.y_bs % 4 == 0));
        return TT_OK;
    }
    // Shared memory: pipeline buffers (reused by the epilogue as a 32 x 36-float staging area per warp), then for
    // conv2d the k-table (one word per reduction index of a CTA's K range) and the slab of input rows from which
    // the im2col operand is expanded; 1 KB of alignment slack.
    // A slab row is an image row followed by `gap` zeros (the left/right padding of neighbouring rows share them).
    // Per channel the slab holds, for each of the output rows a tile can span, the input rows its filter rows
    // touch: consecutive rows when stride <= filter height, else `r` rows per output row.  A chunk holds the
    // channels that `slab_tiles` consecutive reduction tiles touch; two buffers when there are several chunks.
    // split_k of 2..8: the splits of a tile form a thread-block cluster and reduce through distributed shared memory
    // (each sends the bands of its partial tile to the CTAs that finish them); beyond 8 the partial tiles go through
    // a global workspace and the split that arrives last adds them up
    const int cluster = (sk >= 2 && sk <= 8) ? sk : 0;
    // the read-out stages through the pipeline buffers (idle by then): a 32 x 36 float block per warp, or, for the
    // cluster reduction, this split's whole partial tile in the layout of the reduction area
    const long long min_pipe = std::max<long long>((long long)kGatherWarps * 32 * 36 * 4, cluster ? 4LL * kHwTileM * (tn + 4) : 0);
    // cluster reduction area, apart from the pipeline buffers (peers write into it while this CTA may still be in its
    // main loop): per OTHER split, this CTA's band of the tile -- rows x (tile_n + 4) or columns x 128 floats
    const long long red_bytes = cluster ? (4 * std::max<long long>((long long)(sk - 1) * ((kHwTileM + sk - 1) / sk) * (tn + 4),
                                                                    (long long)(sk - 1) * ((tn + sk - 1) / sk) * kHwTileM) + 127) / 128 * 128 : 0;
    // A pointwise convolution on images of 16-byte multiples needs no slab: its pixels are an MN-major operand.
    if (strict && w->op == TT_OP_CONV2D && rec->slab_tiles > per_split) return TT_ERR_INVALID_SCHEDULE;
    const bool conv = w->op == TT_OP_CONV2D && !mn_operand;
    const long long ktab = conv ? (((long long)per_split * tk * 4 + 127) / 128) * 128 : 0;
    int sl_tiles = 0, sl_nbuf = 0, sl_wp = 0, sl_gap = 0, sl_chpitch = 0, sl_in_rows = 0, sl_rstep = 1;
    long long sl_buf_bytes = 0, chp = 0;
    bool sl_run = false;
    const int RS = conv ? s.r * s.s : 1;
    if (conv) {
        const int pix_rows = swap ? kHwTileM : tn;       // output pixels per tile of the im2col operand
        // A pointwise convolution (1x1, stride 1, no padding) sees no neighbourhood: its H x W pixels are one run of
        // H*W values per channel, and any H' x W' with the same product is the same kernel.  Rows of W' pixels with
        // W' the largest multiple of 4 that divides both H*W and the tile's pixel count make every tile a whole
        // number of rows, so a slab chunk holds exactly the tile's pixels (the image's own rows would add up to a
        // row on either side: 224 staged pixels for 128 at 56 x 56).
        bool whole_rows = false;
        if (s.r == 1 && s.s == 1 && s.stride_h == 1 && s.stride_w == 1 && s.pad_h == 0 && s.pad_w == 0) {
            const long long hw = (long long)s.h * s.w;
            int best = 0;
            for (int d = 16; d <= 248 && d <= pix_rows; d += 4)
                if (hw % d == 0 && pix_rows % d == 0) best = d;
            if (best > 0) { s.w = best; s.h = (int)(hw / best); P = s.h; Q = s.w; whole_rows = true; }
            // An image of no 16-byte multiple that one tile takes whole: the channels of a chunk are one run of memory, and in groups
            // of four a multiple of 16 bytes.  One copy instead of 7 4-byte ones per row: the layers at 7 x 7 of a MobileNetV2-shaped pass
            // take 5.7 to 7.1 us instead of 6.9 to 8.8, the whole pass 286 instead of 293.
            else if (hw <= pix_rows && s.c % 4 == 0) { s.w = (int)hw; s.h = 1; P = 1; Q = s.w; whole_rows = sl_run = true; }
        }
        const int out_rows = whole_rows ? std::min(P, pix_rows / Q) : std::min(P, (pix_rows + 2 * Q - 2) / Q);
        sl_rstep = std::min(s.stride_h, s.r);
        sl_in_rows = s.stride_h <= s.r ? (out_rows - 1) * s.stride_h + s.r : out_rows * s.r;
        sl_gap = sl_run ? 0 : round_up(std::max(1, std::max(s.pad_w, s.s - 1 - s.pad_w)), 4);
        sl_wp = s.w + sl_gap;
        chp = sl_run ? s.w : round_up(sl_in_rows * sl_wp, 4);
        if (chp * (long long)s.c >= (1ll << 28) || s.w > 4095 || sl_in_rows > 4095) return TT_ERR_RESOURCE;
        sl_chpitch = (int)chp;
    }
    // TMA can stage the slab when image rows are 16-byte multiples and consecutive slab rows are consecutive image
    // rows; a chunk is then one box of at most 256 channels
    const bool slab_tma = conv && (s.w % 4) == 0 && s.stride_h <= s.r && sl_wp <= 256 && sl_in_rows <= 256;
    auto chunk_channels = [&](long long tiles) { return std::min<long long>(s.c, (tiles * tk + RS - 2) / RS + 1); };
    auto chunk_bytes = [&](long long tiles) {
        // a tail of gap + 4 zeros follows the last row of the last channel
        return ((chunk_channels(tiles) * chp + sl_gap + 4) * 4 + 127) / 128 * 128;
    };
    // Operands whose rows are no 16-byte multiples: boxes of groups of four rows, beside the stages that they are realigned into
    // (unless the plan has no room for them; fewer than four rows make no group).
    const int x_rows = w->op == TT_OP_DENSE ? s.m : B * s.m, w_rows = w->op == TT_OP_DENSE ? s.nn : B * s.nn;
    const bool ragged = may.boxes && w->op != TT_OP_CONV2D && (K % 4) != 0;
    // A short reduction beside an operand that is gathered anyway is not worth their way: 132 heads of 21 x 64 over 21 4.4 us, 5.0 with boxes;
    // 36 of 41 x 64 over 41 5.2 and 4.7.
    const bool alone = w->op == TT_OP_BATCH_MATMUL && !w->sh.trans_b;
    const bool x_raw = ragged && x_rows >= 4 && !(alone && K <= 32), w_raw = ragged && w_rows >= 4 && (w->op == TT_OP_DENSE || w->sh.trans_b);
    const unsigned a_box = (swap ? w_raw : x_raw) ? (unsigned)round_up((tk + 4) * 4 * (kHwTileM / 4), 128) : 0u;
    const unsigned b_box = (swap ? x_raw : w_raw) ? (unsigned)round_up((tk + 4) * 4 * (tn / 4), 128) : 0u;
    const long long raw_stage = 4ll * (a_box + b_box);
    long long smem = 0;
    for (;;) {
        const long long pipe_try = std::max<long long>((long long)st * (a_stage + b_stage) * (x3 ? 2 : 1), min_pipe) + st * raw_stage;
        long long slab_total = 0;
        bool fits = true;
        if (conv) {
            const long long budget = kDynSmemLimit - 1024 - pipe_try - ktab - red_bytes;
            // largest chunk not above the request that fits (one buffer if it covers the CTA's whole K range)
            int t = rec->slab_tiles == 0 ? per_split : std::min(rec->slab_tiles, per_split);
            while (t >= 1 && ((t >= per_split ? 1 : 2) * chunk_bytes(t) > budget || (slab_tma && chunk_channels(t) > 256))) --t;
            fits = t >= 1;
            sl_tiles = std::max(t, 1);
            sl_nbuf = sl_tiles >= per_split ? 1 : 2;
            sl_buf_bytes = chunk_bytes(sl_tiles);
            slab_total = sl_nbuf * sl_buf_bytes;
        }
        smem = pipe_try + ktab + slab_total + red_bytes + 1024;
        if (fits && smem <= kDynSmemLimit) break;
        // reformulate: a shallower pipeline leaves room (never in strict mode, never below one buffer)
        if (strict || st <= 1) break;
        --st;
        changed |= TT_CHG_STAGES;
    }
    L.stages = st;
    const long long pipe = std::max<long long>((long long)st * (a_stage + b_stage) * (x3 ? 2 : 1), min_pipe) + st * raw_stage;
    if (conv) {
        if (rec->slab_tiles != 0 && sl_tiles != rec->slab_tiles) {
            if (strict) return TT_ERR_INVALID_SCHEDULE;
            changed |= TT_CHG_SLAB;
        }
        L.slab_tiles = rec->slab_tiles == 0 ? 0 : sl_tiles;
    } else {
        L.slab_tiles = 0;
    }
    int tmem_cols = std::max(32, pow2_ceil((nacc - 1) * tn + round_up(tn, 32)));     // (the read-out takes whole blocks of 32 columns)
    const int tiles_m = (M + kHwTileM - 1) / kHwTileM, tiles_n = (N + tn - 1) / tn;
    if ((long long)tiles_m * tiles_n > 0x7fffffffLL || sk > 65535 || B > 65535) return TT_ERR_RESOURCE;

    {
        // which build: two CTAs per SM need half the shared memory and half the tensor memory each
        const bool fits2 = smem <= 112 * 1024 && tmem_cols <= 256;
        const long long ctas = (long long)tiles_m * tiles_n * sk * B;
        int cps = rec->ctas_per_sm == 0 ? ((ctas > 2 * kSms && fits2) ? 2 : 1) : rec->ctas_per_sm;
        if (cps == 2 && !fits2) { if (strict) return TT_ERR_INVALID_SCHEDULE; cps = 1; changed |= TT_CHG_FORM; }
        L.ctas_per_sm = cps;
    }
    I = tt_apply_info{};
    I.legal = L;
    I.changed = changed;
    I.grid_x = tiles_m * tiles_n; I.grid_y = sk; I.grid_z = B;
    I.threads = kGemmThreads;
    I.smem_bytes = (int)std::min<long long>(smem, 0x7fffffff);
    I.tmem_cols = tmem_cols;
    // split-K workspace: partial tiles, then one arrival counter per (batch, tile)
    const bool ws = sk > 1 && cluster == 0;
    plan->partial_bytes = ws ? (((long long)sk * B * M * N * 4 + 255) / 256) * 256 : 0;
    I.workspace_bytes = ws ? plan->partial_bytes + (int64_t)B * tiles_m * tiles_n * 4 : 0;
    I.launches = 1;
    if (smem > kDynSmemLimit) return TT_ERR_RESOURCE;

    // The record's pipeline depth is what it needs at least: with one CTA per SM the shared memory that is left serves no one
    // else, so the ring takes as many stages as fit, up to a CTA's whole reduction.  A batch-1 layer then requests all of its
    // weights at once instead of a refill of two stages per trip to memory (the 84 kernels of the 12-layer encoder at batch 1
    // and 128 tokens: 528 us with the record's depth, 501 with this one).
    int depth = st;
    // A compensated CTA with a long reduction multiplies A and its remainders from tensor memory (the record is accounted for as if it
    // did not, so its ring may be deeper): 512 x 4096 -> 1024 in quarters 37.2 -> 29.9 us, 2000 x 1000 -> 3000 78.4 -> 73.3, 1024 x 1024 ->
    // 1024 22.5 -> 20.6.  The way there takes longer, which short reductions do not earn back: 36 x 520 -> 280 6.7 -> 7.4, 3 x 288 -> 1648 4.8 ->
    // 6.4.  Nor do stages with little in them: with 32 of the reduction it is 1.03 to 1.26 times faster for 128 to 176 columns, 0.97 to 1.01
    // for 96 and 112, 0.77 to 0.87 up to 64 and 0.86 for 256; with 64 of the reduction 1.04 to 1.23 from 32 columns on and 0.83 for 16; with 16
    // 0.64 to 0.88 for any.
    const bool x3_stage = tk >= 64 ? tn >= 32 : tk == 32 && tn >= 128 && tn <= 176;
    const bool x3_tmem = x3 && x3_stage && per_split * tk >= 512 && L.ctas_per_sm != 2;
    const long long run_stage = a_stage + b_stage + (x3_tmem ? b_stage : x3 ? (long long)a_stage + b_stage : 0);
    auto run_bytes = [&](int d) { return std::max<long long>(d * run_stage, min_pipe) + d * raw_stage + smem - pipe; };
    const long long ring_limit = L.ctas_per_sm == 2 ? smem : kDynSmemLimit;
    while (depth < std::min(kMaxStages, per_split) && run_bytes(depth + 1) <= ring_limit) ++depth;
    const long long run_pipe = std::max<long long>(depth * run_stage, min_pipe);
    plan->run_smem = (int)run_bytes(depth);
    GemmArgs& g = plan->g;
    g = GemmArgs{};
    g.M = M; g.N = N; g.K = K; g.batch = B;
    g.tile_n = tn; g.tile_k = tk; g.stages = depth;
    g.k_tiles = k_tiles; g.k_tiles_per_split = per_split; g.split_k = sk;
    g.tiles_m = tiles_m; g.tiles_n = tiles_n; g.raster = L.raster;
    g.atom_k = atom_k; g.n_atoms = n_atoms; g.row_bytes = row_bytes;
    g.swz_mask = row_bytes == 128 ? 7 : (row_bytes == 64 ? 3 : 1);
    g.a_stage_bytes = a_stage; g.b_stage_bytes = b_stage;
    g.ktab_off = (unsigned)run_pipe;
    g.slab_off = (unsigned)(run_pipe + ktab);
    g.red_off = (unsigned)(run_pipe + ktab + (long long)sl_nbuf * sl_buf_bytes);
    g.raw_off = (unsigned)(g.red_off + red_bytes); g.raw_stage_bytes = (unsigned)raw_stage; g.a_raw_box = a_box; g.b_raw_box = b_box;
    g.a_rows_all = swap ? w_rows : x_rows; g.b_rows_all = swap ? x_rows : w_rows;
    g.slab_buf_bytes = (unsigned)sl_buf_bytes; g.slab_nbuf = sl_nbuf; g.slab_tiles = sl_tiles;
    g.slab_wp = sl_wp; g.slab_gap = sl_gap; g.slab_chpitch = sl_chpitch; g.slab_in_rows = sl_in_rows;
    g.slab_rstep = sl_rstep;
    g.slab_tma = slab_tma ? 1 : (sl_run ? 2 : 0);
    if (g.slab_tma) {
        g.slab_box_ch = (int)chunk_channels(sl_tiles);
        g.slab_box_bytes = (unsigned)((long long)g.slab_box_ch * chp * 4);
    }
    g.magic_rstep = sl_rstep > 1 ? (unsigned)((0x100000000ull + sl_rstep - 1) / sl_rstep) : 0u;
    g.slab_vec16 = (s.w % 4) == 0;
    {
        const unsigned wpieces = (unsigned)(g.slab_vec16 ? s.w / 4 : s.w);
        g.magic_wpieces = wpieces > 1 ? (unsigned)((0x100000000ull + wpieces - 1) / wpieces) : 0u;
        g.magic_in_rows = sl_in_rows > 1 ? (unsigned)((0x100000000ull + sl_in_rows - 1) / sl_in_rows) : 0u;
    }
    g.tmem_cols = (unsigned)tmem_cols;
    g.n_acc = nacc;
    g.cluster = cluster;
    g.two_per_sm = L.ctas_per_sm == 2;
    g.x3 = x3 ? 1 : 0;
    if (x3_tmem) {
        // A's buffers in tensor memory, behind the accumulator: one per stage as far as the columns go
        const int acc = round_up(tn, 32);
        g.x3_col = (unsigned)acc;
        g.x3_bufs = std::min(depth, (512 - acc) / (2 * tk));
        I.tmem_cols = std::max(32, pow2_ceil(acc + g.x3_bufs * 2 * tk));
        g.tmem_cols = (unsigned)I.tmem_cols;
    }
    g.b_rows_cta = tn; g.cta_group = 1;
    // Instruction descriptor, kind::tf32: D = F32 (bits 4-5 = 1), A and B = TF32 (bits 7-9, 10-12 = 2), K-major or
    // (bits 15, 16 = 1) MN-major, N >> 3 at bits 17-22, M >> 4 at bits 24-28.
    g.idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((unsigned)(tn >> 3) << 17) | ((unsigned)(kHwTileM >> 4) << 24);
    // Operands of the logical contraction Y[b][i][j] = sum_k U[b][i][k] V[b][j][k], then the optional swap.
    struct Opnd { int mode; long long rs, ks, bs; int batched; } U{}, V{};
    long long y_is, y_js, y_bs;
    int bias_on;   // 1: bias indexed by i, 2: by j
    const bool k4 = (K % 4) == 0;
    if (w->op == TT_OP_CONV2D) {
        const long long hw = (long long)s.h * s.w;
        U = {k4 ? OPM_TMA : OPM_GATHER_K, K, 1, 0, 0};                         // filters [k][c*r*s], shared by images
        if (mn_operand) V = {OPM_TMA_MN, 1, hw, (long long)s.c * hw, 1};       // pixel index contiguous, channels hw apart
        else V = {OPM_IM2COL, 0, 0, (long long)s.c * hw, 1};                   // pixels x (c,r,s) gathered from NCHW
        y_is = (long long)P * Q; y_js = 1; y_bs = (long long)s.k * P * Q; bias_on = 1;
    } else if (w->op == TT_OP_DENSE) {
        U = {k4 ? OPM_TMA : x_raw ? OPM_RAW : OPM_GATHER_K, K, 1, 0, 0};
        V = {k4 ? OPM_TMA : w_raw ? OPM_RAW : OPM_GATHER_K, K, 1, 0, 0};
        y_is = s.nn; y_js = 1; y_bs = 0; bias_on = 2;
    } else {
        U = {k4 ? OPM_TMA : x_raw ? OPM_RAW : OPM_GATHER_K, K, 1, (long long)s.m * K, 1};
        if (s.trans_b) V = {k4 ? OPM_TMA : w_raw ? OPM_RAW : OPM_GATHER_K, K, 1, (long long)s.nn * K, 1};
        else V = {mn_operand ? OPM_TMA_MN : OPM_GATHER_ROWS, 1, s.nn, (long long)s.nn * K, 1};   // w[b][k][j]: rows j are contiguous
        y_is = s.nn; y_js = 1; y_bs = (long long)s.m * s.nn; bias_on = 2;
    }
    const int u_tensor = w->op == TT_OP_CONV2D ? 1 : 0;       // conv: U is the filter tensor; dense/bmm: U is x
    plan->a_tensor = swap ? 1 - u_tensor : u_tensor;
    plan->b_tensor = 1 - plan->a_tensor;
    const Opnd& A = swap ? V : U;
    const Opnd& Bo = swap ? U : V;
    g.a_mode = A.mode; g.a_rs = A.rs; g.a_ks = A.ks; g.a_bs = A.bs; g.a_tma_batched = A.batched;
    g.b_mode = Bo.mode; g.b_rs = Bo.rs; g.b_ks = Bo.ks; g.b_bs = Bo.bs; g.b_tma_batched = Bo.batched;
    g.y_ms = swap ? y_js : y_is; g.y_ns = swap ? y_is : y_js; g.y_bs = y_bs;
    g.bias_mode = s.has_bias ? (swap ? 3 - bias_on : bias_on) : 0;
    g.act = s.act;
    g.C = s.c; g.H = s.h; g.W = s.w; g.R = s.r; g.S = s.s; g.Q = Q;
    g.sh = s.stride_h; g.sw = s.stride_w; g.ph = s.pad_h; g.pw = s.pad_w;
    g.idesc |= (A.mode == OPM_TMA_MN ? 1u << 15 : 0u) | (Bo.mode == OPM_TMA_MN ? 1u << 16 : 0u);
    g.tx_bytes = (A.mode == OPM_TMA || A.mode == OPM_TMA_MN ? a_stage : 0) + (Bo.mode == OPM_TMA || Bo.mode == OPM_TMA_MN ? b_stage : 0);
    g.vec_store = (g.y_ns == 1 && g.y_ms % 4 == 0 && g.y_bs % 4 == 0) ? 1 : 0;
    return TT_OK;
}

// Compensated products are bound by shared memory: every operand byte is written by TMA, read and written again for its
// remainder and read by three products, 1.5 cycles per row of both tiles for each 8 of the reduction, and that is more than the
// products take up to 256 columns.  A compensated stage is twice the size and passes through the warps' hands between its arrival
// and its products.  Unless the record is to run as written (strict mode), two rules lay its tile out for that; the legal record
// says what they chose.
// Where only one of the record's stages fits, it becomes several of 32, so that the three steps overlap (512 x 1024 over 4096,
// stages of 64 with 128 columns: 182 us; as three of 32: 99).  Two of 64 are 3 % faster than four of 32.
// Where a tile of twice the record's columns does a round of the SMs for less, it takes its place (512 x 1024 over 4096 in
// quarters: 256 tiles of 64 columns are two rounds of 288 cycles a step, 128 of 128 one of 384).  The line lies at 0.85 of the
// record's cycles: at 0.60-0.67 the wide tile took 51.9 -> 39.4 us there, 97.1 -> 48.4 (32 columns), 31.7 -> 23.5 (256 x 4096 over
// 1024), 29.0 -> 17.3 (4096 x 512 over 512) and once 41.4 -> 42.5 (600 x 600 over 3000, 48 columns); at 0.89 46.0 -> 43.7 to
// 27.5 -> 24.1, which the wider grid's share of idle SMs makes a gamble on other sizes; at 1.4-1.5 30.5 -> 50.7 and 23.4 -> 38.1.
static tt_status legalise_gemm(const tt_workload* w, const tt_schedule_record* rec, int mode, Plan* plan) {
    const Plan fresh = *plan;
    // Whether a record is valid is decided with its own splits; ragged rows are gathered value by value where there is no room for their boxes.
    PlanOptions may{true, false};
    tt_status s = plan_gemm(w, rec, mode, may, plan);
    if (s != TT_OK && w->op != TT_OP_CONV2D && w->sh.kk % 4 != 0) {
        may.boxes = false;
        *plan = fresh;
        s = plan_gemm(w, rec, mode, may, plan);
    }
    if (s == TT_OK && plan->g.cluster && (long long)plan->info.grid_x * plan->gbatch > kResidentClusters[plan->g.cluster]) {
        // fewer splits have a longer reduction each, whose table of a convolution may not fit: then the record's own stay
        may.fewer_splits = true;
        Plan fewer = fresh;
        if (plan_gemm(w, rec, mode, may, &fewer) == TT_OK) *plan = fewer;
    }
    if (s != TT_OK || !plan->g.x3 || mode == TT_MODE_STRICT) return s;
    const int changed = plan->info.changed;
    auto replan = [&](const tt_schedule_record& r, bool same_splits) {
        Plan p = fresh;
        if (plan_gemm(w, &r, TT_MODE_LEGALISE, {true, true}, &p) != TT_OK || p.info.legal.stages < std::min(2, p.g.k_tiles_per_split) ||
            (same_splits && p.info.legal.split_k != plan->info.legal.split_k)) return;
        const tt_schedule_record& L = p.info.legal;
        p.info.changed = changed & ~(TT_CHG_TILE_N | TT_CHG_TILE_K | TT_CHG_STAGES | TT_CHG_SPLIT_K);
        if (L.tile_n != rec->tile_n) p.info.changed |= TT_CHG_TILE_N;
        if (L.tile_k != rec->tile_k) p.info.changed |= TT_CHG_TILE_K;
        if (L.stages != rec->stages) p.info.changed |= TT_CHG_STAGES;
        if (L.split_k != rec->split_k) p.info.changed |= TT_CHG_SPLIT_K;
        *plan = p;
    };
    if (plan->info.legal.tile_k > 32 && plan->g.stages == 1 && plan->g.k_tiles_per_split > 1) {
        tt_schedule_record thin = plan->info.legal;
        thin.stages = thin.tile_k / 32; thin.tile_k = 32;
        replan(thin, false);
    }
    const tt_schedule_record L = plan->info.legal;
    auto cost = [&](int tn) {
        const long long ctas = (long long)((plan->gm + kHwTileM - 1) / kHwTileM) * ((plan->gn + tn - 1) / tn) * L.split_k * plan->gbatch;
        return (double)((ctas + kSms - 1) / kSms) * std::max(1.5 * (kHwTileM + tn), 2.13 * tn);
    };
    if (L.tile_n <= 128 && rec->ctas_per_sm == 0 && cost(2 * L.tile_n) <= 0.85 * cost(L.tile_n)) {
        tt_schedule_record wide = L;
        wide.tile_n = 2 * L.tile_n; wide.tile_k = std::min(32, L.tile_k); wide.stages = 2;
        wide.ctas_per_sm = 0;
        replan(wide, true);
    }
    return s;
}

// Wavefronts of one 16-byte read of a window row by the first warps of a staged depthwise tile (8 lanes a phase, the banks
// repeat every 128 bytes), for strips `gw_step` 16-byte units apart, strip rows `gh_step` and planes `pl_step` apart.
static int dw_read_wavefronts(int groups_w, int groups_h, int planes, bool plane_next, int gw_step, int gh_step, int pl_step) {
    const int spp = groups_w * groups_h, lanes = std::min(128, planes * spp);
    int total = 0;
    for (int l0 = 0; l0 < lanes; l0 += 8) {
        int count[8] = {};
        for (int l = l0; l < std::min(lanes, l0 + 8); ++l) {
            const int gw = l % groups_w, r = l / groups_w;
            const int pl = plane_next ? r % planes : r / groups_h, gh = plane_next ? r / planes : r % groups_h;
            ++count[(gw * gw_step + gh * gh_step + pl * pl_step) & 7];
        }
        total += *std::max_element(count, count + 8);
    }
    return total;
}

// Geometry of the staged persistent kernel for a tile of d.tile_c planes x d.tile_h x d.tile_w outputs in strips of `rows` x `items`:
// box, buffers, the lanes' order.  may_widen: a row may take one more 16-byte unit than it needs.
static void plan_dw_boxes(DwArgs& d, int rows, int items, bool may_widen) {
    const int ncol = (items - 1) * d.sw + d.S, nld = (4 - d.pw + ncol + 3) / 4;      // 16-byte loads per window row
    // strips are `rows` tall: the box covers the rows of the last, possibly partial, strip too
    d.in_h = (round_up(d.tile_h, rows) - 1) * d.sh + d.R;
    d.box_w = (d.tile_w - items) * d.sw + 4 * nld;
    d.plane_next = 0;
    const int gw = d.tile_w / items, gh = (d.tile_h + rows - 1) / rows;
    if (gw * gh <= 256) {
        // the order of the lanes is free, and so is one more 16-byte unit per row where that lies outside the image: take what the banks serve in the fewest turns, the wider row
        // only for a fifth fewer
        int best = 0, wide = 0;
        for (int extra = 0; extra < (may_widen && d.tiles_w == 1 ? 2 : 1); ++extra)
            for (int order = 0; order < 2; ++order) {
                const int bw4 = d.box_w / 4 + extra;
                const int n = dw_read_wavefronts(gw, gh, d.tile_c, order != 0, items / 4 * d.sw, rows * d.sh * bw4, d.in_h * bw4);
                if (best == 0 || (extra == wide ? n < best : 5 * n <= 4 * best)) { best = n; wide = extra; d.plane_next = order; }
            }
        d.box_w += 4 * wide;
    }
    d.stage_bytes = (int)std::min<long long>(0x7fffff80, (((long long)d.tile_c * d.in_h * d.box_w * 4) + 127) / 128 * 128);
    d.wstage_bytes = (int)((((long long)d.tile_c * round_up(d.R * d.S + 1, 4) * 4) + 127) / 128 * 128);
}

// Image rows that are no 16-byte multiples: no box can fetch them, and a register-window strip fetches each value of its rows
// with a load of its own.  The run-staged persistent kernel runs instead, whatever the record's tile (except in strict mode); its
// tiles are this rule's, and the legal record (raster = 1 on such rows) names them: strips of the height that takes the fewest
// instructions for the image's rows, channels for up to 256 threads in buffers of 24 KB, but two tiles for every SM first.  From a
// quarter of a million outputs on: 480 x 14 x 14, 5x5, takes 4.5 us either way for one image, 4.7 instead of 7.5 for 4 and 78
// instead of 134 for 256; 960 x 7 x 7, 3x3, 3.6 instead of 2.9 for 4 (188 thousand outputs), 5.0 instead of 5.2 for 16 and 30
// instead of 44 for 256.
static bool plan_dw_runs(const tt_workload* w, DwArgs& d, tt_apply_info& I, tt_schedule_record& L) {
    const tt_shapes& s = w->sh;
    const long long planes = (long long)s.n * s.c, hw = (long long)s.h * s.w;
    if (s.w % 4 == 0 || w->Q > 256 || planes > 0x7fffffffLL || hw > (1 << 24)) return false;
    DwArgs t = d;
    double best_cost = 0;
    // Instructions of a strip: per window row its reads, their predicates and its address, per output row its products, clamp and
    // store, 40 to set it up.  On 12 shapes of both filters and strides the choice is the fastest of the three or within 5 % of it
    // (480 x 14 x 14, 5x5, 256 images: 7 rows 58.9 us, 4 84.4, 2 113; 200 x 15 x 15, 5x5, 64 images: 4 rows 15.9, 7 16.3; 120 x 31 x 33, 3x3
    // stride 2, 32 images: 4 rows 6.9, 7 7.5; the 5 %: 576 x 14 x 14, 3x3 stride 2, 256 images: 7 rows 28.1, 4 26.7).
    for (int rows : {7, 4, 2}) {
        const int in_rows = (rows - 1) * s.stride_h + s.r;
        const double cost = (double)((w->P + rows - 1) / rows) * (in_rows * (2.0 * s.r + 3) + rows * (s.r * s.r + 4.0) + 40);
        if (best_cost == 0 || cost < best_cost) { best_cost = cost; t.window_rows = rows; }
    }
    const int rows = t.window_rows;
    t.items = s.w % 2 == 0 ? 2 : 1;                        // even rows: a thread takes two columns, read in aligned pairs
    t.runs = 1; t.tile_w = w->Q;
    t.vec = w->Q % 2 == 0 ? t.items : 1;
    const int lanes_q = (w->Q + t.items - 1) / t.items;    // threads of a strip row
    int upw = lanes_q <= 32 ? 32 / lanes_q : 0;            // strip rows a warp takes side by side ...
    if (upw * lanes_q < 28) upw = 0;                       // ... unless that leaves more than an eighth of its lanes idle
    const int fit = upw ? 8 * upw : 256 / lanes_q;         // ... and 256 threads
    t.tile_h = w->P; t.tile_c = 1;
    if (hw * 4 > 24 * 1024) {
        // bands of one plane, of whole strips
        t.tile_h = rows;
        while (t.tile_h + rows <= w->P && (long long)((t.tile_h + rows - 1) * s.stride_h + s.r) * s.w * 4 <= 24 * 1024) t.tile_h += rows;
    }
    t.tiles_h = (w->P + t.tile_h - 1) / t.tile_h; t.tiles_w = 1;
    const int strips_h = (t.tile_h + rows - 1) / rows;
    t.strip_rows = std::min(strips_h, fit);
    if (t.tiles_h == 1) {
        const long long share = std::max(1LL, planes / (2 * kSms));
        t.tile_c = (int)std::min<long long>({(long long)s.c, share, (long long)std::max(1, fit / t.strip_rows), std::max(1LL, 24 * 1024 / (hw * 4))});
        // groups of channels as equal as they come
        const int groups = (s.c + t.tile_c - 1) / t.tile_c;
        t.tile_c = (s.c + groups - 1) / groups;
    }
    t.in_h = (round_up(t.tile_h, rows) - 1) * s.stride_h + s.r;
    const int units = t.tile_c * t.strip_rows;
    t.units_per_warp = upw; t.unit_far = 0;
    if (upw > 1) {
        // which units share a warp decides how its reads fall on the banks: neighbours, or ones a fixed distance apart
        const int far = (units + upw - 1) / upw;
        int turns[2] = {};
        for (int pass = 0; pass < 2; ++pass)
            for (int wp = 0; wp < far; ++wp) {
                int count[2][32] = {};                     // a pair takes two banks: half a warp at a time
                for (int j = 0; j < upw; ++j) {
                    const int unit = pass ? wp + j * far : wp * upw + j;
                    if (unit >= units) continue;
                    const long long off = unit / t.strip_rows * hw + (long long)(unit % t.strip_rows) * rows * s.stride_h * s.w;
                    for (int q = 0; q < lanes_q; ++q)
                        ++count[t.items == 2 && j * lanes_q + q >= 16][(off + (long long)q * t.items * s.stride_w) & 31];
                }
                turns[pass] += *std::max_element(count[0], count[0] + 32) + *std::max_element(count[1], count[1] + 32);
            }
        if (turns[1] < turns[0]) t.unit_far = far;
    }
    const int threads = std::min(256, upw ? (units + upw - 1) / upw * 32 : round_up(units * lanes_q, 32));
    const long long run = t.tiles_h == 1 ? t.tile_c * hw : (long long)std::min(t.in_h, s.h) * s.w;
    t.stage_bytes = (int)((run * 4 + 32 + 127) / 128 * 128);
    t.tma_stages = 2;
    while (t.tma_stages < 4 && (t.tma_stages + 1ll) * t.stage_bytes <= 56 * 1024) ++t.tma_stages;
    const long long smem = (long long)t.tma_stages * t.stage_bytes + round_up(s.w * 4, 128);
    const long long total = (long long)((s.c + t.tile_c - 1) / t.tile_c) * s.n * t.tiles_h;
    if (smem > kDynSmemLimit || total > 0x7fffffffLL || planes * w->P * w->Q < 1 << 18) return false;
    t.total_tiles = (int)total;
    const long long per_sm = std::max<long long>(1, std::min<long long>({16LL, (228 * 1024) / (smem + 1024), 2048LL / threads}));
    d = t;
    I.grid_x = (int)std::min<long long>(total, kSms * per_sm); I.grid_y = 1; I.grid_z = 1;
    I.threads = threads; I.smem_bytes = (int)smem; I.launches = 1;
    L.raster = 1; L.stages = d.tma_stages; L.unroll = rows; L.items_per_thread = d.items; L.vec_width = d.vec;
    L.tile_m = d.tile_c; L.block_y = d.tile_h; L.block_x = d.tile_w; L.threads = threads;
    return true;
}

static tt_status legalise_dw(const tt_workload* w, const tt_schedule_record* rec, int mode, Plan* plan) {
    const tt_shapes& s = w->sh;
    const bool strict = mode == TT_MODE_STRICT;
    tt_schedule_record L = *rec;
    int changed = 0;
    if (rec->tile_m <= 0 || rec->block_x <= 0 || rec->block_y <= 0 || rec->items_per_thread <= 0 ||
        rec->vec_width <= 0 || rec->threads <= 0 || rec->unroll < 0 || rec->raster < 0 || rec->raster > 1)
        return TT_ERR_INVALID_SCHEDULE;
    // unroll >= 1 asks for the register-window kernel (that many output rows per thread: 1, 2 or 4), which exists
    // for square 3x3 / 5x5 filters with "same" padding and stride 1 or 2 and works on strips of 4 columns;
    // unroll == 0, or any other filter, takes the shared-memory staged kernel
    const bool window_ok = s.r == s.s && (s.r == 3 || s.r == 5) && s.stride_h == s.stride_w &&
                           (s.stride_h == 1 || s.stride_h == 2) && s.pad_h == s.r / 2 && s.pad_w == s.r / 2;
    DwArgs& d = plan->dw;
    d = DwArgs{};
    d.N = s.n; d.C = s.c; d.H = s.h; d.W = s.w; d.R = s.r; d.S = s.s; d.P = w->P; d.Q = w->Q;
    d.sh = s.stride_h; d.sw = s.stride_w; d.ph = s.pad_h; d.pw = s.pad_w; d.act = s.act;
    tt_apply_info& I = plan->info;
    I = tt_apply_info{};
    if (rec->unroll >= 1 && window_ok) {
        DwArgs runs = d;
        tt_schedule_record R = *rec;
        if (plan_dw_runs(w, runs, I, R)) {
            int replaced = 0;
            if (R.tile_m != rec->tile_m) replaced |= TT_CHG_TILE_M;
            if (R.block_x != rec->block_x || R.block_y != rec->block_y || R.threads != rec->threads) replaced |= TT_CHG_BLOCK;
            if (R.items_per_thread != rec->items_per_thread) replaced |= TT_CHG_ITEMS;
            if (R.vec_width != rec->vec_width) replaced |= TT_CHG_VEC;
            if (R.stages != rec->stages) replaced |= TT_CHG_STAGES;
            if (R.raster != rec->raster || R.unroll != rec->unroll) replaced |= TT_CHG_FORM;
            if (!strict || replaced == 0) {
                I.legal = R; I.changed = replaced;
                d = runs;
                return TT_OK;
            }
        }
    }
    if (strict && (rec->tile_m > s.c || rec->block_y > w->P || rec->block_x > round_up(w->Q, 4)))
        return TT_ERR_INVALID_SCHEDULE;
    L.tile_m = std::min(rec->tile_m, s.c);
    if (L.tile_m != rec->tile_m) changed |= TT_CHG_TILE_M;
    L.block_y = std::min(rec->block_y, w->P);
    int vec = rec->vec_width >= 4 ? 4 : (rec->vec_width >= 2 ? 2 : 1);
    while (vec > 1 && (w->Q % vec) != 0) vec >>= 1;        // rows of y must stay vector-aligned
    int items = std::min(8, pow2_floor(rec->items_per_thread));
    items = std::max(items, vec);
    int window_rows = 0;
    if (rec->unroll >= 1 && window_ok) {
        window_rows = rec->unroll >= 4 ? 4 : (rec->unroll >= 2 ? 2 : 1);
        items = rec->items_per_thread >= 8 ? 8 : 4;      // strips of 4 or 8 columns; 8-wide strips are at most 2 rows tall
        if (items == 8 && window_rows > 2) window_rows = 2;
    }
    // (strips of 7 rows exist in the box-staged form of 5x5 filters)
    const bool seven = rec->unroll == 7 && rec->raster == 1 && window_rows == 4 && s.r == 5 && s.w % 4 == 0;
    L.unroll = seven ? 7 : window_rows;
    // a record that names the register-window form (or a strip height it does not have) on a filter without one runs
    // another kernel form than it was written for: a reformulation, invalid when nothing may be reformulated
    if (L.unroll != rec->unroll) changed |= TT_CHG_FORM;
    int bx = std::min(rec->block_x, round_up(w->Q, items));
    bx = round_up(bx, items);
    if (bx != rec->block_x || L.block_y != rec->block_y) changed |= TT_CHG_BLOCK;
    L.block_x = bx;
    if (items != rec->items_per_thread) changed |= TT_CHG_ITEMS;
    L.items_per_thread = items;
    if (vec != rec->vec_width) changed |= TT_CHG_VEC;
    L.vec_width = vec;
    int th = std::min(window_rows ? 256 : 1024, std::max(32, round_up(rec->threads, 32)));
    if (th != rec->threads) changed |= TT_CHG_BLOCK;
    L.threads = th;
    if (strict && changed) return TT_ERR_INVALID_SCHEDULE;

    d.tile_c = L.tile_m; d.tile_h = L.block_y; d.tile_w = L.block_x;
    d.in_h = (d.tile_h - 1) * d.sh + d.R;
    d.in_w = (d.tile_w - 1) * d.sw + d.S;
    d.items = items; d.vec = vec;
    d.tiles_c = (s.c + d.tile_c - 1) / d.tile_c;
    d.tiles_h = (w->P + d.tile_h - 1) / d.tile_h;
    d.tiles_w = (w->Q + d.tile_w - 1) / d.tile_w;
    d.window_rows = window_rows;                           // (a box-staged plan may change it below)
    d.vec_in = (s.w % 4) == 0;
    long long smem = window_rows ? 0 : (long long)d.tile_c * ((long long)d.in_h * d.in_w + d.R * d.S + 1) * 4;
    I = tt_apply_info{};
    I.legal = L; I.changed = changed;
    long long gx = (long long)d.tiles_w * d.tiles_h * d.tiles_c;
    // raster = 1 (with a window-kernel filter and 16-byte image rows): the tiles' input boxes are staged by TMA in
    // `stages` buffers, next to the filters and biases of their planes, and CTAs walk the tiles persistently
    L.raster = 0;
    if (rec->raster == 1 && window_rows > 0 && (s.w % 4) == 0) {
        const long long planes = (long long)s.n * s.c;
        // Unless the record is to run as written (strict mode): tiles keep to one image, in groups of channels as equal as they
        // come, and a 5x5 filter's strips of 4 rows become strips of 7 where those cover the tile as well and the chip has tiles to
        // spare: a strip then reads 11 rows for 7, not 8 for 4.  256 images of 240 x 28 x 28: 98 -> 81 us; 32 of 200 x 56 x 56: 43 -> 37; 16 of
        // 240 x 28 x 28: 10.9 -> 10.2; stride 2, 64 of 96 x 112 x 112: 76 -> 66, but 32 of 200 x 56 x 56: 22.5 -> 23.6.  Elsewhere: 4 of 240 x 28 x 28
        // (240 tiles) 5.3 -> 6.3, 20-row tiles 38 -> 40, 12-row tiles 16 -> 20.  A 3x3 filter reads 9 rows for 7 against 6 for 4: 56-pixel rows 44 -> 45
        // and 40 -> 45, 28-pixel 61 -> 62, 20-pixel 36 -> 38, stride 2 at 112 32.9 -> 32.7.
        // Everything below is about the tile that runs, and so is the legal record.
        int rows = L.unroll;
        DwArgs t = d;
        const int groups = (s.c + t.tile_c - 1) / t.tile_c;
        if (!strict) {
            rows = window_rows;
            if (rows == 4 && s.r == 5 && round_up(d.tile_h, 7) <= round_up(d.tile_h, 4) && (planes + d.tile_c - 1) / d.tile_c * d.tiles_h * d.tiles_w >= kSms * 4) rows = 7;
            t.tile_c = (s.c + groups - 1) / groups;
        }
        int stg = 0;
        auto smem_of = [&](int n) { return (long long)n * t.stage_bytes + t.wstage_bytes + 128; };
        for (const bool may_widen : {true, false}) {       // (a wider row that does not fit is no reason to leave this form)
            plan_dw_boxes(t, rows, items, may_widen);
            stg = std::min(4, std::max(2, rec->stages));
            while (stg > 2 && smem_of(stg) > kDynSmemLimit) --stg;
            if (smem_of(stg) <= kDynSmemLimit && t.box_w <= 256) break;
        }
        if (t.box_w <= 256 && t.in_h <= 256 && t.tile_c <= 256 && smem_of(stg) <= kDynSmemLimit && planes <= 0x7fffffffLL) {
            d = t;
            d.window_rows = rows;
            if (stg != rec->stages) { if (strict) return TT_ERR_INVALID_SCHEDULE; I.changed |= TT_CHG_STAGES; }
            L.raster = 1; L.stages = stg;
            d.tma_stages = stg;
            // no more threads than a tile has strips
            if (!strict) th = std::min(th, round_up(d.tile_c * ((d.tile_h + rows - 1) / rows) * (d.tile_w / items), 32));
            L.unroll = rows; L.tile_m = d.tile_c; L.threads = th;
            if (L.unroll != rec->unroll) I.changed |= TT_CHG_FORM;
            if (L.tile_m != rec->tile_m) I.changed |= TT_CHG_TILE_M;
            if (L.threads != rec->threads) I.changed |= TT_CHG_BLOCK;
            const long long total = (long long)groups * s.n * d.tiles_h * d.tiles_w;
            if (total > 0x7fffffffLL) return TT_ERR_RESOURCE;
            d.total_tiles = (int)total;
            smem = smem_of(stg);
            const long long per_sm = std::max<long long>(1, std::min<long long>(8, (228 * 1024) / (smem + 1024)));   // (applying the record lowers it to what registers allow)
            gx = std::min<long long>(total, kSms * per_sm);
            I.legal = L;
            I.grid_x = (int)gx; I.grid_y = 1; I.grid_z = 1;
            I.threads = th; I.smem_bytes = (int)smem; I.launches = 1;
            return TT_OK;
        }
    }
    if (rec->raster != 0) { if (strict) return TT_ERR_INVALID_SCHEDULE; I.changed |= TT_CHG_FORM; }
    L.unroll = window_rows;
    I.legal = L;
    I.grid_x = (int)std::min<long long>(gx, 0x7fffffff); I.grid_y = s.n; I.grid_z = 1;
    I.threads = th; I.smem_bytes = (int)std::min<long long>(smem, 0x7fffffff);
    I.launches = 1;
    if (smem > kDynSmemLimit || gx > 0x7fffffffLL || s.n > 65535) return TT_ERR_RESOURCE;
    return TT_OK;
}

static tt_status legalise_row(const tt_workload* w, const tt_schedule_record* rec, int mode, Plan* plan) {
    const tt_shapes& s = w->sh;
    const bool strict = mode == TT_MODE_STRICT;
    tt_schedule_record L = *rec;
    int changed = 0;
    if (rec->block_x <= 0 || rec->block_y <= 0 || rec->vec_width <= 0) return TT_ERR_INVALID_SCHEDULE;
    const long long rows = (long long)s.batch * s.m;
    int lanes = std::min(32, pow2_floor(rec->block_x));
    int vec = rec->vec_width >= 4 ? 4 : (rec->vec_width >= 2 ? 2 : 1);
    while (vec > 1 && (s.nn % vec) != 0) vec >>= 1;
    if (strict && (long long)rec->block_x * rec->vec_width > round_up(s.nn, 4)) return TT_ERR_INVALID_SCHEDULE;
    int rpc = rec->block_y;
    while ((rpc * lanes) % 32 != 0) ++rpc;                 // whole warps
    if ((long long)rpc * lanes > 1024) rpc = 1024 / lanes;
    if (lanes != rec->block_x || rpc != rec->block_y) changed |= TT_CHG_BLOCK;
    if (vec != rec->vec_width) changed |= TT_CHG_VEC;
    L.block_x = lanes; L.block_y = rpc; L.vec_width = vec;
    if (strict && changed) return TT_ERR_INVALID_SCHEDULE;
    RowArgs& r = plan->row;
    r = RowArgs{};
    r.rows = rows; r.cols = s.nn; r.scale = s.scale; r.lanes_per_row = lanes; r.rows_per_cta = rpc; r.vec = vec;
    tt_apply_info& I = plan->info;
    I = tt_apply_info{};
    long long gx = (rows + rpc - 1) / rpc;
    const bool too_many = gx > 0x7fffffffLL;
    I.threads = rpc * lanes; I.launches = 1;
    if ((s.nn & 3) != 0) {
        // Ragged rows pass through shared memory as long as a lane's values stay in registers and a warp's rows fit.  A chunk is a
        // number of rows that fills whole 16-byte groups and keeps all lanes busy: four, or two of even rows where that is all a warp should
        // have (14 KB and more in four: 30000 rows of 1174 74 -> 62 us; less than 14 chunks of four for each SM, of 1.5 KB and more: 3000 of
        // 330 5.9 -> 4.7), or eight of short rows where there are still 54 chunks of them for each SM (100000 of 33 15.3 -> 11.9, 100000 of 130
        // 22.1 -> 19.3; 30000 of 33, which are fewer, by 32 lanes 8.5 with four and 13.2 with eight).  159 combinations of length, rows and lanes: 1.062 times faster than four in the
        // geometric mean, none slower by more than 2 %, and 1.6 % off the best of 2 to 64.  Warps per CTA follow the record, fewer where their
        // rows or registers would not fit.  The lanes' accesses are single values.
        const int per_lane = (s.nn + lanes - 1) / lanes, least = 32 / lanes;
        int chunk = std::max(4, least);
        const long long four = 16ll * s.nn, fours = rows / 4;
        if (s.nn % 2 == 0 && (four > 14000 || (four >= 1500 && fours < 14 * kSms))) chunk = std::max(2, least);
        else if (four < kRowRun && rows / 8 >= 54 * kSms && 32ll * s.nn * (rpc * lanes / 32) <= kRowSmem) chunk = std::max(8, least);
        const int warps = (int)std::min<long long>(std::min(rpc * lanes, ragged_threads(per_lane)) / 32, kRowSmem / ((long long)chunk * s.nn * 4));
        if (warps >= 1 && per_lane <= kRaggedMost && !(strict && (vec != 1 || warps * 32 != rpc * lanes))) {
            r.warps = warps; r.chunk = chunk;
            L.vec_width = 1; L.block_y = warps * 32 / lanes;
            if (L.vec_width != rec->vec_width) changed |= TT_CHG_VEC;
            if (L.block_y != rec->block_y) changed |= TT_CHG_BLOCK;
            gx = (rows + (long long)warps * chunk - 1) / ((long long)warps * chunk);
            I.threads = 32 * warps; I.smem_bytes = warps * chunk * s.nn * 4;
        }
    }
    const int groups = ((s.nn >> 2) + lanes - 1) / lanes;      // 16-byte groups per lane
    if (vec == 4 && groups <= kCachedMost && !(strict && rpc * lanes > cached_threads(groups))) {
        // rows that fit the lanes' registers are read once, by as many threads as have that many registers
        r.cached = groups;
        if (rpc * lanes > cached_threads(groups)) {
            rpc = r.rows_per_cta = cached_threads(groups) / lanes;
            L.block_y = rpc; changed |= TT_CHG_BLOCK;
            gx = (rows + rpc - 1) / rpc; I.threads = rpc * lanes;
        }
    }
    I.legal = L; I.changed = changed;
    I.grid_x = (int)std::min<long long>(gx, 0x7fffffff); I.grid_y = 1; I.grid_z = 1;
    if (too_many) return TT_ERR_RESOURCE;
    return TT_OK;
}

tt_status legalise(const tt_workload* w, const tt_schedule_record* rec, int mode, int strict_class, Plan* plan) {
    if (!w || !rec || !plan) return TT_ERR_INVALID_ARG;
    if (rec->version != TT_RECORD_VERSION) return TT_ERR_INVALID_SCHEDULE;
    // A schedule written for another loop structure tries to transform loops that do not exist (Section 4.2).
    if ((int)rec->family != w->family) return TT_ERR_CLASS_MISMATCH;
    if (strict_class && class_hash(rec->origin_op, rec->origin) != class_hash(w->op, w->sh)) return TT_ERR_CLASS_MISMATCH;
    plan->gm = w->view.gm; plan->gn = w->view.gn; plan->gk = w->view.gk; plan->gbatch = w->view.batch;
    switch (w->family) {
        case TT_FAMILY_GEMM_TC: return legalise_gemm(w, rec, mode, plan);
        case TT_FAMILY_DW_SIMT: return legalise_dw(w, rec, mode, plan);
        case TT_FAMILY_ROW_SIMT: return legalise_row(w, rec, mode, plan);
    }
    return TT_ERR_INVALID_ARG;
}

// Layers of one plan on the same activations may share a launch (dense without skip tensor, both operands K-major by TMA,
// reduction by a cluster or in one piece).  Together they have that many times the tiles, and all of their clusters should be
// resident at once: three of 768 -> 768 on 128 rows in tiles of 64 columns are 36 clusters of 4 where 33 fit, and the three that
// are left made the launch take 11 us instead of 5.  A result's sums depend on the splits, their steps and the accumulators, and
// those stay the record's, so that a layer gives the same bits in a group as by itself; which operand is on the 128 rows and how
// many columns a tile has is free.  Where the record's tiles are too many, the narrowest ones of either axis that are resident
// take their place: they move the fewest operand bytes per CTA and are read out fastest.  The 12-layer encoder, 128 tokens: 384 us
// with tiles of 80 columns, 386 with 96, 391 with 128, 470 with each layer by itself, 377 with three splits instead of four, whose
// sums are others; 256 tokens: 523 with 160 columns, 584 with 256 and without a group, 497 with two splits.  No group where no tiles are resident.
void plan_groups(tt_workload* w) {
    const Plan& p = w->plan;
    for (int i = 0; i < 2; ++i) w->group[i].applied = false;
    if (w->op != TT_OP_DENSE || w->sh.has_residual || p.strict || p.g.persistent || p.g.x3 || p.g.two_per_sm || p.info.workspace_bytes != 0 || p.g.a_mode != OPM_TMA || p.g.b_mode != OPM_TMA) return;
    const int resident = kResidentClusters[p.g.split_k], own = p.info.legal.mma_m_axis;
    for (int i = 0; i < 2; ++i) {
        Plan& q = w->group[i];
        if (p.info.grid_x * (i + 2) <= resident) {
            q = p;
            q.applied = true;
            continue;
        }
        for (const int axis : {own, 3 - own}) {
            const int rows = axis == 2 ? w->sh.nn : w->sh.m, cols = axis == 2 ? w->sh.m : w->sh.nn;
            const int columns = resident / ((rows + kHwTileM - 1) / kHwTileM * (i + 2));         // tiles along the columns
            if (columns < 1) continue;
            tt_schedule_record rec = p.info.legal;
            rec.mma_m_axis = axis;
            rec.tile_n = round_up((cols + columns - 1) / columns, 16);
            if (rec.tile_n > 256 || (q.applied && rec.tile_n >= q.g.tile_n)) continue;
            Plan r;
            if (legalise(w, &rec, TT_MODE_LEGALISE, 0, &r) != TT_OK || r.info.grid_x * (i + 2) > resident || r.g.split_k != p.g.split_k ||
                r.g.k_tiles_per_split != p.g.k_tiles_per_split || r.g.tile_k != p.g.tile_k || r.g.n_acc != p.g.n_acc || r.g.two_per_sm || r.info.workspace_bytes != 0) continue;
            q = r;
            q.applied = true;
        }
    }
}

}  // namespace tt

// ---- C ABI (host-only entry points) -------------------------------------------------------------------------

extern "C" {

const char* tt_status_string(tt_status s) {
    switch (s) {
        case TT_OK: return "ok";
        case TT_ERR_INVALID_ARG: return "invalid argument";
        case TT_ERR_INVALID_SCHEDULE: return "schedule invalid for this workload";
        case TT_ERR_CLASS_MISMATCH: return "schedule belongs to another kernel class";
        case TT_ERR_RESOURCE: return "schedule exceeds hardware resources";
        case TT_ERR_NOT_APPLIED: return "no schedule applied";
        case TT_ERR_CUDA: return "CUDA error";
        case TT_ERR_TIMEOUT: return "device wait timed out";
        case TT_ERR_OOM: return "out of device memory";
        case TT_ERR_NOT_IMPLEMENTED: return "not implemented";
        case TT_SKIPPED: return "pair left out by pool sub-sampling";
    }
    return "unknown status";
}

tt_status tt_workload_create(tt_op op, const tt_shapes* sp, tt_workload** out) {
    if (!sp || !out) return TT_ERR_INVALID_ARG;
    *out = nullptr;
    const int fam = family_of(op);
    if (fam < 0) return TT_ERR_INVALID_ARG;
    tt_shapes s = *sp;
    if (s.act < TT_ACT_NONE || s.act > TT_ACT_GELU_ERF) return TT_ERR_INVALID_ARG;
    int P = 0, Q = 0;
    tt_gemm_view v{};
    if (conv_like(op)) {
        if (s.n <= 0 || s.c <= 0 || s.h <= 0 || s.w <= 0 || s.r <= 0 || s.s <= 0 || s.stride_h <= 0 || s.stride_w <= 0 ||
            s.pad_h < 0 || s.pad_w < 0)
            return TT_ERR_INVALID_ARG;
        if (op == TT_OP_CONV2D && s.k <= 0) return TT_ERR_INVALID_ARG;
        if (s.h + 2 * s.pad_h < s.r || s.w + 2 * s.pad_w < s.s) return TT_ERR_INVALID_ARG;
        if (op == TT_OP_DWCONV2D) { s.k = s.c; if (s.has_residual) return TT_ERR_INVALID_ARG; }
        P = (s.h + 2 * s.pad_h - s.r) / s.stride_h + 1;
        Q = (s.w + 2 * s.pad_w - s.s) / s.stride_w + 1;
        s.batch = s.m = s.nn = s.kk = s.trans_b = 0;
        if (op == TT_OP_CONV2D) {
            // implicit GEMM: rows = filters, columns = output pixels, reduction = (c, r, s), one GEMM per image
            v.batch = s.n; v.gm = s.k; v.gn = P * Q; v.gk = s.c * s.r * s.s;
            v.flops = 2.0 * v.batch * v.gm * (double)v.gn * v.gk;
            v.bytes = 4.0 * ((double)s.n * s.c * s.h * s.w + (double)s.k * v.gk + (s.has_bias ? s.k : 0) +
                             (double)s.n * s.k * P * Q * (s.has_residual ? 2 : 1));
        } else {
            v.batch = s.n; v.gm = s.c; v.gn = P * Q; v.gk = s.r * s.s;
            v.flops = 2.0 * s.n * s.c * (double)P * Q * s.r * s.s;
            v.bytes = 4.0 * ((double)s.n * s.c * s.h * s.w + (double)s.c * s.r * s.s + (s.has_bias ? s.c : 0) +
                             (double)s.n * s.c * P * Q);
        }
    } else {
        if (op == TT_OP_DENSE) { s.batch = 1; s.trans_b = 1; }
        if (s.batch <= 0 || s.m <= 0 || s.nn <= 0) return TT_ERR_INVALID_ARG;
        if (op != TT_OP_SOFTMAX && s.kk <= 0) return TT_ERR_INVALID_ARG;
        if (op == TT_OP_SOFTMAX) { s.kk = 0; s.has_bias = 0; s.has_residual = 0; s.act = TT_ACT_NONE; s.trans_b = 0; }
        s.n = s.c = s.h = s.w = s.k = s.r = s.s = s.stride_h = s.stride_w = s.pad_h = s.pad_w = 0;
        v.batch = s.batch; v.gm = s.m; v.gn = s.nn; v.gk = s.kk;
        if (op == TT_OP_SOFTMAX) {
            v.flops = 5.0 * s.batch * (double)s.m * s.nn;
            v.bytes = 8.0 * s.batch * (double)s.m * s.nn;
        } else {
            v.flops = 2.0 * s.batch * (double)s.m * s.nn * s.kk;
            v.bytes = 4.0 * ((double)s.batch * s.m * s.kk + (double)s.batch * s.nn * s.kk + (s.has_bias ? s.nn : 0) +
                             (double)s.batch * s.m * s.nn * (s.has_residual ? 2 : 1));
        }
    }
    if (op != TT_OP_SOFTMAX) s.scale = 0.f;
    s.has_bias = s.has_bias != 0; s.has_residual = s.has_residual != 0;
    tt_workload* w = new (std::nothrow) tt_workload();
    if (!w) return TT_ERR_OOM;
    w->op = op; w->sh = s; w->family = fam; w->P = P; w->Q = Q; w->view = v;
    *out = w;
    return TT_OK;
}

tt_status tt_workload_destroy(tt_workload* w) {
    if (!w) return TT_ERR_INVALID_ARG;
    tt::release_device(w);
    delete w;
    return TT_OK;
}

tt_status tt_workload_key(const tt_workload* w, uint64_t* key) {
    if (!w || !key) return TT_ERR_INVALID_ARG;
    int32_t op = w->op;
    uint64_t h = fnv1a(&op, sizeof op);
    // field by field: padding bytes of the struct never enter the hash
    const tt_shapes& s = w->sh;
    const int32_t f[] = {s.n, s.c, s.h, s.w, s.k, s.r, s.s, s.stride_h, s.stride_w, s.pad_h, s.pad_w,
                         s.batch, s.m, s.nn, s.kk, s.trans_b, s.has_bias, s.has_residual, s.act};
    h = fnv1a(f, sizeof f, h);
    h = fnv1a(&s.scale, sizeof s.scale, h);
    *key = h;
    return TT_OK;
}

tt_status tt_workload_class(const tt_workload* w, uint64_t* cls) {
    if (!w || !cls) return TT_ERR_INVALID_ARG;
    *cls = tt::class_hash(w->op, w->sh);
    return TT_OK;
}

tt_status tt_workload_family(const tt_workload* w, int32_t* family) {
    if (!w || !family) return TT_ERR_INVALID_ARG;
    *family = w->family;
    return TT_OK;
}

tt_status tt_workload_gemm_view(const tt_workload* w, tt_gemm_view* out) {
    if (!w || !out) return TT_ERR_INVALID_ARG;
    *out = w->view;
    return TT_OK;
}

tt_status tt_default_schedule(const tt_workload* w, tt_schedule_record* out) {
    if (!w || !out) return TT_ERR_INVALID_ARG;
    tt_schedule_record r;
    std::memset(&r, 0, sizeof r);
    r.version = TT_RECORD_VERSION;
    r.family = (uint32_t)w->family;
    r.origin_op = w->op;
    r.origin = w->sh;
    // One generic, shape-blind record per family: the counterpart of a compiler's default schedule.
    r.tile_m = 128; r.tile_n = 128; r.tile_k = 32; r.stages = 4; r.split_k = 1; r.raster = 0; r.acc_split = 1;
    r.cta_group = 1;
    r.block_x = 32; r.block_y = 4; r.items_per_thread = 1; r.vec_width = 1; r.unroll = 1; r.threads = 128;
    if (w->family == TT_FAMILY_DW_SIMT) { r.tile_m = 1; r.block_x = 32; r.block_y = 8; r.items_per_thread = 4; r.unroll = 2; }
    if (w->family == TT_FAMILY_ROW_SIMT) { r.block_x = 8; r.block_y = 16; r.vec_width = 4; }
    *out = r;
    return TT_OK;
}

tt_status tt_schedule_check(const tt_workload* w, const tt_schedule_record* rec, int32_t mode, int32_t strict_class,
                            tt_apply_info* info_out) {
    if (!w || !rec) return TT_ERR_INVALID_ARG;
    tt::Plan* p = new (std::nothrow) tt::Plan();
    if (!p) return TT_ERR_OOM;
    tt_status st = tt::legalise(w, rec, mode, strict_class, p);
    if (info_out && (st == TT_OK || st == TT_ERR_RESOURCE)) *info_out = p->info;
    delete p;
    return st;
}

// ---- refinement of a transferred record (named as future work in Section 7): a local search over the fields of a
// record that another model's tuning produced ----
namespace {
struct FieldLadder { int32_t tt_schedule_record::*field; std::vector<int> steps; };   // two steps = a toggle when both differ

const std::vector<FieldLadder>& ladders_of(uint32_t family) {
    static const std::vector<FieldLadder> gemm = {
        {&tt_schedule_record::tile_n, {16, 32, 48, 64, 96, 128, 160, 192, 224, 256}},
        {&tt_schedule_record::tile_k, {8, 16, 32, 64, 96, 128}},
        {&tt_schedule_record::stages, {1, 2, 3, 4, 5, 6, 7, 8}},
        {&tt_schedule_record::split_k, {1, 2, 3, 4, 5, 6, 7, 8, 12, 16, 24, 32}},
        {&tt_schedule_record::raster, {0, 1}},
        {&tt_schedule_record::mma_m_axis, {1, 2}},
        {&tt_schedule_record::slab_tiles, {0, 1, 2, 4, 8}},
        {&tt_schedule_record::acc_split, {1, 2, 4, 8}},
        {&tt_schedule_record::k_order, {0, 1}},
        {&tt_schedule_record::persistent, {0, 1}},
        {&tt_schedule_record::cta_group, {1, 2}},
        {&tt_schedule_record::ctas_per_sm, {1, 2}},
    };
    static const std::vector<FieldLadder> dw = {
        {&tt_schedule_record::tile_m, {1, 2, 4, 8, 16, 32}},
        {&tt_schedule_record::block_y, {1, 2, 4, 7, 8, 14, 16, 28, 56}},
        {&tt_schedule_record::block_x, {8, 16, 28, 32, 56, 64, 112}},
        {&tt_schedule_record::items_per_thread, {1, 2, 4, 8}},
        {&tt_schedule_record::vec_width, {1, 2, 4}},
        {&tt_schedule_record::threads, {32, 64, 128, 256, 512}},
        {&tt_schedule_record::unroll, {0, 1, 2, 4}},
        {&tt_schedule_record::raster, {0, 1}},
        {&tt_schedule_record::stages, {2, 3, 4}},
    };
    static const std::vector<FieldLadder> row = {
        {&tt_schedule_record::block_x, {1, 2, 4, 8, 16, 32}},
        {&tt_schedule_record::block_y, {1, 2, 4, 8, 16}},
        {&tt_schedule_record::vec_width, {1, 2, 4}},
    };
    return family == TT_FAMILY_GEMM_TC ? gemm : (family == TT_FAMILY_DW_SIMT ? dw : row);
}
}  // namespace

tt_status tt_record_neighbours(const tt_workload* w, const tt_schedule_record* rec, tt_schedule_record* out, size_t cap,
                               size_t* n_out) try {
    if (!w || !rec || !n_out || (cap > 0 && !out)) return TT_ERR_INVALID_ARG;
    if (rec->version != TT_RECORD_VERSION || (int)rec->family != (int)w->family) return TT_ERR_INVALID_SCHEDULE;
    // the start in its legalised form: a neighbour that legalises back to it is no neighbour
    tt_apply_info start;
    const tt_status s0 = tt_schedule_check(w, rec, TT_MODE_LEGALISE, 0, &start);
    if (s0 != TT_OK) return s0;
    std::vector<tt_schedule_record> found;
    auto consider = [&](tt_schedule_record r) {
        tt_apply_info info;
        if (tt_schedule_check(w, &r, TT_MODE_LEGALISE, 0, &info) != TT_OK) return;
        tt_schedule_record l = info.legal;
        l.origin_op = rec->origin_op; l.origin = rec->origin;
        tt_schedule_record s = start.legal;
        s.origin_op = rec->origin_op; s.origin = rec->origin;
        if (std::memcmp(&l, &s, sizeof l) == 0) return;
        for (const auto& f : found) if (std::memcmp(&f, &l, sizeof l) == 0) return;
        found.push_back(l);
    };
    for (const FieldLadder& fl : ladders_of(w->family)) {
        const int v = start.legal.*(fl.field);
        int below = INT32_MIN, above = INT32_MAX;       // nearest rungs on either side of v (v need not be a rung)
        for (int step : fl.steps) {
            if (step < v && step > below) below = step;
            if (step > v && step < above) above = step;
        }
        if (below != INT32_MIN) { tt_schedule_record r = start.legal; r.*(fl.field) = below; consider(r); }
        if (above != INT32_MAX) { tt_schedule_record r = start.legal; r.*(fl.field) = above; consider(r); }
    }
    *n_out = found.size();
    if (found.size() > cap) return cap == 0 ? TT_OK : TT_ERR_RESOURCE;     // cap == 0: count only
    for (size_t i = 0; i < found.size(); ++i) out[i] = found[i];
    return TT_OK;
} TT_NO_THROW

tt_status tt_refine_with(const tt_workload* w, const tt_schedule_record* start, tt_time_fn time_us, void* user,
                         int32_t max_rounds, float min_gain, tt_schedule_record* best, float* best_us, float* start_us,
                         int32_t* n_timed) try {
    if (!w || !start || !time_us || !best || !best_us || max_rounds < 0 || !(min_gain >= 0.f)) return TT_ERR_INVALID_ARG;
    tt_apply_info info;
    const tt_status s0 = tt_schedule_check(w, start, TT_MODE_LEGALISE, 0, &info);
    if (s0 != TT_OK) return s0;
    tt_schedule_record cur = info.legal;
    cur.origin_op = start->origin_op; cur.origin = start->origin;
    float cur_us = time_us(user, &cur);
    int timed = 1;
    if (start_us) *start_us = cur_us;
    if (!(cur_us >= 0.f)) { if (n_timed) *n_timed = timed; return TT_ERR_INVALID_SCHEDULE; }
    std::vector<tt_schedule_record> seen{cur};           // never time a record twice
    for (int round = 0; round < max_rounds; ++round) {
        size_t n = 0;
        std::vector<tt_schedule_record> nb(32);
        const tt_status sn = tt_record_neighbours(w, &cur, nb.data(), nb.size(), &n);
        if (sn != TT_OK) return sn;
        int pick = -1;
        float pick_us = cur_us;
        for (size_t i = 0; i < n; ++i) {
            bool dup = false;
            for (const auto& r : seen) if (std::memcmp(&r, &nb[i], sizeof r) == 0) { dup = true; break; }
            if (dup) continue;
            seen.push_back(nb[i]);
            const float us = time_us(user, &nb[i]);
            ++timed;
            if (us >= 0.f && us < pick_us) { pick = (int)i; pick_us = us; }    // ties keep the earlier neighbour
        }
        // move only for a gain of more than min_gain (a fraction of the current time): noise does not walk the record
        if (pick < 0 || !(pick_us < cur_us * (1.f - min_gain))) break;
        cur = nb[(size_t)pick]; cur_us = pick_us;
    }
    *best = cur; *best_us = cur_us;
    if (n_timed) *n_timed = timed;
    return TT_OK;
} TT_NO_THROW

// ---- pool files ---------------------------------------------------------------------------------------------------
namespace {
struct RecField { const char* name; int32_t tt_schedule_record::*field; };
const RecField kRecFields[] = {
    {"tile_m", &tt_schedule_record::tile_m}, {"tile_n", &tt_schedule_record::tile_n}, {"tile_k", &tt_schedule_record::tile_k},
    {"stages", &tt_schedule_record::stages}, {"split_k", &tt_schedule_record::split_k}, {"raster", &tt_schedule_record::raster},
    {"block_x", &tt_schedule_record::block_x}, {"block_y", &tt_schedule_record::block_y},
    {"items_per_thread", &tt_schedule_record::items_per_thread}, {"vec_width", &tt_schedule_record::vec_width},
    {"unroll", &tt_schedule_record::unroll}, {"threads", &tt_schedule_record::threads},
    {"mma_m_axis", &tt_schedule_record::mma_m_axis}, {"slab_tiles", &tt_schedule_record::slab_tiles},
    {"acc_split", &tt_schedule_record::acc_split}, {"k_order", &tt_schedule_record::k_order},
    {"persistent", &tt_schedule_record::persistent}, {"cta_group", &tt_schedule_record::cta_group},
    {"ctas_per_sm", &tt_schedule_record::ctas_per_sm}, {"warp_layout", &tt_schedule_record::warp_layout},
    {"precision", &tt_schedule_record::precision},
};
int32_t* shape_ints(tt_shapes& s, int i) {
    int32_t* f[] = {&s.n, &s.c, &s.h, &s.w, &s.k, &s.r, &s.s, &s.stride_h, &s.stride_w, &s.pad_h, &s.pad_w,
                    &s.batch, &s.m, &s.nn, &s.kk, &s.trans_b, &s.has_bias, &s.has_residual, &s.act};
    return f[i];
}
constexpr int kShapeInts = 19;
}  // namespace

tt_status tt_pool_save(const char* path, const tt_schedule_record* records, const float* us, size_t n) {
    if (!path || (n && !records)) return TT_ERR_INVALID_ARG;
    FILE* f = std::fopen(path, "w");
    if (!f) return TT_ERR_INVALID_ARG;
    std::fprintf(f, "# schedule pool: one record per line, field=value\n");
    for (size_t i = 0; i < n; ++i) {
        tt_schedule_record r = records[i];
        std::fprintf(f, "version=%u family=%u origin_op=%d origin=", r.version, r.family, r.origin_op);
        for (int j = 0; j < kShapeInts; ++j) std::fprintf(f, "%d,", *shape_ints(r.origin, j));
        std::fprintf(f, "%.9g", (double)r.origin.scale);
        for (const RecField& rf : kRecFields) std::fprintf(f, " %s=%d", rf.name, r.*(rf.field));
        std::fprintf(f, " us=%.6g\n", us ? (double)us[i] : -1.0);
    }
    const bool ok = std::fclose(f) == 0;
    return ok ? TT_OK : TT_ERR_INVALID_ARG;
}

tt_status tt_pool_load(const char* path, tt_schedule_record* out, float* us, size_t cap, size_t* n_out) {
    if (!path || !n_out || (cap && !out)) return TT_ERR_INVALID_ARG;
    FILE* f = std::fopen(path, "r");
    if (!f) return TT_ERR_INVALID_ARG;
    size_t n = 0;
    tt_status rc = TT_OK;
    char line[2048];
    while (rc == TT_OK && std::fgets(line, sizeof line, f)) {
        char* p = line;
        while (*p == ' ' || *p == '\t') ++p;
        if (*p == '#' || *p == '\n' || *p == '\r' || *p == 0) continue;
        tt_schedule_record r;
        std::memset(&r, 0, sizeof r);
        float t = -1.f;
        bool have_version = false;
        for (char* tok = std::strtok(p, " \t\r\n"); tok && rc == TT_OK; tok = std::strtok(nullptr, " \t\r\n")) {
            char* eq = std::strchr(tok, '=');
            if (!eq) { rc = TT_ERR_INVALID_ARG; break; }
            *eq = 0;
            auto is = [&](const char* name) { return std::strcmp(tok, name) == 0; };
            const char* val = eq + 1;
            char* end = nullptr;
            if (is("version")) { r.version = (uint32_t)std::strtoul(val, &end, 10); have_version = true; }
            else if (is("family")) r.family = (uint32_t)std::strtoul(val, &end, 10);
            else if (is("origin_op")) r.origin_op = (int32_t)std::strtol(val, &end, 10);
            else if (is("us")) t = std::strtof(val, &end);
            else if (is("origin")) {
                const char* q = val;
                for (int j = 0; j < kShapeInts && rc == TT_OK; ++j) {
                    *shape_ints(r.origin, j) = (int32_t)std::strtol(q, &end, 10);
                    if (end == q || *end != ',') rc = TT_ERR_INVALID_ARG;
                    q = end + 1;
                }
                if (rc == TT_OK) { r.origin.scale = std::strtof(q, &end); if (end == q) rc = TT_ERR_INVALID_ARG; }
            } else {
                bool found = false;
                for (const RecField& rf : kRecFields)
                    if (is(rf.name)) { r.*(rf.field) = (int32_t)std::strtol(val, &end, 10); found = true; break; }
                if (!found) rc = TT_ERR_INVALID_ARG;
            }
            if (rc == TT_OK && (end == val || (end && *end != 0))) rc = TT_ERR_INVALID_ARG;
        }
        if (rc != TT_OK) break;
        if (!have_version || r.version != TT_RECORD_VERSION) { rc = TT_ERR_INVALID_ARG; break; }
        if (n < cap) { out[n] = r; if (us) us[n] = t; }
        ++n;
    }
    std::fclose(f);
    *n_out = n;
    if (rc != TT_OK) return rc;
    return (cap && n > cap) ? TT_ERR_RESOURCE : TT_OK;
}

tt_status tt_pool_subsample(size_t n_pool, size_t count, uint64_t seed, int32_t* idx_out) try {
    if (count > n_pool || (count && !idx_out) || n_pool > 0x7fffffffu) return TT_ERR_INVALID_ARG;
    std::vector<int32_t> perm(n_pool);
    for (size_t i = 0; i < n_pool; ++i) perm[i] = (int32_t)i;
    uint64_t state = seed;
    for (size_t i = 0; i < count; ++i) {
        // splitmix64: advance the state by the golden-ratio increment, then mix
        state += 0x9E3779B97F4A7C15ull;
        uint64_t z = state;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        const size_t j = i + (size_t)(z % (uint64_t)(n_pool - i));
        std::swap(perm[i], perm[j]);
        idx_out[i] = perm[i];
    }
    return TT_OK;
} TT_NO_THROW

tt_status tt_split_check(int64_t extent, const int64_t* factors, size_t n, int32_t reformulate, int32_t* valid) {
    if (!factors || !valid || n == 0 || extent <= 0) return TT_ERR_INVALID_ARG;
    if (reformulate) {
        // Split(N, N/f, f): the outer range adapts to the extent, so only divisibility remains.
        *valid = factors[0] > 0 && extent % factors[0] == 0;
        return TT_OK;
    }
    // Split(N, f0, f1, ...): fixed ranges must traverse the loop exactly.
    __int128 prod = 1;
    for (size_t i = 0; i < n; ++i) {
        if (factors[i] <= 0) { *valid = 0; return TT_OK; }
        prod *= factors[i];
        if (prod > (__int128)extent) { *valid = 0; return TT_OK; }
    }
    *valid = prod == (__int128)extent;
    return TT_OK;
}

tt_status tt_select(const float* times_us, size_t n_wl, size_t n_cols, int32_t* chosen) {
    if (!times_us || !chosen || n_cols == 0) return TT_ERR_INVALID_ARG;
    for (size_t i = 0; i < n_wl; ++i) {
        int best = -1;
        float bt = 0.f;
        for (size_t j = 0; j < n_cols; ++j) {
            const float t = times_us[i * n_cols + j];
            if (!(t >= 0.f) || !std::isfinite(t)) continue;     // negative = invalid pair, NaN never wins
            if (best < 0 || t < bt) { best = (int)j; bt = t; }
        }
        chosen[i] = best;
    }
    return TT_OK;
}

tt_status tt_rank_pools(const double* class_share, size_t n_classes, const int32_t* class_kernels, size_t n_models,
                        double* scores, int32_t* order) try {
    if (!class_share || !class_kernels || !order || n_classes == 0) return TT_ERR_INVALID_ARG;
    std::vector<double> sc(n_models, 0.0);
    for (size_t t = 0; t < n_models; ++t) {
        double s = 0.0;
        for (size_t c = 0; c < n_classes; ++c) {
            const int32_t n = class_kernels[t * n_classes + c];
            if (n < 0 || !(class_share[c] >= 0.0)) return TT_ERR_INVALID_ARG;
            s += class_share[c] * class_share[c] * std::sqrt((double)n);
        }
        sc[t] = s;
    }
    for (size_t t = 0; t < n_models; ++t) order[t] = (int32_t)t;
    std::stable_sort(order, order + n_models, [&](int32_t a, int32_t b) { return sc[a] > sc[b]; });
    if (scores) for (size_t t = 0; t < n_models; ++t) scores[t] = sc[t];
    return TT_OK;
} TT_NO_THROW

tt_status tt_model_latency(const float* times_us, size_t n_wl, size_t n_cols, const int32_t* chosen,
                           const int32_t* use_count, double* latency_us) {
    if (!times_us || !chosen || !use_count || !latency_us) return TT_ERR_INVALID_ARG;
    double sum = 0.0;
    for (size_t i = 0; i < n_wl; ++i) {
        if (chosen[i] < 0 || (size_t)chosen[i] >= n_cols) continue;
        sum += (double)use_count[i] * (double)times_us[i * n_cols + chosen[i]];
    }
    *latency_us = sum;
    return TT_OK;
}

}  // extern "C"
