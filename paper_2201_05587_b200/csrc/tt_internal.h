// Internal declarations shared by the host logic and the CUDA launchers of libtt.
#pragma once
#include <cstdint>
#include <cstddef>
#include <vector>
#include "tt.h"

namespace tt {

constexpr int kHwTileM = 128;           // tcgen05 accumulator rows per CTA (cta_group::1, M = 128)
constexpr int kMaxStages = 8;
constexpr int kSms = 148;               // SMs that the layout rules deal tiles over (a launch is right on any number)
// Clusters of 1..8 CTAs that a B200 holds at once with one CTA per SM (what the driver's occupancy query answers): a cluster keeps to
// one group of SMs, so clusters of 8 leave 28 of the 148 idle and clusters of 7 leave 43.
constexpr int kResidentClusters[9] = {0, 148, 74, 45, 33, 26, 22, 15, 15};
constexpr int kSmemLimit = 232448;      // 227 KB opt-in shared memory per CTA on sm_100
constexpr int kDynSmemLimit = kSmemLimit - 6144;  // what is left for dynamic shared memory beside barriers
constexpr int kRowSmem = 100 * 1024;    // shared memory of a CTA of the ragged softmax, so that two fit an SM
constexpr int kRowRun = 3000;            // ... the bytes of four rows below which a warp may take eight
constexpr int kRaggedMost = 65;         // ... and the values a lane of it keeps in registers at most
constexpr int kCachedMost = 16;         // 16-byte groups a lane of the register-resident softmax keeps at most
// Threads that their registers (both kernels are compiled for it) leave room for: values, or groups, per lane.
constexpr int ragged_threads(int values) { return values <= 17 ? 1024 : values <= 27 ? 768 : values <= 32 ? 640 : 256; }
constexpr int cached_threads(int groups) { return groups <= 8 ? 1024 : 512; }
constexpr int kGatherWarps = 8;
constexpr int kGatherThreads = kGatherWarps * 32;
constexpr int kGemmThreads = 64 + kGatherThreads;   // warp 0 TMA, warp 1 MMA + TMEM, warps 2-9 gather + epilogue

// How one operand of the contraction reaches shared memory.
enum OperandMode : int {
    OPM_TMA = 0,          // K-major 2-D/3-D tensor map, hardware swizzle
    OPM_GATHER_ROWS = 1,  // strided view, lanes walk rows (row stride 1): 16-byte swizzled stores
    OPM_GATHER_K = 2,     // strided view, lanes walk k (k stride 1): 4-byte swizzled stores
    OPM_IM2COL = 3,       // rows are output pixels, k = (c, r, s): expanded from a slab of NCHW input rows
    OPM_RAW = 4,          // k contiguous, rows of any length: groups of four rows by TMA, turned into K-major rows by the warps
    OPM_TMA_MN = 5        // the row index is the contiguous one in memory: [tile_k][32 rows] boxes by TMA, multiplied as
                          // they lie (an MN-major tile)
};

// What a launch of a chained pass brings into the L2 for the launches behind it: weights, which nothing in front of them writes
// (and if something did: the L2 is where memory is coherent).
struct Ahead { const void* p[3]; unsigned bytes[3]; };      // 16-byte aligned, multiples of 16 bytes, the first ones used

// Device-side arguments of the GEMM_TC kernel (plain data, passed by value).
struct GemmArgs {
    int M, N, K, batch;
    int tile_n, tile_k, stages;
    int k_tiles, k_tiles_per_split, split_k;
    int tiles_m, tiles_n, raster;
    int atom_k, n_atoms, swz_mask, row_bytes;
    int a_mode, b_mode;
    const float* a; long long a_rs, a_ks, a_bs; int a_tma_batched;
    const float* b; long long b_rs, b_ks, b_bs; int b_tma_batched;
    int C, H, W, R, S, Q, sh, sw, ph, pw;       // im2col geometry of operand B
    float* y; long long y_ms, y_ns, y_bs;
    const float* bias; int bias_mode;           // 0 none, 1 per row (m), 2 per column (n)
    int act;
    const float* residual;
    float* partial;                             // split-K partial sums [split][batch][M][N]
    unsigned* counters;                         // split-K arrival counters [batch][tiles], zero between launches
    unsigned* status;
    unsigned idesc, tmem_cols;
    unsigned red_off;                           // cluster reduction area: byte offset from the aligned tile base
    int cluster;                                // > 0: split-K over a thread-block cluster of this many CTAs (= split_k)
    int n_acc;                                  // accumulators of tile_n columns each, reduction steps dealt round-robin
    unsigned a_stage_bytes, b_stage_bytes, tx_bytes;
    unsigned ktab_off;                          // im2col k-table: byte offset from the aligned tile base
    int vec_store;                              // bit 0: y rows allow aligned float4 stores; bit 1: so does bias
    // im2col slab: the input rows a CTA's pixels need, staged once in shared memory per chunk of reduction tiles
    unsigned slab_off;                          // byte offset of the first slab buffer from the aligned tile base
    unsigned slab_buf_bytes;                    // bytes per slab buffer (multiple of 16)
    int slab_nbuf;                              // 1: the CTA's whole K range in one chunk; 2: double-buffered chunks
    int slab_tiles;                             // reduction tiles per chunk
    int slab_wp, slab_gap, slab_chpitch;        // row pitch (W + gap), zero gap, channel pitch, in elements
    int slab_in_rows;                           // slab rows per channel (the most a tile can need)
    int slab_rstep;                             // slab rows per output row: min(stride_h, r)
    int slab_vec16;                             // rows copied 16 bytes at a time (W % 4 == 0 and x aligned)
    unsigned magic_wpieces, magic_in_rows, magic_rstep;
    // slab by TMA (rows 16-byte aligned, stride <= filter height): a chunk is one box [box_ch channels][in_rows][W + gap]
    // starting `gap` columns left of the image, so the hardware's zero fill writes the gaps and the rows outside
    int slab_tma;                               // 1: chunks arrive by TMA; 2: as one run of whole channels (images of one tile, pointwise;
                                                // x on 16 bytes); 0: by cp.async from the gather warps
    int slab_box_ch;                            // channels per box
    unsigned slab_box_bytes;
    const int* ktab_dev;                        // per reduction index: byte offset of (c, r, s) inside the slab (absolute channel)
    unsigned long long wait_ns;                 // limit of every bounded wait inside the kernel
    unsigned extra_tx;                          // test facility: bytes added to what the first stage's barrier expects
    int w_operand;                              // 1 / 2: operand A / B is constant (weights the caller promised nobody is
                                                // writing): its first stages are requested before the wait on the kernel in front
    int two_per_sm;                             // the register-capped build, so that two CTAs share an SM
    // operands of ragged rows (OPM_RAW): raw stages behind the pipeline's, A's part in front of B's, four boxes each
    unsigned raw_off, raw_stage_bytes, a_raw_box, b_raw_box;     // (0: the operand has none)
    int a_rows_all, b_rows_all;                 // rows of the whole tensor
    int x3;                                     // error-compensated products: a stage holds [A][B][A lo][B lo], or
    int x3_bufs; unsigned x3_col;               // (> 0) [A][B][B lo], A and its remainders multiplied from this many buffers of 2 * tile_k
                                                // columns of tensor memory, from this one on
    // persistent kernel (record field persistent = 1)
    int persistent, cta_group;
    int total_tiles;                            // tiles_m * tiles_n * batch; tiles_m counts 128 * cta_group rows
    int a_mn, b_mn;                             // the operand's tiles are MN-major
    int b_rows_cta;                             // rows of operand B one CTA loads: tile_n / cta_group
    unsigned epi_off;                           // read-out staging area: byte offset from the aligned tile base
    int epi_warps;                              // read-out warps: 4 or 8
    int epi_late;                               // 4 of them: the other four help with the last tile, over the idle pipeline
    int epi_bufs;                               // 32 x 32 blocks in each read-out warp's ring
    unsigned epi_warp_bytes;                    // ... and its bytes
    int epi_tma;                                // outputs leave by TMA stores (contiguous along the tile's columns)
    int res_tma;                                // the residual comes in by TMA, one block ahead
    int y_tma_batched;                          // the output's tensor map has the batch as its third dimension
};

// What the one-tile kernel does beside its layer in a chained pass: layers of one plan on the same activations share a launch (both
// operands K-major by TMA, no batch; gridDim.z = group, the further members' bias and output here, their weights' tensor maps
// beside the first member's).  An argument of an instantiation of its own: in the one that every call takes it cost 0.1 us a launch
// (7 x 1960 -> 104 3.77 -> 3.85 us between graph nodes, the MobileNetV2-shaped pass of 53 launches 254 -> 258).
struct ChainArgs {
    int group, w_member;                        // layers of the launch; which operand (1 A, 2 B) the weights are
    const float* bias_more[2]; float* y_more[2];
    Ahead ahead;
};

// conv2d by channel blocks and taps over a pixel-major slab (tt_conv_pm_kernel).
constexpr int kPmMaxPlanes = 16;
constexpr unsigned kPmTapBytes = kHwTileM * 32 * 4;         // one tap's filters: 128 x 32 channels
constexpr unsigned kPmEpiBlockBytes = 32 * 36 * 4;          // a staged 32 x 32 block of the read-out
// The taps of one parity class of (row, column) and the sub-image they read: padded input coordinates stride * i + a,
// stride * j + b.  Its first tap is (r0, s0) and reads position (row + f0, column + e0) of the sub-image; the next ones of
// the class follow at (+1, +1).
struct ConvPlane { signed char a, b, f0, e0; unsigned char nr, ns, r0, s0; };
struct ConvPmArgs {
    const float* x; float* y; const float* bias; const float* residual;
    float* partial;                             // clusters: what the CTAs leave to one another
    unsigned* status; unsigned long long wait_ns;
    unsigned extra_tx; int early_filters;
    int M, C, H, W, R, S, P, Q, images, sh, sw, act;
    int blocks;                                 // channel blocks of 32
    int wp, image_pitch;                        // positions per row and per image of the padded-linear numbering
    unsigned magic_wp, magic_image;             // floor(2^32 / divisor)
    int shift_min, slab_lines;                  // the slab of a tile: positions n0 + shift_min .. + slab_lines - 1
    int n_planes; ConvPlane planes[kPmMaxPlanes];
    int tile_n, tiles_m, tiles_n, total_tiles, raster, split, stages, taps_per_stage, slab_bufs;
    unsigned slab_off, slab_bytes, epi_off, idesc, tmem_cols;
};

// The attention of a chained pass in one launch (tt_attention_kernel).
constexpr int kAttnRows = 32;                               // query rows of a CTA
constexpr unsigned kAttnSumLine = 17 * 16;                  // bytes of a row's partial sums, a lane's 16 away from every bank of the next one's
constexpr int kAttnMaps = 3;                                // its tensor maps, beside those of the plans (TmapPair)
struct AttnArgs {
    // (what every launch reads comes first: a launch meets a cold constant cache, line by line)
    int tiles_m, m, n, dv;                      // CTAs per head; query rows and keys of a head, columns of its values
    int n16, n8, n_blocks;                      // keys in 16s, in 8s, in blocks of 32
    int d_atoms, d_steps, v_boxes;              // head size in 32s and 8s, value columns in 32s
    unsigned p_off, k_off, v_off, x_off, idesc_s, idesc_o, tmem_cols, extra_tx;
    int o_col;                                  // the context's accumulators behind the scores'
    float scale;
    int lanes4, lane_groups;                    // the softmax record's lanes of a row / 4; their shares are groups of four values or single ones
    int scores_vec, probs_vec, ctx_vec;         // rows allow 16-byte stores
    float* scores; float* probs; float* ctx;
    Ahead ahead;
    int s_accs, s_per, o_accs, o_per;           // accumulators of the products' records, steps of the reduction to each (0: dealt one by one)
    int smem_bytes;
    unsigned* status; unsigned* status_more[2]; // of the three layers
    unsigned long long wait_ns;
};

struct DwArgs {
    const float* x; const float* w; const float* bias; float* y;
    int N, C, H, W, R, S, P, Q, sh, sw, ph, pw, act;
    int tile_c, tile_h, tile_w, in_h, in_w, items, vec;
    int tiles_c, tiles_h, tiles_w;
    int window_rows;   // > 0: register-window kernel with this many output rows per thread; 0: staged kernel
    int vec_in;        // input rows start on 16-byte boundaries (W % 4 == 0 and x aligned)
    // persistent kernels: tiles of tile_c planes x tile_h x tile_w outputs, whose input lands in `tma_stages` shared-memory buffers:
    // as boxes [tile_c][in_h][box_w] by TMA (zero fill = padding), or (runs) as packed planes or rows of a plane
    int tma_stages;    // > 0 selects them
    int box_w, stage_bytes, total_tiles;   // box width in floats (multiple of 4), bytes per buffer (multiple of 128)
    int wstage_bytes;  // boxes: bytes of the filter-and-bias buffer (multiple of 128)
    int plane_next;    // boxes: lanes after a row of strips continue with the next plane's strips, not with the next strip row
    int step;          // how a CTA's tiles follow each other (dw_walk); set when the record is applied
    int runs;
    int strip_rows;    // runs: strip rows of a plane that are computed at a time
    int units_per_warp, unit_far;   // runs: strip rows side by side in a warp (0: they run on through the warps), their distance (0: 1)
    unsigned* status;  // the workload's status word (bounded waits)
    unsigned long long wait_ns;   // limit of every bounded wait inside the kernel
};

struct RowArgs {
    const float* x; float* y; long long rows; int cols; float scale;
    int lanes_per_row, rows_per_cta, vec;
    int cached;        // > 0: 16-byte groups per lane, kept in registers (x and y on 16-byte boundaries)
    int warps, chunk;  // > 0: ragged rows through shared memory, `chunk` rows a warp (x and y on 16-byte boundaries)
    unsigned* status; unsigned long long wait_ns;   // the workload's status word and wait limit
};

// Host-side plan of an applied record.
struct Plan {
    bool applied = false;
    bool strict = false;              // the record is to run as written
    tt_apply_info info{};
    // GEMM lowering
    int gm = 0, gn = 0, gk = 0, gbatch = 1;
    bool swap_ab = false;
    int a_tensor = 0, b_tensor = 1;   // which caller tensor feeds operand A / B: 0 = x, 1 = w
    GemmArgs g{};
    long long partial_bytes = 0;      // counters start here inside the workspace
    int run_smem = 0;                 // one-tile GEMM: shared memory of a launch (the ring may be deeper than the record's)
    bool repack = false;              // tap-major convolution: pm applies, filters are re-packed into the workspace
    ConvPmArgs pm{};
    DwArgs dw{};
    RowArgs row{};
};

constexpr int kMaxEpiBufs = 3;
constexpr unsigned kLateRingBytes = 8192;   // two 32 x 32 blocks per warp

// The tensor maps of a launch, cached by the plan and the pointers they were made for.
struct TmapPair {
    int plan;                               // 0: the applied one, 1 and 2: of a group of two and three layers, kAttnMaps
    const void* a_ptr; const void* b_ptr;
    const void* y_ptr; const void* r_ptr;   // persistent form with TMA read-out; null elsewhere
    alignas(64) unsigned char y[128];
    alignas(64) unsigned char r[128];
    alignas(64) unsigned char a[128];
    alignas(64) unsigned char b[128];
    alignas(64) unsigned char x[128];   // conv2d: the image as a (W, H, C, N) tensor, for the slab
};

}  // namespace tt

// Nothing throws across the C ABI: a function whose containers may run out of memory is a try block that ends in this.
#define TT_NO_THROW catch (...) { return TT_ERR_OOM; }

struct tt_workload {
    tt_op op;
    tt_shapes sh;
    int family;
    int P, Q;                    // conv output size
    tt_gemm_view view;
    tt::Plan plan;
    tt::Plan group[2];           // the plan of two and of three layers in one launch of a chained pass (applied: there is one)
    void* workspace = nullptr;   // device: split-K partials
    int* ktab_dev = nullptr;     // device: conv2d reduction-index table of the applied record
    size_t ktab_bytes = 0;
    size_t workspace_bytes = 0;
    void* exchange = nullptr;    // device: what the CTAs of a tap-major convolution's clusters leave to one another
    size_t exchange_bytes = 0;
    unsigned* status_word = nullptr;  // device
    unsigned long long wait_ns = 1000000000ull;   // one second per wait inside a kernel, then the kernel gives up
    unsigned extra_tx = 0;            // test facility (tt_workload_test_stall)
    bool constant_weights = false;    // the caller's promise of tt_workload_set_constant_weights
    // tap-major convolution: the workspace holds the re-packed filters of ...
    const void* repacked_for = nullptr;   // ... these weights (null: of none that the next call may take for its own),
    unsigned long long repacked_in = 0;   // put there by a call that ran (0) or only inside this capture
    bool captured_read = false;           // a captured pass reads them as they are now: they are not to be overwritten
    bool captured_fill = false;           // a captured pass fills the workspace itself: what else is put there does not last
    std::vector<void*> kept;              // workspaces that captured passes still read, until the next apply
    // device staging buffers of tt_run_host
    void* hbuf[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    size_t hbytes[5] = {0, 0, 0, 0, 0};
    size_t tmap_next = 0;             // where the next look-up in tmaps begins
    std::vector<tt::TmapPair> tmaps;  // tensor maps encoded so far for the applied record, by operand pointers
};

namespace tt {
// host logic (tt_host.cpp)
tt_status legalise(const tt_workload* w, const tt_schedule_record* rec, int mode, int strict_class, Plan* plan);
void plan_groups(tt_workload* w);                               // from the applied plan
uint64_t class_hash(int op, const tt_shapes& s);
size_t tensor_elems(const tt_workload* w, int which);   // 0 x, 1 w, 2 bias, 3 residual, 4 y
// device side (launch.cu)
tt_status bind_device(tt_workload* w);                          // workspace + status word
tt_status launch(tt_workload* w, const tt_tensors* t, void* stream);
void release_device(tt_workload* w);
}  // namespace tt
