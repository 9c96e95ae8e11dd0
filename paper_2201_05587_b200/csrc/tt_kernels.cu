// Device code of libtt for sm_100a: the schedule-parameterised kernel families.
//
//   GEMM_TC  tcgen05.mma kind::tf32, accumulator in tensor memory, `stages`-deep mbarrier pipeline.  Operands reach
//            shared memory by TMA (K-major tensors, and row-contiguous ones that are multiplied MN-major), by expansion
//            from a slab of input rows that TMA (or cp.async) staged once per CTA (im2col of NCHW activations), or by
//            gathers (strided views).  Bias/activation are
//            fused into the accumulator read-out.  Split-K of 2..8 runs as a thread-block cluster that reduces
//            through distributed shared memory; more splits go through a workspace and the last-arriving CTA adds
//            them up, both in fixed split order.  Launched with programmatic stream serialization.  Built twice:
//            with all registers (one CTA per SM) and capped so that two CTAs share an SM on large grids.
//   DW_SIMT  depthwise convolution, fp32 FMA: persistent kernels whose tiles' inputs arrive as TMA boxes (3x3 / 5x5,
//            16-byte image rows) or as packed runs (other rows), a register-window kernel (3x3 / 5x5) and a shared-memory staged kernel.
//   ROW_SIMT row softmax with sub-warp shuffles, register-resident rows when they fit, whole groups of ragged rows by bulk copies.
//
// Every tile size, the pipeline depth, split-K and the tile order are run-time values taken from the applied
// schedule record, so applying a record never recompiles anything.
//
// Every wait on an mbarrier is bounded: when it expires the CTA records TT_ERR_TIMEOUT in the workload's status
// word, all roles leave their loops, tensor memory is released and the kernel returns normally.
#include <cuda_runtime.h>
#include <cuda.h>
#include <cstdint>
#include <cstring>
#include <algorithm>
#include <type_traits>
#include <utility>
#include "tt_ptx.cuh"

namespace tt {

// ------------------------------------------------------------------------------------------------------------
// Operand producers that do not go through TMA.
//
// im2col operand of conv2d (rows = output pixels, k = (c, r, s), gathered from an NCHW image).  The input rows a
// CTA's pixels need are staged ONCE per chunk of reduction tiles in a shared-memory slab by cp.async: per
// channel, the rows [ih_lo, ih_lo + in_rows) one after the other, each followed by `gap` zeros, so that the
// left/right padding of a row and rows outside the image read as zero without any test.  A pipeline stage is
// then expanded from the slab: element (pixel, k) sits at rowoff[pixel] + koff[k], two table look-ups, and a
// lane assembles four consecutive k of its pixel and writes one 16-byte chunk of the swizzled K-major tile.
// Global memory is read once per CTA (not once per filter tap), and no load of the main loop waits on DRAM or L2.
//
// Strided views (the NN operand of batch_matmul) and K-contiguous operands with K % 4 != 0 are gathered from
// global memory directly: the 8 gather warps form 1, 2 or 4 groups, group g fills stages g, g + groups, ...
// ------------------------------------------------------------------------------------------------------------
// Split-K over a cluster.  The output tile is cut into one band per CTA, along the direction in which the output is
// NOT contiguous (bands of rows when outputs are contiguous along columns, bands of columns otherwise).  Every CTA
// first writes its partial tile into its own shared memory (the pipeline buffers, idle by then) in the layout of the
// reduction area, so that a band is one contiguous run of bytes; one thread per peer then sends that peer's band with
// a single bulk copy (cp.async.bulk, shared::cta -> shared::cluster) into the peer's reduction area, which is not part
// of the pipeline buffers (a fast peer cannot disturb a slower one's main loop).  The copy reports its bytes to a
// barrier of the receiving CTA, which expects the bands of all other splits: a CTA starts adding as soon as ITS bands
// have landed, in split order, its own band read from its own staging copy.  Area layout, per source split (the
// CTA's own split has no slot):
//   bands of rows:    [row in band][col], pitch tile_n + 4 floats;   bands of columns: [col in band][row], pitch 128.
constexpr int kRedColPitch = kHwTileM;
// All gather threads meet and learn whether every one of them is still healthy (named barrier 1).
__device__ __forceinline__ bool gather_vote(bool ok) {
    uint32_t all;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "bar.red.and.pred p, 1, %2, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(all) : "r"((uint32_t)ok), "n"(kGatherThreads) : "memory");
    return all != 0u;
}

// n / d for the small ranges of the slab loader: magic = ceil(2^32 / d) is exact while n * d < 2^32; d == 1 has magic 0.
__device__ __forceinline__ int small_div(int n, unsigned magic) { return magic ? (int)__umulhi((unsigned)n, magic) : n; }

// Stage the input rows of channels [c_first, c_first + nch) that this CTA's pixels need into one slab buffer.
// Pieces (16 bytes when the rows allow it, else 4) are dealt round-robin to the gather threads; rows outside the
// image or beyond the CTA's own range are skipped and keep the zeros written at kernel start.
__device__ __forceinline__ void slab_load_chunk(const GemmArgs& g, const float* __restrict__ img, uint32_t buf, int c_first,
                                                int nch, int ih_lo, int in_rows_cta, bool vec16, int gt) {
    const int wpieces = vec16 ? g.W >> 2 : g.W;
    const bool use_magic = vec16 == (g.slab_vec16 != 0);  // the host's magic number is for its own piece width
    if (wpieces <= 16) {
        // short rows (small images): one thread copies a whole row, so the row's address arithmetic is done once
        const int n_rows = nch * g.slab_in_rows;
        for (int row = gt; row < n_rows; row += kGatherThreads) {
            const int cl = small_div(row, g.magic_in_rows);
            const int rl = row - cl * g.slab_in_rows;
            int ih = ih_lo + rl;
            if (g.sh > g.R) {
                const int po = small_div(rl, g.magic_rstep);
                ih = ih_lo + po * g.sh + (rl - po * g.slab_rstep);
            }
            if (rl >= in_rows_cta || (unsigned)ih >= (unsigned)g.H) continue;
            const float* src = img + ((long long)(c_first + cl) * g.H + ih) * g.W;
            const uint32_t dst = buf + 4u * (uint32_t)(cl * g.slab_chpitch + rl * g.slab_wp + g.slab_gap);
            if (vec16) {
                for (int pc = 0; pc < wpieces; ++pc) cp_async_16(dst + 16u * (uint32_t)pc, src + 4 * pc);
            } else {
                for (int pc = 0; pc < wpieces; ++pc) cp_async_4(dst + 4u * (uint32_t)pc, src + pc);
            }
        }
        return;
    }
    const int total = nch * g.slab_in_rows * wpieces;
    for (int idx = gt; idx < total; idx += kGatherThreads) {
        const int t1 = use_magic ? small_div(idx, g.magic_wpieces) : idx / wpieces;
        const int pc = idx - t1 * wpieces;
        const int cl = small_div(t1, g.magic_in_rows);
        const int rl = t1 - cl * g.slab_in_rows;
        // slab row -> image row: consecutive rows when stride <= filter height, else r rows per output row
        int ih = ih_lo + rl;
        if (g.sh > g.R) {
            const int po = small_div(rl, g.magic_rstep);
            ih = ih_lo + po * g.sh + (rl - po * g.slab_rstep);
        }
        if (rl >= in_rows_cta || (unsigned)ih >= (unsigned)g.H) continue;
        const int col = vec16 ? pc << 2 : pc;
        const float* src = img + ((long long)(c_first + cl) * g.H + ih) * g.W + col;
        const uint32_t dst = buf + 4u * (uint32_t)(cl * g.slab_chpitch + rl * g.slab_wp + g.slab_gap + col);
        if (vec16) cp_async_16(dst, src); else cp_async_4(dst, src);
    }
}

// The chunks c0, c0 + step, ... of one tile row per lane, KB at a time, in three rounds without a branch between
// loads: all table entries, all slab values, then the stores (chunks past the tile re-read the last one and are
// not stored).
template <int KB>
__device__ __forceinline__ void expand_chunks(int c0, int step, int n_ch, uint32_t origin, uint32_t ktab_smem, uint32_t dst_row,
                                              uint32_t swz, int atom_shift, int atom_k, uint32_t atom_bytes, bool in_tile) {
    for (; c0 < n_ch; c0 += step * KB) {
        uint4 e[KB];
        float val[KB][4];
#pragma unroll
        for (int b = 0; b < KB; ++b)
            e[b] = ld_shared_v4u(ktab_smem + 16u * (uint32_t)min(c0 + b * step, n_ch - 1));   // same address in every lane
#pragma unroll
        for (int b = 0; b < KB; ++b) {
            val[b][0] = ld_shared_f32(origin + e[b].x);
            val[b][1] = ld_shared_f32(origin + e[b].y);
            val[b][2] = ld_shared_f32(origin + e[b].z);
            val[b][3] = ld_shared_f32(origin + e[b].w);
        }
#pragma unroll
        for (int b = 0; b < KB; ++b) {
            const int ci = c0 + b * step;
            if (ci < n_ch && in_tile) {
                const int kk = ci << 2;
                st_shared_v4(dst_row + (uint32_t)(kk >> atom_shift) * atom_bytes + ((uint32_t)((kk & (atom_k - 1)) << 2) ^ swz),
                             val[b][0], val[b][1], val[b][2], val[b][3]);
            }
        }
    }
}

// What a gather thread needs to expand its share of any stage, worked out once per kernel: which tile row it
// serves, where that row's window starts in a slab channel, where the row lands in a K-major tile, which
// chunks of four reduction indices it takes.
struct ExpandPlan {
    bool fast, in_tile;          // fast: 1, 2, 4 or 8 row blocks, so a warp keeps one row block for the whole kernel
    uint32_t row_origin;         // byte offset of the row's window origin inside a slab channel
    uint32_t dst_row, swz;       // byte offset of the row inside a tile; its swizzle term
    int c0, step, n_ch, mine;    // first chunk, chunk stride, chunks per tile, chunks this warp takes
    int atom_shift, atom_k;
    uint32_t atom_bytes;
};

__device__ __forceinline__ ExpandPlan make_expand_plan(int rows, uint32_t rowoff_smem, int tile_k, int atom_k, int row_bytes,
                                                       int swz_mask, int gw, int lane) {
    ExpandPlan p;
    const int n_rb = (rows + 31) >> 5;
    p.fast = (kGatherWarps % n_rb) == 0;
    p.atom_shift = atom_k == 32 ? 5 : (atom_k == 16 ? 4 : 3);
    p.atom_k = atom_k;
    p.atom_bytes = (uint32_t)rows * (uint32_t)row_bytes;
    p.n_ch = tile_k >> 2;
    const int shift = row_bytes == 128 ? 0 : (row_bytes == 64 ? 1 : 2);
    const int rb = p.fast ? gw % n_rb : 0;
    p.step = p.fast ? kGatherWarps / n_rb : 1;
    p.c0 = p.fast ? gw / n_rb : 0;
    p.mine = (p.n_ch - p.c0 + p.step - 1) / p.step;
    const int row = rb * 32 + lane;
    p.in_tile = row < rows;
    p.row_origin = ld_shared_u32(rowoff_smem + 4u * (uint32_t)(p.in_tile ? row : rows - 1));
    p.dst_row = (uint32_t)row * (uint32_t)row_bytes;
    p.swz = (uint32_t)((row >> shift) & swz_mask) << 4;
    return p;
}

// Expand one pipeline stage of the im2col operand from the slab.  A warp takes (32-row block, 4-wide k chunk)
// tasks gw, gw + 8, ...; the loads of four tasks are issued before the first store.
// rowoff_smem: per tile row, the byte offset of its pixel's window origin inside a channel of the slab;
// ktab_smem: per reduction index of this tile, the byte offset of (channel, tap) relative to that origin.
__device__ __forceinline__ void expand_stage(const ExpandPlan& xp, uint32_t tile_smem, int rows, uint32_t slab, uint32_t rowoff_smem,
                                             uint32_t ktab_smem, int tile_k, int atom_k, int row_bytes, int swz_mask,
                                             int gw, int lane) {
    if (xp.fast) {
        const uint32_t origin = slab + xp.row_origin, dst_row = tile_smem + xp.dst_row;
        if (xp.mine <= 2) expand_chunks<2>(xp.c0, xp.step, xp.n_ch, origin, ktab_smem, dst_row, xp.swz, xp.atom_shift, xp.atom_k, xp.atom_bytes, xp.in_tile);
        else if (xp.mine <= 4) expand_chunks<4>(xp.c0, xp.step, xp.n_ch, origin, ktab_smem, dst_row, xp.swz, xp.atom_shift, xp.atom_k, xp.atom_bytes, xp.in_tile);
        else expand_chunks<8>(xp.c0, xp.step, xp.n_ch, origin, ktab_smem, dst_row, xp.swz, xp.atom_shift, xp.atom_k, xp.atom_bytes, xp.in_tile);
        return;
    }
    const int atom_shift = atom_k == 32 ? 5 : (atom_k == 16 ? 4 : 3);
    const int shift = row_bytes == 128 ? 0 : (row_bytes == 64 ? 1 : 2);
    const uint32_t atom_bytes = (uint32_t)rows * (uint32_t)row_bytes;
    const int n_rb = (rows + 31) >> 5;
    const int n_tasks = n_rb * (tile_k >> 2);
    const uint32_t inv_rb = (65536u + (uint32_t)n_rb - 1u) / (uint32_t)n_rb;     // t / n_rb == (t * inv_rb) >> 16 for small t
    constexpr int kBatch = 4;
    for (int t0 = gw; t0 < n_tasks; t0 += kGatherWarps * kBatch) {
        float val[kBatch][4];
        uint32_t dst[kBatch];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int t = t0 + b * kGatherWarps;
            const bool live = t < n_tasks;               // warp-uniform
            const int tt = live ? t : 0;
            const int ci = (int)(((uint32_t)tt * inv_rb) >> 16);
            const int rb = tt - ci * n_rb;
            const int kk = ci << 2;
            const int row = rb * 32 + lane;
            const bool in_tile = live && row < rows;
            dst[b] = in_tile ? tile_smem + (uint32_t)(kk >> atom_shift) * atom_bytes + (uint32_t)row * (uint32_t)row_bytes +
                                   ((uint32_t)((kk & (atom_k - 1)) << 2) ^ ((uint32_t)((row >> shift) & swz_mask) << 4))
                             : 0xffffffffu;
            const uint32_t origin = slab + ld_shared_u32(rowoff_smem + 4u * (uint32_t)(row < rows ? row : rows - 1));
            const uint4 e = ld_shared_v4u(ktab_smem + 16u * (uint32_t)ci);       // same address in every lane
            val[b][0] = ld_shared_f32(origin + e.x);
            val[b][1] = ld_shared_f32(origin + e.y);
            val[b][2] = ld_shared_f32(origin + e.z);
            val[b][3] = ld_shared_f32(origin + e.w);
        }
#pragma unroll
        for (int b = 0; b < kBatch; ++b)
            if (dst[b] != 0xffffffffu) st_shared_v4(dst[b], val[b][0], val[b][1], val[b][2], val[b][3]);
    }
}

// One stage of a strided view whose rows are contiguous across lanes (unit row stride): lanes walk rows
// (coalesced loads), each lane assembles four consecutive reduction indices of its row in registers and writes
// one 16-byte chunk into the swizzled K-major tile.  Loads of eight tasks are issued before the first store.
__device__ __forceinline__ void gather_rows_stage(uint32_t tile_smem, int rows, const float* __restrict__ src,
                                                  long long rs, long long ks, int row0, int row_extent, int k0, int K,
                                                  int tile_k, int atom_k, int row_bytes, int swz_mask, int wig, int wpg,
                                                  int lane) {
    const int atom_shift = atom_k == 32 ? 5 : (atom_k == 16 ? 4 : 3);
    const int shift = row_bytes == 128 ? 0 : (row_bytes == 64 ? 1 : 2);
    const uint32_t atom_bytes = (uint32_t)rows * (uint32_t)row_bytes;
    const int n_rb = (rows + 31) >> 5;
    const int n_ch = tile_k >> 2;
    const int my_ch = (n_ch - wig + wpg - 1) / wpg;      // chunks wig, wig + wpg, ... belong to this warp
    const int n_tasks = my_ch > 0 ? my_ch * n_rb : 0;    // task = (chunk, 32-row block)
    const uint32_t inv_rb = (65536u + (uint32_t)n_rb - 1u) / (uint32_t)n_rb;
    constexpr int kBatch = 8;
    for (int t0 = 0; t0 < n_tasks; t0 += kBatch) {
        float val[kBatch][4];
        uint32_t dst[kBatch];
#pragma unroll
        for (int b = 0; b < kBatch; ++b) {
            const int t = t0 + b;
            const bool live = t < n_tasks;               // warp-uniform
            const int tt = live ? t : 0;
            const int ci = (int)(((uint32_t)tt * inv_rb) >> 16);
            const int rb = tt - ci * n_rb;
            const int kk = (wig + ci * wpg) * 4;
            const int row = rb * 32 + lane;
            const bool in_tile = live && row < rows;
            dst[b] = in_tile ? tile_smem + (uint32_t)(kk >> atom_shift) * atom_bytes + (uint32_t)row * (uint32_t)row_bytes +
                                   ((uint32_t)((kk & (atom_k - 1)) << 2) ^ ((uint32_t)((row >> shift) & swz_mask) << 4))
                             : 0xffffffffu;
            const int grow = row0 + row;
            const bool rv = in_tile && grow < row_extent;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int k = k0 + kk + j;
                val[b][j] = (rv && k < K) ? __ldg(src + (long long)grow * rs + (long long)k * ks) : 0.f;
            }
        }
#pragma unroll
        for (int b = 0; b < kBatch; ++b)
            if (dst[b] != 0xffffffffu) st_shared_v4(dst[b], val[b][0], val[b][1], val[b][2], val[b][3]);
    }
}

// One stage of an operand whose reduction index is contiguous in memory but cannot go through TMA (K % 4 != 0):
// a warp takes rows, its lanes walk k; 4-byte stores stay inside one swizzled row (conflict-free).
__device__ __forceinline__ void gather_k_stage(uint32_t tile_smem, int rows, const float* __restrict__ src, long long rs,
                                               long long ks, int row0, int row_extent, int k0, int K, int tile_k,
                                               int atom_k, int row_bytes, int swz_mask, int wig, int wpg, int lane) {
    const int atom_shift = atom_k == 32 ? 5 : (atom_k == 16 ? 4 : 3);
    const int shift = row_bytes == 128 ? 0 : (row_bytes == 64 ? 1 : 2);
    const uint32_t atom_bytes = (uint32_t)rows * (uint32_t)row_bytes;
    for (int kk = lane; kk < tile_k; kk += 32) {
        const int k = k0 + kk;
        const uint32_t kterm = (uint32_t)(kk >> atom_shift) * atom_bytes;
        const uint32_t kb = (uint32_t)((kk & (atom_k - 1)) << 2);
        for (int r0 = wig; r0 < rows; r0 += wpg * 4) {
            float val[4];
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int r = r0 + b * wpg;
                const int grow = row0 + r;
                val[b] = (r < rows && grow < row_extent && k < K) ? __ldg(src + (long long)grow * rs + (long long)k * ks) : 0.f;
            }
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int r = r0 + b * wpg;
                if (r < rows)
                    st_shared_f32(tile_smem + kterm + (uint32_t)r * (uint32_t)row_bytes + (kb ^ ((uint32_t)((r >> shift) & swz_mask) << 4)), val[b]);
            }
        }
    }
}

// One stage of an operand of ragged rows (OPM_RAW).  Four rows of K floats are a multiple of 16 bytes, so the tensor in groups of
// four rows is a matrix that TMA can read: row 4 l + c lies in line l from column c K on.  Its box starts at the 16-byte boundary in
// front of that, the same distance s for every fourth row, and is one 16-byte group wider than the tile.
// Eight lanes (fewer where the tile has fewer columns) take a row, each four neighbouring values of it: they read them one by one,
// s floats further on than the box begins, and write them as one 16-byte group of the swizzled K-major row.  The lanes of a quarter
// warp fill a whole 128-byte line, and rows side by side differ in s where K is odd: neither side meets a bank twice.  What a whole
// tile does not need (the end of the rows; rows behind the last group of four, which come from memory directly) is an instantiation
// of its own.  Bound by the instructions of eight warps beside the products: 2048 x 2048 over 1023 takes 62 us, 41 without this step,
// 25 over 1024.  Gathered value by value from memory before, with whole tunings of a pool: 1001 x 777 over 1003 143 -> 43 us, 4000 x 3001 over
// 2047 928 -> 384, 300 heads of 506 x 64 over 506 281 -> 133, 36 of 297 x 64 over 297 41 -> 19.
struct RealignArgs {
    uint32_t tile, raw, box_bytes;
    int rows, row_first, rows_all, k0, K, tile_k, atom_k, row_bytes, swz_mask, wig, wpg;
};
template <bool EDGE>
__device__ __forceinline__ void realign_rows(const RealignArgs& r, const float* __restrict__ src, int lane) {
    const int per_row = r.atom_k >> 2, shift = r.atom_k == 32 ? 3 : (r.atom_k == 16 ? 2 : 1);          // lanes of a row
    const int chunk = lane & (per_row - 1), ri = lane >> shift, step = 32 >> shift;       // rows at a time: 4, 8 or 16
    const int swz_shift = r.row_bytes == 128 ? 0 : (r.row_bytes == 64 ? 1 : 2), j = ri & 3;
    const int s = (((r.row_first + j) & 3) * r.K) & 3;
    const uint32_t pitch = 4u * (uint32_t)(r.tile_k + 4), atom_bytes = (uint32_t)(r.rows * r.row_bytes);
    uint32_t from0 = r.raw + (uint32_t)j * r.box_bytes + (uint32_t)(ri >> 2) * pitch + 16u * (uint32_t)chunk + 4u * (uint32_t)s, to0 = r.tile;
#pragma unroll 1
    for (int k = 0; k < r.tile_k; k += r.atom_k, from0 += (uint32_t)r.row_bytes, to0 += atom_bytes) {
        constexpr int kBatch = 4;
#pragma unroll 1
        for (int r0 = r.wig * step; r0 < r.rows; r0 += r.wpg * step * kBatch) {
            float v[kBatch][4];
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const int row0 = r0 + b * r.wpg * step;
                if (row0 >= r.rows) break;               // (warp-uniform)
                const uint32_t from = from0 + (uint32_t)(row0 >> 2) * pitch;
#pragma unroll
                for (int e = 0; e < 4; ++e) v[b][e] = ld_shared_f32(from + 4u * (uint32_t)e);
                if (EDGE) {
                    const int row = r.row_first + row0 + ri, k_here = r.k0 + k + 4 * chunk;
                    const bool direct = row >= (r.rows_all & ~3) && row < r.rows_all;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        // (what lies behind a row's end in its box is the next row)
                        if (k_here + e >= r.K) v[b][e] = 0.f;
                        else if (direct) v[b][e] = __ldg(src + (long long)row * r.K + k_here + e);
                    }
                }
            }
#pragma unroll
            for (int b = 0; b < kBatch; ++b) {
                const int row = r0 + b * r.wpg * step + ri;
                if (row >= r.rows) break;
                st_shared_v4(to0 + (uint32_t)(row * r.row_bytes) + ((uint32_t)(chunk ^ ((row >> swz_shift) & r.swz_mask)) << 4), v[b][0], v[b][1], v[b][2], v[b][3]);
            }
        }
    }
}
__device__ __forceinline__ void realign_stage(const RealignArgs& r, const float* __restrict__ src, int lane) {
    if (r.k0 + r.tile_k > r.K || r.row_first + r.rows > (r.rows_all & ~3)) realign_rows<true>(r, src, lane);
    else realign_rows<false>(r, src, lane);
}
// ... and the request of its four boxes (one thread).
__device__ __forceinline__ void load_raw_boxes(uint32_t dst, const void* tmap, uint32_t bar, uint32_t box_bytes, int row_first, int K, int k0) {
#pragma unroll 1
    for (int j = 0; j < 4; ++j, dst += box_bytes)
        tma_load_3d(dst, tmap, bar, ((((row_first + j) & 3) * K) & ~3) + k0, (row_first + j) >> 2, 0);
}

__device__ __forceinline__ void gather_stage(int mode, uint32_t tile_smem, int rows, const float* __restrict__ src,
                                             long long rs, long long ks, int row0, int row_extent, int k0, int K,
                                             int tile_k, int atom_k, int row_bytes, int swz_mask, int wig, int wpg,
                                             int lane) {
    if (mode == OPM_GATHER_ROWS)
        gather_rows_stage(tile_smem, rows, src, rs, ks, row0, row_extent, k0, K, tile_k, atom_k, row_bytes, swz_mask, wig, wpg, lane);
    else
        gather_k_stage(tile_smem, rows, src, rs, ks, row0, row_extent, k0, K, tile_k, atom_k, row_bytes, swz_mask, wig, wpg, lane);
}

// ------------------------------------------------------------------------------------------------------------
// Epilogue helpers
// ------------------------------------------------------------------------------------------------------------
constexpr int kStagePitch = 36;                          // floats per staged row: 16-byte accesses stay conflict-free
constexpr int kStageBytesPerWarp = 32 * kStagePitch * 4;

// ReLU, ReLU6 and "none" are one clamp with per-kernel bounds (no branch per element); GELU is a separate path.
struct EpiArgs {
    float* ybase; const float* rbase; long long y_ms, y_ns; int M; float lo, hi; bool gelu, vec;
};

__device__ __forceinline__ float finish_one(float v, const EpiArgs& e) {
    if (e.gelu) return gelu_erf(v);              // uniform per kernel
    return fminf(fmaxf(v, e.lo), e.hi);
}

// Store one 32-row x 32-column block of pre-activation values (bias already added) whose rows are this warp's
// lanes.  Row-major outputs (y_ns == 1) are transposed through the warp's shared-memory staging area so that
// eight lanes write one 128-byte row segment; otherwise lanes are contiguous in memory and each column is one
// coalesced store.  FULL: all 32 rows and 32 columns exist and 16-byte accesses are aligned.
// POST: a residual is added, so the activation runs here, after it; otherwise the values arrive activated.
template <bool FULL, bool POST>
__device__ __forceinline__ void epilogue_block(float (&v)[32], const EpiArgs& e, int m_first, int nb, int cnt,
                                               uint32_t stg, int lane, bool transposed) {
    if (transposed) {
#pragma unroll
        for (int j = 0; j < 32; j += 4) st_shared_v4(stg + (uint32_t)(lane * kStagePitch + j) * 4u, v[j], v[j + 1], v[j + 2], v[j + 3]);
        __syncwarp();
        const int cc = (lane & 7) * 4;
#pragma unroll
        for (int itr = 0; itr < 8; ++itr) {
            const int rr = itr * 4 + (lane >> 3);
            const int m = m_first + rr;
            float4 t;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(t.x), "=f"(t.y), "=f"(t.z), "=f"(t.w)
                         : "r"(stg + (uint32_t)(rr * kStagePitch + cc) * 4u));
            const long long o = (long long)m * e.y_ms + nb + cc;
            if (FULL) {
                if (POST) {
                    const float4 r4 = __ldg(reinterpret_cast<const float4*>(e.rbase + o));
                    t.x = finish_one(t.x + r4.x, e); t.y = finish_one(t.y + r4.y, e);
                    t.z = finish_one(t.z + r4.z, e); t.w = finish_one(t.w + r4.w, e);
                }
                *reinterpret_cast<float4*>(e.ybase + o) = t;
            } else {
                const float tv[4] = {t.x, t.y, t.z, t.w};
                const bool row_ok = m < e.M;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const bool ok = row_ok && cc + j < cnt;
                    float out = tv[j];
                    if (POST) out = finish_one(out + (ok ? __ldg(e.rbase + o + j) : 0.f), e);
                    if (ok) e.ybase[o + j] = out;
                }
            }
        }
        __syncwarp();
    } else {
        const int m = m_first + lane;
        const bool row_ok = FULL || m < e.M;
        long long o = (long long)m * e.y_ms + (long long)nb * e.y_ns;
#pragma unroll
        for (int j = 0; j < 32; ++j, o += e.y_ns) {
            const bool ok = row_ok && (FULL || j < cnt);
            float out = v[j];
            if (POST) out = finish_one(out + (ok ? __ldg(e.rbase + o) : 0.f), e);
            if (ok) e.ybase[o] = out;
        }
    }
}

// ------------------------------------------------------------------------------------------------------------
// GEMM_TC kernel.  grid = (tiles_m * tiles_n, split_k, batch), block = 320 threads:
// warp 0 TMA producer, warp 1 MMA issuer + tensor-memory owner, warps 2-9 gather producers, then epilogue.
// Built for each way its operands reach shared memory (GemmForm), with and without the cluster reduction, so that a kernel carries only the code it runs: the
// launches of a batch-1 model pass are a few microseconds long and meet a cold instruction cache.
// Two builds of each: MIN_CTAS = 1 (all registers), and MIN_CTAS = 2 (registers capped so that two CTAs share an SM when a
// record's shared memory and tensor memory allow it: one CTA's set-up and read-out then overlap the other's main loop).
// ------------------------------------------------------------------------------------------------------------
// Split-K over a cluster: extent (rows or columns) and bytes of the band of the output tile that split `owner` finishes.
__device__ __forceinline__ int red_band_extent(const GemmArgs& g, int owner) {
    const int whole = g.y_ns == 1 ? kHwTileM : g.tile_n;
    const int per = (whole + g.split_k - 1) / g.split_k;
    return max(0, min(whole, (owner + 1) * per) - owner * per);
}
__device__ __forceinline__ uint32_t red_band_bytes(const GemmArgs& g, int owner) {
    return (uint32_t)red_band_extent(g, owner) * 4u * (uint32_t)(g.y_ns == 1 ? g.tile_n + 4 : kRedColPitch);
}

enum GemmForm {
    kFormTma = 0,       // both operands K-major by TMA
    kFormMn = 1,        // both by TMA, one of them (or both) MN-major
    kFormIm2col = 2,    // one operand expanded from a slab of input rows, the other by TMA or gathered
    kFormIm2colRun = 6, // the same where the slab's channels are one run of memory: in the form above that copy cost every convolution 0.3 us
                        // (3x3 over 344 x 7 x 7 -> 32 9.02 us between graph nodes, 9.37 with it), more than two builds in turn do (the 53 layers of the
                        // MobileNetV2-shaped pass 256.5 us, 254.9 with one build)
    kFormX3 = 4,        // both K-major by TMA, error-compensated products, A and its remainders multiplied from shared memory ...
    kFormX3Tmem = 5,    // ... or from tensor memory
    kFormGather = 3,    // an operand gathered from global memory (the other one any way but by expansion)
    kFormRaw = 7        // an operand of ragged rows by boxes (the other one any way but by expansion): its code in the form above cost short
                        // launches there 0.2 to 0.5 us (132 heads of 21 x 64 over 21 4.4 us, 4.8 with it)
};

// CHAIN: a launch of a chained pass that does more than its layer (ChainArgs).
template <bool CHAIN> struct ChainParam {};
template <> struct ChainParam<true> { CUtensorMap tmap_z; ChainArgs a; };

template <int MIN_CTAS, int FORM, bool CLUSTER, bool CHAIN = false>
__global__ void __launch_bounds__(kGemmThreads, MIN_CTAS)
tt_gemm_tc_kernel(const __grid_constant__ CUtensorMap tmap_a0, const __grid_constant__ CUtensorMap tmap_b0,
                  const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ GemmArgs g, const __grid_constant__ ChainParam<CHAIN> chain) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_bar[kMaxStages];
    __shared__ uint64_t empty_bar[kMaxStages];
    __shared__ uint64_t accum_bar;
    __shared__ uint64_t slab_full[2];     // a slab chunk has landed (TMA)
    __shared__ uint64_t slab_empty[2];    // all gather warps are done with a slab buffer
    __shared__ uint64_t red_bar;          // split-K over a cluster: the other splits' bands of this CTA's output have landed
    __shared__ uint64_t lo_bar[kMaxStages];   // error-compensated products: the remainders of a stage's operand tiles are written;
                                              // operands of ragged rows: a stage's boxes have landed
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ int last_split_flag;
    __shared__ __align__(16) float s_bias[256];
    __shared__ int s_rowoff[256];

    // the warp index is broadcast from lane 0 so that the compiler knows it is the same in all lanes of a warp and
    // keeps the role loops (addresses, descriptors, counters) on the uniform datapath
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    volatile int* abortp = &abort_flag;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the next kernel of the stream may begin its set-up

    // tile coordinates
    int tm, tn;
    if (g.raster == 0) { tm = blockIdx.x % g.tiles_m; tn = blockIdx.x / g.tiles_m; }
    else               { tn = blockIdx.x % g.tiles_n; tm = blockIdx.x / g.tiles_n; }
    const int m0 = tm * kHwTileM, n0 = tn * g.tile_n;
    const int split = blockIdx.y, bz = CHAIN ? 0 : (int)blockIdx.z;
    // CHAIN: which layer of a group (a dense layer has no batch).  The first one's weights are in their operand's slot, the others' in
    // the image's and the last; what only they need is only read by them.
    const CUtensorMap *map_a = &tmap_a0, *map_b = &tmap_b0;
    const float* g_bias = g.bias;
    float* g_y = g.y;
    if constexpr (CHAIN) {
        if (blockIdx.z != 0u) {
            const CUtensorMap* w_map = blockIdx.z == 1u ? &tmap_x : &chain.tmap_z;
            if (chain.a.w_member == 1) map_a = w_map; else map_b = w_map;
            g_bias = blockIdx.z == 1u ? chain.a.bias_more[0] : chain.a.bias_more[1];
            g_y = blockIdx.z == 1u ? chain.a.y_more[0] : chain.a.y_more[1];
        }
    }
    const CUtensorMap &tmap_a = *map_a, &tmap_b = *map_b;
    const int kt_begin = split * g.k_tiles_per_split;
    const int kt_end = min(g.k_tiles, kt_begin + g.k_tiles_per_split);
    const int iters = kt_end - kt_begin;

    const uint32_t tiles_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    // (error-compensated products: a stage holds the two operand tiles and, behind them, their remainders, or B's alone)
    constexpr bool x3_tmem = FORM == kFormX3Tmem, x3 = FORM == kFormX3 || x3_tmem;
    const uint32_t lo_off = FORM == kFormX3Tmem ? g.b_stage_bytes : g.a_stage_bytes + g.b_stage_bytes;      // from an operand to its remainders
    const uint32_t stage_bytes = g.a_stage_bytes + g.b_stage_bytes + (x3 ? lo_off : 0u);
    // what the instantiation is made for (GemmForm); within it only the modes that its form leaves open are looked at
    constexpr bool slab_run = FORM == kFormIm2colRun, im2col = FORM == kFormIm2col || slab_run;
    constexpr bool gathers = FORM == kFormGather || FORM == kFormRaw, may_mn = FORM == kFormMn || gathers;
    const bool a_mn = may_mn && g.a_mode == OPM_TMA_MN, b_mn = may_mn && g.b_mode == OPM_TMA_MN;
    const bool a_tma = FORM == kFormTma || x3 || FORM == kFormMn || g.a_mode == OPM_TMA || a_mn;
    const bool b_tma = FORM == kFormTma || x3 || FORM == kFormMn || g.b_mode == OPM_TMA || b_mn;
    const bool any_tma = a_tma || b_tma, any_gather = !a_tma || !b_tma;
    const bool a_raw = FORM == kFormRaw && g.a_mode == OPM_RAW, b_raw = FORM == kFormRaw && g.b_mode == OPM_RAW;
    const bool any_raw = a_raw || b_raw;
    const int a_row0 = bz * g.M + m0, b_row0 = (g.b_tma_batched ? bz * g.N : 0) + n0;      // OPM_RAW: the tile's first row in the whole tensor
    const bool slab_tma = slab_run || (im2col && g.slab_tma != 0);
    // im2col geometry of this CTA: first output row of its pixels, the image row its slab starts at, slab chunks
    int ic_p_first = 0, ic_ih_lo = 0, ic_chunks = 0;
    if (im2col) {
        const int row0 = g.a_mode == OPM_IM2COL ? m0 : n0;
        ic_p_first = row0 / g.Q;
        ic_ih_lo = ic_p_first * g.sh - g.ph;
        ic_chunks = (iters + g.slab_tiles - 1) / g.slab_tiles;
    }
    // gather groups (global gathers only): 4 groups of 2 warps from 4 stages up, 2 groups of 4 warps for 2-3 stages,
    // else one group; the im2col expansion keeps all eight warps on one stage
    const int n_groups = im2col ? 1 : (g.stages >= 4 ? 4 : (g.stages >= 2 ? 2 : 1));
    const int wpg = kGatherWarps / n_groups;

    if (threadIdx.x == 32) {
        // the tensor maps are fetched ahead of their first use (they are kernel parameters: nothing the previous
        // kernel of the stream could still be writing)
        if (a_tma || a_raw) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_a) : "memory");
        if (b_tma || b_raw) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_b) : "memory");
        if (slab_tma && !slab_run) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_x) : "memory");
    }
    if (threadIdx.x == 0) {
        const uint32_t full_count = (any_tma ? 1u : 0u) + (any_gather ? (uint32_t)wpg : 0u);
        for (int s = 0; s < g.stages; ++s) {
            mbar_init(smem_u32(&full_bar[s]), full_count);
            mbar_init(smem_u32(&empty_bar[s]), 1u);
        }
        mbar_init(smem_u32(&accum_bar), 1u);
        if (x3) for (int s = 0; s < g.stages; ++s) mbar_init(smem_u32(&lo_bar[s]), (uint32_t)(x3_tmem ? kGatherWarps / 2 : kGatherWarps));
        if (any_raw) for (int s = 0; s < g.stages; ++s) mbar_init(smem_u32(&lo_bar[s]), 1u);
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&slab_full[b]), 1u);
            mbar_init(smem_u32(&slab_empty[b]), (uint32_t)kGatherWarps);
        }
        if (CLUSTER) {
            // the bands this CTA finishes arrive from the other splits: rows x (tile_n + 4) or columns x 128 floats each
            mbar_init(smem_u32(&red_bar), 1u);
            mbar_expect_tx(smem_u32(&red_bar), (uint32_t)(g.split_k - 1) * red_band_bytes(g, split));
        }
        abort_flag = 0;
        last_split_flag = 0;
        fence_mbar_init();
        fence_proxy_async_shared();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(&tmem_slot), g.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *(volatile uint32_t*)&tmem_slot;
    // A CTA's reduction area and its barrier may be used by a peer only once they exist: every thread announces
    // itself here (the barrier above is initialised) and checks, just before the first copy to a peer could be issued,
    // that all peers have done the same.
    if (CLUSTER) cluster_arrive();
    // Programmatic dependent launch: everything above (barriers, tensor memory) touched no global memory and may
    // run while the previous kernel of the stream is still draining; from here on its results are needed.  The
    // kernel that follows this one was allowed to start its own set-up at this kernel's entry.  (Without the launch
    // attribute both instructions do nothing.)
    // (The TMA warp waits a little later: it first requests the constant operand's first stages, see below.)
    if constexpr (CHAIN) {
        if (threadIdx.x == 64) prefetch_ahead(chain.a.ahead, blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z), gridDim.x * gridDim.y * gridDim.z);
    }
    if (warp != 0) asm volatile("griddepcontrol.wait;" ::: "memory");

    // Warps 0 and 1 run their loops with all 32 lanes: waits, counters and descriptor arithmetic stay
    // warp-uniform, and one elected lane issues the asynchronous instructions.
    if (warp == 0) {
        // ---------------- TMA producer ----------------
        const bool leader = elect_one();                 // this lane arms the barriers and issues every load
        const uint32_t a_atom = (uint32_t)(kHwTileM * g.row_bytes), b_atom = (uint32_t)(g.tile_n * g.row_bytes);
        const int a_bz = g.a_tma_batched ? bz : 0, b_bz = g.b_tma_batched ? bz : 0;
        // Constant operand (the caller promised that the weights are not written by the kernel in front of this one): its
        // tiles for the first pipeline stages are requested before the wait on that kernel, so they stream in while
        // it is still running.  The barrier only learns of the bytes here; the arrival comes with the stage's other operand.
        int n_pref = 0;
        if (g.w_operand) {
            n_pref = min(g.stages, iters);
            if (leader) {
                int kc0 = kt_begin * g.tile_k;
                for (int it = 0; it < n_pref; ++it, kc0 += g.tile_k) {
                    const uint32_t bar = smem_u32(&full_bar[it]);
                    uint32_t dst = tiles_base + (uint32_t)it * stage_bytes + (g.w_operand == 2 ? g.a_stage_bytes : 0u);
                    mbar_expect_tx_only(bar, g.w_operand == 2 ? g.b_stage_bytes : g.a_stage_bytes);
                    int kc = kc0;
#pragma unroll 1
                    for (int at = 0; at < g.n_atoms; ++at, kc += g.atom_k) {
                        if (g.w_operand == 1) { tma_load_3d(dst, &tmap_a, bar, kc, m0, a_bz); dst += a_atom; }
                        else { tma_load_3d(dst, &tmap_b, bar, kc, n0, b_bz); dst += b_atom; }
                    }
                }
            }
            __syncwarp();
        }
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (any_tma || slab_tma || any_raw) {
            int armed = n_pref;   // stages whose loads were issued
            uint32_t st = 0, ph = 0;
            const uint32_t full0 = smem_u32(&full_bar[0]), empty0 = smem_u32(&empty_bar[0]);
            int k0 = kt_begin * g.tile_k;
            uint32_t a_stage = tiles_base, full_addr = full0, empty_addr = empty0;
            // conv2d: slab chunk j (the input rows behind reduction tiles j*T .. j*T+T-1) goes to buffer j & 1 as one
            // box that starts `gap` columns left of the image: the zero fill writes gaps and rows outside the image
            const int RS = g.R * g.S, T = g.slab_tiles;
            const uint32_t slab0 = tiles_base + g.slab_off;
            int slab_issued = 0;
            auto issue_chunk = [&](int j) {
                const int b = j & 1;
                const uint32_t bar = smem_u32(&slab_full[b]), dst = slab0 + (uint32_t)b * g.slab_buf_bytes;
                const int c_first = (kt_begin * g.tile_k + j * T * g.tile_k) / RS;
                if (!slab_run) {
                    mbar_expect_tx(bar, g.slab_box_bytes);
                    tma_load_4d(dst, &tmap_x, bar, -g.slab_gap, ic_ih_lo, c_first, bz);
                } else {
                    // (c_first, the channels and a chunk's length are multiples of four)
                    const bool on_a = g.a_mode == OPM_IM2COL;
                    const float* img = (on_a ? g.a : g.b) + (long long)bz * (on_a ? g.a_bs : g.b_bs);
                    const uint32_t bytes = 4u * (uint32_t)(min(g.slab_box_ch, g.C - c_first) * g.slab_chpitch);
                    mbar_expect_tx(bar, bytes);
                    bulk_load(dst, img + (long long)c_first * g.slab_chpitch, bytes, bar);
                }
            };
            if (slab_tma) {
                if (leader) { issue_chunk(0); if (ic_chunks > 1) issue_chunk(1); }
                slab_issued = min(ic_chunks, 2);
            }
            int next_slab_it = slab_tma ? (slab_issued - 1) * T : 0x7fffffff;   // chunk `slab_issued` is requested when chunk slab_issued-1 starts
            bool ok = true;
            for (int it = 0; it < iters; ++it, k0 += g.tile_k) {
                if (it == next_slab_it) {
                    next_slab_it += T;
                    if (slab_issued < ic_chunks) {
                        // its buffer is free once the gather warps have left chunk slab_issued - 2
                        const int j = slab_issued;
                        const bool freed = mbar_wait(smem_u32(&slab_empty[j & 1]), (uint32_t)((j - 2) >> 1) & 1u, abortp, g.status, 5u, g.wait_ns);
                        if (!__all_sync(0xffffffffu, freed)) { ok = false; break; }
                        if (leader) issue_chunk(j);
                        ++slab_issued;
                    }
                }
                if (!any_tma && !any_raw) continue;
                const bool got = mbar_wait(empty_addr, ph ^ 1u, abortp, g.status, 1u, g.wait_ns);
                if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
                if (leader && any_raw) {
                    // (a stage whose products are done has been realigned, too: its boxes' buffer is free)
                    const uint32_t bar = smem_u32(&lo_bar[st]), dst = tiles_base + g.raw_off + st * g.raw_stage_bytes;
                    const uint32_t boxes = 4u * (uint32_t)(g.tile_k + 4);
                    mbar_expect_tx(bar, (a_raw ? boxes * (uint32_t)kHwTileM : 0u) + (b_raw ? boxes * (uint32_t)g.tile_n : 0u));
                    if (a_raw) load_raw_boxes(dst, &tmap_a, bar, g.a_raw_box, a_row0, g.K, k0);
                    if (b_raw) load_raw_boxes(dst + 4u * g.a_raw_box, &tmap_b, bar, g.b_raw_box, b_row0, g.K, k0);
                }
                if (leader && any_tma) {
                    // (test facility: split 0 may be told to expect more than arrives, see tt_workload_test_stall)
                    const bool a_here = a_tma && !(it < n_pref && g.w_operand == 1), b_here = b_tma && !(it < n_pref && g.w_operand == 2);
                    mbar_expect_tx(full_addr, (a_here ? g.a_stage_bytes : 0u) + (b_here ? g.b_stage_bytes : 0u) +
                                                  ((it == 0 && split == 0) ? g.extra_tx : 0u));
                    if (a_here) {
                        uint32_t dst = a_stage;
                        int kc = k0;
                        if (a_mn) load_mn_boxes(dst, &tmap_a, full_addr, m0, kHwTileM, k0, g.tile_k, a_bz);
                        else
#pragma unroll 1
                        for (int at = 0; at < g.n_atoms; ++at, dst += a_atom, kc += g.atom_k) tma_load_3d(dst, &tmap_a, full_addr, kc, m0, a_bz);
                    }
                    if (b_here) {
                        uint32_t dst = a_stage + g.a_stage_bytes;
                        int kc = k0;
                        if (b_mn) load_mn_boxes(dst, &tmap_b, full_addr, n0, g.tile_n, k0, g.tile_k, b_bz);
                        else
#pragma unroll 1
                        for (int at = 0; at < g.n_atoms; ++at, dst += b_atom, kc += g.atom_k) tma_load_3d(dst, &tmap_b, full_addr, kc, n0, b_bz);
                    }
                }
                __syncwarp();
                armed = max(armed, it + 1);
                a_stage += stage_bytes; full_addr += 8u; empty_addr += 8u;
                if (++st == (uint32_t)g.stages) { st = 0; ph ^= 1u; a_stage = tiles_base; full_addr = full0; empty_addr = empty0; }
            }
            if ((!ok || *abortp) && lane == 0) {
                // let copies in flight land before shared memory is given back (bounded)
                const int first = max(0, armed - g.stages);
                for (int it = first; it < armed; ++it) {
                    const unsigned long long t0 = global_timer_ns();
                    while (!mbar_try_wait(smem_u32(&full_bar[it % g.stages]), (uint32_t)(it / g.stages) & 1u)) {
                        if (global_timer_ns() - t0 > 2000000ull) break;
                    }
                    while (any_raw && !mbar_try_wait(smem_u32(&lo_bar[it % g.stages]), (uint32_t)(it / g.stages) & 1u)) {
                        if (global_timer_ns() - t0 > 4000000ull) break;
                    }
                }
                for (int j = max(0, slab_issued - 2); j < slab_issued; ++j) {
                    const unsigned long long t0 = global_timer_ns();
                    while (!mbar_try_wait(smem_u32(&slab_full[j & 1]), (uint32_t)(j >> 1) & 1u)) {
                        if (global_timer_ns() - t0 > 2000000ull) break;
                    }
                }
            }
            __syncwarp();
        }
        if (CLUSTER) cluster_wait();
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        {
            bool ok = true;
            uint32_t st = 0, ph = 0;
            const uint32_t full0 = smem_u32(&full_bar[0]), empty0 = smem_u32(&empty_bar[0]);
            // descriptors differ only in their 14-bit start-address field: keep the constant upper word, step the
            // lower word by (bytes >> 4) per stage, per atom and per 8-wide K slice
            const DescSteps da = desc_steps(a_mn, g.row_bytes, kHwTileM, g.tile_k, g.atom_k);
            const DescSteps db = desc_steps(b_mn, g.row_bytes, g.tile_n, g.tile_k, g.atom_k);
            const bool any_mn = a_mn || b_mn;
            const uint32_t d_hi = da.hi, d_lo = da.lo;
            const uint32_t a_lo0 = d_lo + ((tiles_base & 0x3FFFFu) >> 4);
            const uint32_t b_lo0 = db.lo + (((tiles_base + g.a_stage_bytes) & 0x3FFFFu) >> 4);
            const uint32_t stage_step = stage_bytes >> 4;
            const uint32_t a_atom = da.atom, b_atom = db.atom;
            const int k8_per_atom = g.atom_k >> 3;
            const uint32_t a_next_atom = a_atom - da.k8 * (uint32_t)k8_per_atom, b_next_atom = b_atom - db.k8 * (uint32_t)k8_per_atom;
            const bool leader = elect_one();             // this lane issues every multiply-accumulate and every commit
            // accumulators: reduction steps are dealt round-robin; an accumulator's first step overwrites
            uint32_t d_tmem = tmem_base;
            const uint32_t d_end = tmem_base + (uint32_t)(g.n_acc * g.tile_n);
            int fresh = g.n_acc;                         // accumulators not written yet
            uint32_t x3_buf = 0;
            uint32_t a_stage = a_lo0, b_stage = b_lo0, full_addr = full0, empty_addr = empty0;
            for (int it = 0; it < iters; ++it) {
                bool got = mbar_wait(full_addr, ph, abortp, g.status, 2u, g.wait_ns);
                if (x3) got = mbar_wait(smem_u32(&lo_bar[st]), ph, abortp, g.status, 16u, g.wait_ns) && got;   // the remainders too
                if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
                tc_fence_after();
                if (leader) {
                    // descriptors step by 2 (32 bytes = 8 TF32 along K) inside a swizzle atom, then to the next atom
                    uint32_t a_lo = a_stage, b_lo = b_stage;
                    if (any_mn && g.n_acc == 1) {
                        issue_steps_any(tmem_base, da.hi, db.hi, a_lo, b_lo, da.k8, db.k8, a_atom, b_atom, g.n_atoms, k8_per_atom, g.idesc, it > 0 ? 1u : 0u);
                    } else if (g.n_acc == 1) {
                        // one accumulator: nothing to rotate.  The common tile_k values are unrolled completely, so
                        // that an issue is two additions and the instruction.
                        auto issue_stage = [&](uint32_t a0, uint32_t b0, uint32_t accumulate) {
                            if (g.tile_k == 64) issue_steps<2, 4>(tmem_base, d_hi, a0, b0, a_atom, b_atom, g.idesc, accumulate);
                            else if (g.tile_k == 32) issue_steps<1, 4>(tmem_base, d_hi, a0, b0, a_atom, b_atom, g.idesc, accumulate);
                            else if (g.tile_k == 128) issue_steps<4, 4>(tmem_base, d_hi, a0, b0, a_atom, b_atom, g.idesc, accumulate);
                            else if (g.tile_k == 16) issue_steps<1, 2>(tmem_base, d_hi, a0, b0, a_atom, b_atom, g.idesc, accumulate);
                            else issue_steps<1, 1>(tmem_base, d_hi, a0, b0, a_atom, b_atom, g.idesc, accumulate);
                        };
                        const uint32_t accumulate = it > 0 ? 1u : 0u;
                        if (x3_tmem) {
                            // the two cross terms first (small), then the product of what the tensor core sees of a and b
                            const uint32_t lo = lo_off >> 4, ta = tmem_base + g.x3_col + x3_buf * 2u * (uint32_t)g.tile_k;
                            auto issue = [&](uint32_t a, uint32_t b, uint32_t acc) {
#pragma unroll 1
                                for (int at = 0; at < g.n_atoms; ++at, b += b_atom) {
#pragma unroll 4
                                    for (uint32_t k8 = 0; k8 < (uint32_t)k8_per_atom; ++k8, a += 8u, acc = 1u)
                                        mma_tf32_ta(tmem_base, a, ((uint64_t)d_hi << 32) | (uint64_t)(b + 2u * k8), g.idesc, acc);
                                }
                            };
                            issue(ta + (uint32_t)g.tile_k, b_lo, accumulate);
                            issue(ta, b_lo + lo, 1u);
                            issue(ta, b_lo, 1u);
                            if (++x3_buf == (uint32_t)g.x3_bufs) x3_buf = 0u;
                        } else if (x3) {
                            const uint32_t lo = lo_off >> 4;
                            issue_stage(a_lo + lo, b_lo, accumulate);
                            issue_stage(a_lo, b_lo + lo, 1u);
                            issue_stage(a_lo, b_lo, 1u);
                        } else {
                            issue_stage(a_lo, b_lo, accumulate);
                        }
                    } else
#pragma unroll 1
                    for (int at = 0; at < g.n_atoms; ++at) {
#pragma unroll 4
                        for (int k8 = 0; k8 < k8_per_atom; ++k8) {
                            mma_tf32(d_tmem, ((uint64_t)da.hi << 32) | (uint64_t)a_lo, ((uint64_t)db.hi << 32) | (uint64_t)b_lo, g.idesc,
                                     fresh > 0 ? 0u : 1u);
                            a_lo += da.k8; b_lo += db.k8;
                            if (fresh > 0) --fresh;
                            d_tmem += (uint32_t)g.tile_n;
                            if (d_tmem == d_end) d_tmem = tmem_base;
                        }
                        a_lo += a_next_atom; b_lo += b_next_atom;
                    }
                    if (it + (x3_tmem ? g.x3_bufs : g.stages) < iters) mma_commit(empty_addr);   // stage reusable once these MMAs have read it (if anything follows)
                }
                __syncwarp();
                a_stage += stage_step; b_stage += stage_step; full_addr += 8u; empty_addr += 8u;
                if (++st == (uint32_t)g.stages) { st = 0; ph ^= 1u; a_stage = a_lo0; b_stage = b_lo0; full_addr = full0; empty_addr = empty0; }
            }
            if (ok && leader) mma_commit(smem_u32(&accum_bar));    // accumulator complete
            __syncwarp();
        }
        if (CLUSTER) cluster_wait();
    } else {
        // ---------------- gather producers, then epilogue ----------------
        const int gw = warp - 2;
        const int gt = (int)threadIdx.x - 64;
        const int quad = warp & 3;                       // tensor-memory lane quadrant this warp may read
        const int m = m0 + quad * 32 + lane;
        // bias is fetched now so that its latency hides behind the main loop
        if (g.bias_mode == 2 && gt < g.tile_n) s_bias[gt] = (n0 + gt < g.N) ? __ldg(g_bias + n0 + gt) : 0.f;
        if (CLUSTER && g.bias_mode == 1 && gt < kHwTileM) s_bias[gt] = (m0 + gt < g.M) ? __ldg(g_bias + m0 + gt) : 0.f;   // for the cluster reduction
        const float bias_row = (g.bias_mode == 1 && m < g.M) ? __ldg(g_bias + m) : 0.f;
        if (im2col) {
            // ---- conv2d: slab staging + expansion; all eight warps work on the same stage ----
            const bool on_a = g.a_mode == OPM_IM2COL;
            const int rows = on_a ? kHwTileM : g.tile_n, row0 = on_a ? m0 : n0, ext = on_a ? g.M : g.N;
            const float* img = (on_a ? g.a : g.b) + (long long)bz * (on_a ? g.a_bs : g.b_bs);
            const float* o_src = on_a ? g.b + (long long)bz * g.b_bs : g.a + (long long)bz * g.a_bs;   // the other operand
            const bool o_gather = on_a ? !b_tma : !a_tma;
            const uint32_t ktab = tiles_base + g.ktab_off;
            const uint32_t slab0 = tiles_base + g.slab_off;
            const uint32_t rowoff = smem_u32(s_rowoff);
            const int RS = g.R * g.S, T = g.slab_tiles;
            const int last = min(row0 + rows, ext) - 1;
            const int p_first = ic_p_first, p_last = last / g.Q;
            const int ih_lo = ic_ih_lo;
            const int in_rows_cta = (p_last - p_first) * g.slab_rstep + g.R;
            const int kbeg = kt_begin * g.tile_k;
            const bool vec16 = g.slab_vec16 && ((reinterpret_cast<uintptr_t>(img) & 15u) == 0);
            // per tile row: byte offset of its pixel's window origin inside a slab channel
            if (gt < rows) {
                const int grow = min(row0 + gt, ext - 1);    // rows past the extent repeat the last pixel (never stored)
                const int p = grow / g.Q, q = grow - p * g.Q;
                s_rowoff[gt] = 4 * ((p - p_first) * g.slab_rstep * g.slab_wp + q * g.sw + (g.slab_gap - g.pw));
            }
            // per reduction index of this CTA: byte offset of (c, r, s) inside the slab, channel counted from 0
            // (made by the host when the record was applied); four entries per copy
            for (int i = gt * 4; i < iters * g.tile_k; i += kGatherThreads * 4)
                cp_async_16(ktab + 4u * (uint32_t)i, g.ktab_dev + kbeg + i);
            cp_async_commit();
            // zeros that no copy ever writes: the tail behind each buffer's last row, and, when the gather warps stage
            // the slab themselves, every gap and every row outside the image
            if (slab_tma) {
                const uint32_t tail = 4u * (uint32_t)(g.slab_box_ch * g.slab_chpitch);
                for (int b = 0; b < g.slab_nbuf; ++b)
                    for (uint32_t o = tail + (uint32_t)gt * 4u; o < g.slab_buf_bytes; o += (uint32_t)kGatherThreads * 4u)
                        st_shared_u32(slab0 + (uint32_t)b * g.slab_buf_bytes + o, 0u);
            } else {
                const uint32_t slab_bytes = (uint32_t)g.slab_nbuf * g.slab_buf_bytes;
                for (uint32_t o = (uint32_t)gt * 16u; o < slab_bytes; o += (uint32_t)kGatherThreads * 16u)
                    st_shared_v4(slab0 + o, 0.f, 0.f, 0.f, 0.f);
            }
            bool ok = gather_vote(true);                 // row table and zeros are in place (the k-table may still be in flight)
            const int n_chunks = ic_chunks;
            const ExpandPlan xplan = make_expand_plan(rows, rowoff, g.tile_k, g.atom_k, g.row_bytes, g.swz_mask, gw, lane);   // after the vote: reads s_rowoff
            auto chunk_first_channel = [&](int j) { return (kbeg + j * T * g.tile_k) / RS; };
            auto chunk_load = [&](int j) {               // the gather warps stage chunk j themselves (no TMA)
                const int k_lo = kbeg + j * T * g.tile_k;
                const int k_hi = min(g.K, kbeg + min((j + 1) * T, iters) * g.tile_k);
                if (k_hi > k_lo) {
                    const int c_first = k_lo / RS, c_last = (k_hi - 1) / RS;
                    slab_load_chunk(g, img, slab0 + (uint32_t)(j & 1) * g.slab_buf_bytes, c_first, c_last - c_first + 1, ih_lo,
                                    in_rows_cta, vec16, gt);
                }
                cp_async_commit();
            };
            if (!slab_tma) {
                chunk_load(0);
                if (n_chunks > 1) chunk_load(1);
            }
            const uint32_t full0 = smem_u32(&full_bar[0]), empty0 = smem_u32(&empty_bar[0]);
            uint32_t st = 0, ph = 0;
            for (int j = 0; j < n_chunks; ++j) {
                if (slab_tma) {
                    if (ok && !mbar_wait(smem_u32(&slab_full[j & 1]), (uint32_t)(j >> 1) & 1u, abortp, g.status, 6u, g.wait_ns)) ok = false;
                    if (j == 0) {
                        cp_async_wait<0>();              // the k-table copies of this thread ...
                        ok = gather_vote(ok);            // ... and of every other gather thread have landed
                        if (!ok) break;
                    }
                } else {
                    if (j + 1 < n_chunks) cp_async_wait<1>(); else cp_async_wait<0>();
                    ok = gather_vote(ok);                // every thread's copies of chunk j are visible to all
                    if (!ok) break;
                }
                // table offsets count channels from 0: rebase the buffer by the chunk's first channel
                const uint32_t slab = slab0 + (uint32_t)(j & 1) * g.slab_buf_bytes - 4u * (uint32_t)(chunk_first_channel(j) * g.slab_chpitch);
                const int it_end = min((j + 1) * T, iters);
                for (int it = j * T; it < it_end; ++it) {
                    if (ok && !mbar_wait(empty0 + st * 8u, ph ^ 1u, abortp, g.status, 3u, g.wait_ns)) ok = false;
                    if (ok) {
                        const uint32_t a_s = tiles_base + st * stage_bytes, b_s = a_s + g.a_stage_bytes;
                        const uint32_t kt = ktab + 4u * (uint32_t)(it * g.tile_k);
                        expand_stage(xplan, on_a ? a_s : b_s, rows, slab, rowoff, kt, g.tile_k, g.atom_k, g.row_bytes, g.swz_mask, gw, lane);
                        if (o_gather) {
                            const int k0 = (kt_begin + it) * g.tile_k;
                            if (on_a) gather_stage(g.b_mode, b_s, g.tile_n, o_src, g.b_rs, g.b_ks, n0, g.N, k0, g.K, g.tile_k,
                                                   g.atom_k, g.row_bytes, g.swz_mask, gw, kGatherWarps, lane);
                            else gather_stage(g.a_mode, a_s, kHwTileM, o_src, g.a_rs, g.a_ks, m0, g.M, k0, g.K, g.tile_k,
                                              g.atom_k, g.row_bytes, g.swz_mask, gw, kGatherWarps, lane);
                        }
                        fence_proxy_async_shared();      // generic-proxy stores -> visible to the tensor core's reads
                        __syncwarp();
                        if (lane == 0) mbar_arrive(full0 + st * 8u);
                    }
                    if (++st == (uint32_t)g.stages) { st = 0; ph ^= 1u; }
                }
                if (slab_tma) {
                    // this warp is done with the buffer: the producer may refill it
                    __syncwarp();
                    if (lane == 0 && j + 2 < n_chunks) mbar_arrive(smem_u32(&slab_empty[j & 1]));
                } else if (j + 2 < n_chunks) {
                    ok = gather_vote(ok);                // everyone is done reading this buffer
                    if (!ok) break;
                    chunk_load(j + 2);
                }
            }
            cp_async_wait<0>();
        } else if (any_gather) {
            const float* a_src = g.a + (long long)bz * g.a_bs;
            const float* b_src = g.b + (long long)bz * g.b_bs;
            const int grp = gw / wpg, wig = gw - grp * wpg;
            const uint32_t full0 = smem_u32(&full_bar[0]), empty0 = smem_u32(&empty_bar[0]);
            int st = grp % g.stages;
            uint32_t ph = (uint32_t)(grp / g.stages) & 1u;
            for (int it = grp; it < iters; it += n_groups) {
                if (!mbar_wait(empty0 + (uint32_t)st * 8u, ph ^ 1u, abortp, g.status, 3u, g.wait_ns)) break;
                const uint32_t a_s = tiles_base + (uint32_t)st * stage_bytes, b_s = a_s + g.a_stage_bytes;
                const int k0 = (kt_begin + it) * g.tile_k;
                if (any_raw) {
                    if (!mbar_wait(smem_u32(&lo_bar[st]), ph, abortp, g.status, 18u, g.wait_ns)) break;
                    const uint32_t raw = tiles_base + g.raw_off + (uint32_t)st * g.raw_stage_bytes;
#pragma unroll 1
                    for (int o = 0; o < 2; ++o) {        // (one copy of the code for both operands)
                        if (!(o == 0 ? a_raw : b_raw)) continue;
                        const RealignArgs r{o == 0 ? a_s : b_s, o == 0 ? raw : raw + 4u * g.a_raw_box, o == 0 ? g.a_raw_box : g.b_raw_box, o == 0 ? kHwTileM : g.tile_n,
                                            o == 0 ? a_row0 : b_row0, o == 0 ? g.a_rows_all : g.b_rows_all, k0, g.K, g.tile_k, g.atom_k, g.row_bytes, g.swz_mask, wig, wpg};
                        realign_stage(r, o == 0 ? g.a : g.b, lane);
                    }
                }
                if (!a_tma && !a_raw) gather_stage(g.a_mode, a_s, kHwTileM, a_src, g.a_rs, g.a_ks, m0, g.M, k0, g.K, g.tile_k,
                                         g.atom_k, g.row_bytes, g.swz_mask, wig, wpg, lane);
                if (!b_tma && !b_raw) gather_stage(g.b_mode, b_s, g.tile_n, b_src, g.b_rs, g.b_ks, n0, g.N, k0, g.K, g.tile_k,
                                         g.atom_k, g.row_bytes, g.swz_mask, wig, wpg, lane);
                fence_proxy_async_shared();              // generic-proxy stores -> visible to the tensor core's reads
                __syncwarp();
                if (lane == 0) mbar_arrive(full0 + (uint32_t)st * 8u);
                st += n_groups;
                while (st >= g.stages) { st -= g.stages; ph ^= 1u; }
            }
        }
        if (x3 && !x3_tmem) {
            // ---- error-compensated products: once a stage's operand tiles have landed, the eight warps write, 16 bytes
            // per thread and step, what the tensor core will NOT see of every value (x minus x truncated to TF32's ten
            // mantissa bits: exact in fp32) into the second half of the stage, in the same swizzled layout ----
            const uint32_t full0 = smem_u32(&full_bar[0]);
            uint32_t st = 0, ph = 0;
            for (int it = 0; it < iters; ++it) {
                if (!mbar_wait(full0 + st * 8u, ph, abortp, g.status, 15u, g.wait_ns)) break;
                const uint32_t hi = tiles_base + st * stage_bytes;
                constexpr uint32_t step = 16u * (uint32_t)kGatherThreads;
                for (uint32_t off = 16u * (uint32_t)gt; off < lo_off; off += 4u * step) {      // four reads in flight
                    float4 v[4];
#pragma unroll
                    for (uint32_t j = 0; j < 4u; ++j)
                        if (off + j * step < lo_off) v[j] = ld_shared_v4f(hi + off + j * step);
#pragma unroll
                    for (uint32_t j = 0; j < 4u; ++j)
                        if (off + j * step < lo_off)
                            st_shared_v4(hi + lo_off + off + j * step, v[j].x - __uint_as_float(__float_as_uint(v[j].x) & 0xFFFFE000u),
                                         v[j].y - __uint_as_float(__float_as_uint(v[j].y) & 0xFFFFE000u),
                                         v[j].z - __uint_as_float(__float_as_uint(v[j].z) & 0xFFFFE000u),
                                         v[j].w - __uint_as_float(__float_as_uint(v[j].w) & 0xFFFFE000u));
                }
                fence_proxy_async_shared();              // generic-proxy stores -> visible to the tensor core's reads
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&lo_bar[st]));
                if (++st == (uint32_t)g.stages) { st = 0; ph ^= 1u; }
            }
        }
        if (x3_tmem) {
            // ---- the same where a CTA's reduction is long.  B's remainders go behind the stage, A and its remainders to tensor
            // memory, where all three products read A: that takes two thirds of A's traffic off shared memory, which bounds this form
            // (a step of 8 with 128 columns: 384 cycles with A in shared memory, 256 this way, the products 192). ----
            const uint32_t full0 = smem_u32(&full_bar[0]), empty0 = smem_u32(&empty_bar[0]);
            const int row = quad * 32 + lane, half = gw >> 2, atom_shift = g.atom_k == 32 ? 5 : (g.atom_k == 16 ? 4 : 3);
            const uint32_t swz = (uint32_t)((row >> (g.row_bytes == 128 ? 0 : (g.row_bytes == 64 ? 1 : 2))) & g.swz_mask) << 4;
            const uint32_t line = (uint32_t)(row * g.row_bytes), atom_bytes = (uint32_t)(kHwTileM * g.row_bytes);
            const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16) + g.x3_col;
            auto lo_of = [](float x) { return x - __uint_as_float(__float_as_uint(x) & 0xFFFFE000u); };
            // two groups of four warps (one per lane quadrant) take alternate stages, so that one stage's way through their hands, of which
            // most is waiting (arrival, reads, stores, fence), hides behind the other's
            for (int it = half; it < iters; it += 2) {
                const uint32_t st = (uint32_t)(it % g.stages), buf = (uint32_t)(it % g.x3_bufs);
                bool ok = mbar_wait(full0 + st * 8u, (uint32_t)(it / g.stages) & 1u, abortp, g.status, 15u, g.wait_ns);
                if (it >= g.x3_bufs) {                   // the products that read this buffer of tensor memory are done
                    const int before = it - g.x3_bufs;
                    ok = ok && mbar_wait(empty0 + (uint32_t)(before % g.stages) * 8u, (uint32_t)(before / g.stages) & 1u, abortp, g.status, 19u, g.wait_ns);
                }
                if (!__all_sync(0xffffffffu, ok)) break;
                tc_fence_after();
                const uint32_t hi = tiles_base + st * stage_bytes;
                // A: a lane has one row, 8 columns at a time
                const uint32_t t_buf = t_row + buf * 2u * (uint32_t)g.tile_k;
#pragma unroll 2
                for (int u = 0; u < g.tile_k >> 3; ++u) {
                    const uint32_t at = hi + (uint32_t)((u * 8) >> atom_shift) * atom_bytes + line, in = (uint32_t)((u * 8) & (g.atom_k - 1)) * 4u;
                    const float4 p = ld_shared_v4f(at + (in ^ swz)), q = ld_shared_v4f(at + ((in + 16u) ^ swz));
                    const float a[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
                    const float r[8] = {lo_of(p.x), lo_of(p.y), lo_of(p.z), lo_of(p.w), lo_of(q.x), lo_of(q.y), lo_of(q.z), lo_of(q.w)};
                    tmem_st8(t_buf + (uint32_t)u * 8u, a);
                    tmem_st8(t_buf + (uint32_t)g.tile_k + (uint32_t)u * 8u, r);
                }
                constexpr uint32_t step = 16u * (uint32_t)(kGatherThreads / 2);
                const uint32_t b = hi + g.a_stage_bytes;
                for (uint32_t off = 16u * (uint32_t)(gt & (kGatherThreads / 2 - 1)); off < g.b_stage_bytes; off += 4u * step) {      // four reads in flight
                    float4 v[4];
#pragma unroll
                    for (uint32_t j = 0; j < 4u; ++j)
                        if (off + j * step < g.b_stage_bytes) v[j] = ld_shared_v4f(b + off + j * step);
#pragma unroll
                    for (uint32_t j = 0; j < 4u; ++j)
                        if (off + j * step < g.b_stage_bytes) st_shared_v4(b + lo_off + off + j * step, lo_of(v[j].x), lo_of(v[j].y), lo_of(v[j].z), lo_of(v[j].w));
                }
                fence_proxy_async_shared();              // generic-proxy stores -> visible to the tensor core's reads
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&lo_bar[st]));
            }
        }
        // split-K over a cluster: everything the reduction needs that does not depend on the accumulator is worked out
        // here, while the main loop is still running (divisions, 64-bit products, first reads of kernel parameters)
        struct {
            int sk, whole, per; uint32_t line, slot, red; bool along_cols, gelu, clamp, vec_ok; int bias_mode;
            float lo, hi; float* ybase; const float* rbase; long long y_ms, y_ns;
        } cr;
        if (CLUSTER) {
            cr.sk = g.split_k;
            cr.along_cols = g.y_ns == 1;                                 // bands of rows
            cr.whole = cr.along_cols ? kHwTileM : g.tile_n;
            cr.per = (cr.whole + cr.sk - 1) / cr.sk;                     // lines (rows or columns) per band
            cr.line = 4u * (uint32_t)(cr.along_cols ? g.tile_n + 4 : kRedColPitch);   // bytes per line
            cr.slot = (uint32_t)cr.per * cr.line;                        // bytes between the bands of two consecutive splits
            cr.red = tiles_base + g.red_off;
            cr.ybase = g_y + (long long)bz * g.y_bs;
            cr.rbase = !CHAIN && g.residual ? g.residual + (long long)bz * g.y_bs : nullptr;      // (chained dense layers with a skip tensor take the other kernel)
            cr.lo = g.act == TT_ACT_NONE || g.act == TT_ACT_GELU_ERF ? -INFINITY : 0.f;
            cr.hi = g.act == TT_ACT_RELU6 ? 6.f : INFINITY;
            cr.gelu = g.act == TT_ACT_GELU_ERF; cr.clamp = g.act == TT_ACT_RELU || g.act == TT_ACT_RELU6;
            cr.bias_mode = g.bias_mode; cr.y_ms = g.y_ms; cr.y_ns = g.y_ns;
            const long long lead = cr.along_cols ? g.y_ms : g.y_ns;      // stride of the other output axis
            cr.vec_ok = (lead & 3) == 0 && (g.y_bs & 3) == 0 && (reinterpret_cast<uintptr_t>(cr.ybase) & 15u) == 0 &&
                        (cr.rbase == nullptr || (reinterpret_cast<uintptr_t>(cr.rbase) & 15u) == 0);
            if constexpr (MIN_CTAS == 1) {               // (kept in registers; the register-capped build works them out again)
                int pin = cr.per;
                asm volatile("" : "+r"(pin), "+r"(cr.slot), "+r"(cr.red), "+l"(cr.ybase), "+l"(cr.y_ms), "+l"(cr.y_ns));
                if constexpr (!CHAIN) asm volatile("" : "+l"(cr.rbase));
                cr.per = pin;
            }
        }
        // epilogue: warp w owns tensor-memory lanes 32*(w % 4) .. +31; the two warps of a lane quadrant take
        // alternate 32-column blocks
        const bool have_acc = mbar_wait(smem_u32(&accum_bar), 0u, abortp, g.status, 4u, g.wait_ns);
        // every epilogue thread takes the same decision (named barrier 1 over the epilogue threads); the barrier
        // also orders the bias staging above against its readers below
        uint32_t all_acc;
        asm volatile(
            "{\n\t.reg .pred p, q;\n\t"
            "setp.ne.u32 q, %1, 0;\n\t"
            "bar.red.and.pred p, 1, %2, q;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(all_acc) : "r"((uint32_t)have_acc), "n"(kGatherThreads) : "memory");
        if (CLUSTER) cluster_wait();                   // every peer is set up: its reduction area and barrier may be used
        if (all_acc) {
            tc_fence_after();
            const int half = gw >> 2;
            const bool m_ok = m < g.M;
            const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16);
            const bool split_mode = !CLUSTER && g.split_k > 1;   // splits beyond a cluster go through the workspace
            // a split with fewer reduction steps than accumulators leaves the last ones unwritten
            const int n_acc = min(g.n_acc, iters * (g.tile_k >> 3));
            // split-K workspace [split][batch][N][M]: a column of the tile is contiguous across lanes
            const long long per_split = (long long)g.batch * g.M * (long long)g.N;
            float* pcol = g.partial + (long long)bz * g.M * (long long)g.N + m;
            if (CLUSTER) {
                // split-K over a cluster, step 1: this split's partial tile goes to the pipeline buffers (idle: every
                // multiply-accumulate has completed) in the layout of the reduction area, a band being one run of bytes
                const int row = quad * 32 + lane;
                const uint32_t row_dst = tiles_base + 4u * (uint32_t)(g.y_ns == 1 ? row * (g.tile_n + 4) : row);
#pragma unroll 1
                for (int c0 = half * 32; c0 < g.tile_n; c0 += 64) {
                    uint32_t r[32];
                    tmem_ld32(t_row + (uint32_t)c0, r);
                    tmem_wait_ld();
#pragma unroll 1
                    for (int j = 1; j < n_acc; ++j) {        // the other accumulators, in fixed order
                        uint32_t t2[32];
                        tmem_ld32(t_row + (uint32_t)(j * g.tile_n + c0), t2);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) + __uint_as_float(t2[i]));
                    }
                    if (g.y_ns == 1) {
                        // bands of rows: [row][col], pitch tile_n + 4
                        const uint32_t dst = row_dst + 4u * (uint32_t)c0;
#pragma unroll
                        for (int j = 0; j < 32; j += 4)
                            if (c0 + j < g.tile_n)           // tile_n is a multiple of 16: groups of four are whole
                                st_shared_v4(dst + 4u * (uint32_t)j, __uint_as_float(r[j]), __uint_as_float(r[j + 1]),
                                             __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]));
                    } else {
                        // bands of columns: [col][row], pitch 128 -- the lanes of a warp write 128 contiguous bytes
                        uint32_t dst = row_dst + 4u * (uint32_t)(c0 * kRedColPitch);
#pragma unroll
                        for (int j = 0; j < 32; ++j, dst += 4u * (uint32_t)kRedColPitch)
                            if (c0 + j < g.tile_n) st_shared_u32(dst, r[j]);
                    }
                }
                fence_proxy_async_shared();              // generic-proxy stores -> visible to the bulk copies below
            } else if (split_mode) {
                // 1. park this split's partial tile in the workspace
                float* pmine = pcol + (long long)split * per_split;
#pragma unroll 1
                for (int c0 = half * 32; c0 < g.tile_n; c0 += 64) {
                    uint32_t r[32];
                    tmem_ld32(t_row + (uint32_t)c0, r);
                    tmem_wait_ld();
#pragma unroll 1
                    for (int j = 1; j < n_acc; ++j) {        // the other accumulators, in fixed order
                        uint32_t t2[32];
                        tmem_ld32(t_row + (uint32_t)(j * g.tile_n + c0), t2);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) + __uint_as_float(t2[i]));
                    }
                    const int nb = n0 + c0;
                    const int cnt = min(g.N - nb, g.tile_n - c0);
                    if (!m_ok || cnt <= 0) continue;
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (j < cnt) __stcg(pmine + (long long)(nb + j) * g.M, __uint_as_float(r[j]));
                }
                // 2. the split that arrives last at this tile's counter reduces all of them, in split order
                __threadfence();
                asm volatile("bar.sync 1, %0;" ::"n"(kGatherThreads) : "memory");
                if (threadIdx.x == 64) {
                    unsigned* ctr = g.counters + (size_t)bz * gridDim.x + blockIdx.x;
                    const unsigned old = atomicAdd(ctr, 1u);
                    const int last = old == (unsigned)(g.split_k - 1);
                    if (last) *ctr = 0u;                 // all splits have arrived: ready for the next launch
                    last_split_flag = last;
                }
                asm volatile("bar.sync 1, %0;" ::"n"(kGatherThreads) : "memory");
            }
            const bool finish = !CLUSTER && (!split_mode || (*(volatile int*)&last_split_flag != 0));
            if (finish) {
                if (split_mode) __threadfence();
                EpiArgs e;
                e.ybase = g_y + (long long)bz * g.y_bs;
                e.rbase = !CHAIN && g.residual ? g.residual + (long long)bz * g.y_bs : nullptr;
                e.y_ms = g.y_ms; e.y_ns = g.y_ns; e.M = g.M;
                e.lo = g.act == TT_ACT_NONE || g.act == TT_ACT_GELU_ERF ? -INFINITY : 0.f;
                e.hi = g.act == TT_ACT_RELU6 ? 6.f : INFINITY;
                e.gelu = g.act == TT_ACT_GELU_ERF;
                e.vec = (g.vec_store & 1) != 0;
                const bool transposed = g.y_ns == 1 && g.y_ms != 1;
                const uint32_t stg = tiles_base + (uint32_t)gw * (uint32_t)kStageBytesPerWarp;   // pipeline buffers are idle now
                const int m_first = m0 + quad * 32;
                uint32_t r[32];
                int c0 = half * 32;
                if (!split_mode && c0 < g.tile_n) tmem_ld32(t_row + (uint32_t)c0, r);
#pragma unroll 1
                for (; c0 < g.tile_n; c0 += 64) {
                    float v[32];
                    const int nb = n0 + c0;
                    const int cnt = min(g.N - nb, g.tile_n - c0);
                    if (!split_mode) {
                        // read-out is software-pipelined: the next block's tensor-memory load is in flight while
                        // this block is biased, activated and stored
                        tmem_wait_ld();
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
#pragma unroll 1
                        for (int a = 1; a < n_acc; ++a) {        // the other accumulators, in fixed order
                            tmem_ld32(t_row + (uint32_t)(a * g.tile_n + c0), r);
                            tmem_wait_ld();
#pragma unroll
                            for (int j = 0; j < 32; ++j) v[j] += __uint_as_float(r[j]);
                        }
                        if (c0 + 64 < g.tile_n) tmem_ld32(t_row + (uint32_t)(c0 + 64), r);
                    } else {
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = 0.f;
                        if (m_ok && cnt > 0) {
#pragma unroll 2
                            for (int sp = 0; sp < g.split_k; ++sp) {
                                const float* ps = pcol + (long long)sp * per_split + (long long)nb * g.M;
#pragma unroll
                                for (int j = 0; j < 32; ++j)
                                    if (j < cnt) v[j] += __ldcg(ps + (long long)j * g.M);
                            }
                        }
                    }
                    if (cnt <= 0) continue;              // warp-uniform
                    if (g.bias_mode == 1) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] += bias_row;
                    } else if (g.bias_mode == 2) {
#pragma unroll
                        for (int j = 0; j < 32; j += 4) {
                            const float4 b = *reinterpret_cast<const float4*>(s_bias + c0 + j);
                            v[j] += b.x; v[j + 1] += b.y; v[j + 2] += b.z; v[j + 3] += b.w;
                        }
                    }
                    // full blocks take the unguarded path (16-byte accesses need the aligned layout when transposed)
                    const bool full = cnt >= 32 && m_first + 32 <= g.M && (e.vec || !transposed);
                    if (e.rbase == nullptr) {
                        // no residual: activate here, once, outside the store loops
                        if (e.gelu) {
#pragma unroll
                            for (int j = 0; j < 32; ++j) v[j] = gelu_erf(v[j]);
                        } else if (g.act != TT_ACT_NONE) {
#pragma unroll
                            for (int j = 0; j < 32; ++j) v[j] = fminf(fmaxf(v[j], e.lo), e.hi);
                        }
                        if (full) epilogue_block<true, false>(v, e, m_first, nb, cnt, stg, lane, transposed);
                        else epilogue_block<false, false>(v, e, m_first, nb, cnt, stg, lane, transposed);
                    } else {
                        if (full) epilogue_block<true, true>(v, e, m_first, nb, cnt, stg, lane, transposed);
                        else epilogue_block<false, true>(v, e, m_first, nb, cnt, stg, lane, transposed);
                    }
                }
            }
        }
        if (CLUSTER) {
            // step 2: once every read-out warp has staged its part, one thread per peer sends that peer's band
            asm volatile("bar.sync 1, %0;" ::"n"(kGatherThreads) : "memory");
            if (all_acc && lane == 0 && gw < cr.sk && gw != split) {
                const uint32_t bytes = (uint32_t)max(0, min(cr.whole, (gw + 1) * cr.per) - gw * cr.per) * cr.line;
                if (bytes != 0u) {
                    // (a CTA keeps no slot for its own split: the splits after it move down by one)
                    bulk_copy_to_peer(map_to_peer(cr.red + (uint32_t)(split < gw ? split : split - 1) * cr.slot, (uint32_t)gw),
                                      tiles_base + (uint32_t)gw * cr.slot, bytes, map_to_peer(smem_u32(&red_bar), (uint32_t)gw));
                    bulk_copies_done();                  // (this CTA's shared memory is no longer read, the peer's no longer written)
                }
            }
            __syncwarp();
            cluster_arrive();                            // second round: this warp sends nothing to a peer any more
            // step 3: add up the bands of this CTA once the other splits' copies of them have landed
            const bool landed = __all_sync(0xffffffffu, mbar_wait_cluster(smem_u32(&red_bar), 0u, abortp, g.status, 14u, g.wait_ns));
            // four outputs that are neighbours in memory, first one (mm, nn), `off` bytes into the band: the partial
            // sums of all splits (this split's own from the staging copy, the others' from the reduction area)
            auto load_sums = [&](uint32_t off, float4 (&p)[8]) {
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (q < cr.sk) p[q] = ld_shared_v4f((q == split ? tiles_base + (uint32_t)q * cr.slot : cr.red + (uint32_t)(q < split ? q : q - 1) * cr.slot) + off);
            };
            // ... are added in split order, then bias, residual, activation, one 16-byte store
            auto finish4 = [&](const float4 (&p)[8], int mm, int nn, int valid) {
                float4 acc = p[0];
#pragma unroll
                for (int q = 1; q < 8; ++q)
                    if (q < cr.sk) { acc.x += p[q].x; acc.y += p[q].y; acc.z += p[q].z; acc.w += p[q].w; }
                float v[4] = {acc.x, acc.y, acc.z, acc.w};
                const long long o = (long long)mm * cr.y_ms + (long long)nn * cr.y_ns;   // the four are o, o+1, o+2, o+3
                // the tile's bias values were staged in shared memory before the main loop
                if (cr.bias_mode == 1) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[i] += s_bias[mm - m0 + (cr.along_cols ? 0 : i)];
                } else if (cr.bias_mode == 2) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[i] += s_bias[nn - n0 + (cr.along_cols ? i : 0)];
                }
                if (cr.rbase) {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (i < valid) v[i] += __ldg(cr.rbase + o + i);
                }
                if (cr.gelu) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[i] = gelu_erf(v[i]);
                } else if (cr.clamp) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[i] = fminf(fmaxf(v[i], cr.lo), cr.hi);
                }
                if (valid == 4 && cr.vec_ok) *reinterpret_cast<float4*>(cr.ybase + o) = make_float4(v[0], v[1], v[2], v[3]);
                else {
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (i < valid) cr.ybase[o + i] = v[i];
                }
            };
            // a warp takes two lines (rows or columns) of the band at a time, the loads of both under way together (one
            // line in the register-capped build)
            constexpr int kLines = MIN_CTAS == 1 ? 2 : 1;
            if (!landed) {
                // (the wait recorded the time-out; nothing is stored)
            } else if (cr.along_cols) {
                // this CTA's band of rows; the lanes of a warp walk a row's columns four at a time
                const int rows_here = min(min(kHwTileM, (split + 1) * cr.per), g.M - m0) - split * cr.per;
                const int c_end = min(g.tile_n, g.N - n0);
                for (int rl = gw; rl < rows_here; rl += kLines * kGatherWarps) {
                    const bool two = kLines == 2 && rl + kGatherWarps < rows_here;
                    for (int col = lane * 4; col < c_end; col += 128) {
                        float4 pa[8], pb[8];
                        load_sums((uint32_t)rl * cr.line + 4u * (uint32_t)col, pa);
                        if (two) load_sums((uint32_t)(rl + kGatherWarps) * cr.line + 4u * (uint32_t)col, pb);
                        finish4(pa, m0 + split * cr.per + rl, n0 + col, min(4, c_end - col));
                        if (two) finish4(pb, m0 + split * cr.per + rl + kGatherWarps, n0 + col, min(4, c_end - col));
                    }
                }
            } else {
                // this CTA's band of columns; the lanes of a warp walk a column's 128 rows four at a time
                const int cols_here = min(min(g.tile_n, (split + 1) * cr.per), g.N - n0) - split * cr.per;
                const int r_end = min(kHwTileM, g.M - m0);
                if (lane * 4 < r_end)
                    for (int cl = gw; cl < cols_here; cl += kLines * kGatherWarps) {
                        const bool two = kLines == 2 && cl + kGatherWarps < cols_here;
                        float4 pa[8], pb[8];
                        load_sums((uint32_t)cl * cr.line + 16u * (uint32_t)lane, pa);
                        if (two) load_sums((uint32_t)(cl + kGatherWarps) * cr.line + 16u * (uint32_t)lane, pb);
                        finish4(pa, m0 + lane * 4, n0 + split * cr.per + cl, min(4, r_end - lane * 4));
                        if (two) finish4(pb, m0 + lane * 4, n0 + split * cr.per + cl + kGatherWarps, min(4, r_end - lane * 4));
                    }
            }
        }
    }
    if (CLUSTER) {
        // Every thread of every CTA of the cluster takes part in both rounds of the cluster barrier, also after a
        // tripped wait: the second round completes when no CTA sends any more, so none leaves while a copy into its
        // shared memory could still be under way.
        if (warp < 2) cluster_arrive();
        cluster_wait();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, g.tmem_cols);
    }
}

// ------------------------------------------------------------------------------------------------------------
// GEMM_TC, persistent form (record field `persistent` = 1).  grid = resident CTAs; every CTA walks output tiles
// t = unit, unit + units, ... (a unit is a CTA, or a pair of CTAs when CG = 2) with
//   - the operand pipeline running on across tile boundaries (the loads of the next tile are in flight while this
//     tile's last multiply-accumulates run),
//   - TWO accumulators in tensor memory, used alternately: the read-out warps drain tile t (bias, residual,
//     activation, stores) while the MMA warp already accumulates tile t + 1,
//   - barriers and tensor memory set up once per CTA instead of once per tile.
// Operands arrive by TMA and are multiplied as they lie: K-major tensors in K-major tiles, operands whose ROW index is the
// contiguous one in memory (the image of a 1x1 convolution: pixels; the second operand of an NN batch_matmul) in MN-major
// tiles (make_desc_mn).  No split-K, one accumulator per tile.
// Warps: 0 TMA producer, 1 MMA issuer + tensor-memory owner, 2-9 read-out (two per lane quadrant, alternate 32-column
// blocks; only 6-9 when the record's stages leave shared memory for four staging areas).
// Read-out.  Rows of the output that are contiguous along the tile's columns leave through a ring of `epi_bufs` 32 x 32
// blocks per warp in shared memory (128-byte lines, swizzled so that a lane's 16-byte stores do not conflict) and TMA
// stores, which also clip the ragged edges; a residual comes in through the same ring by TMA one block ahead, so no
// lane waits on a global load.  1x1 convolution 64 -> 256 at 56 x 56 with residual, batch 32: 116 us with the residual
// loaded by the lanes and the image transposed in shared memory, 41 us this way (bytes at the copy rate: 35 us).
// CG = 2: two CTAs of a cluster work on one 256-row tile.  Each loads its own 128 rows of A and its half of B's
// rows with ordinary (non-multicast) TMA; the CTA of rank 0 issues tcgen05.mma.cta_group::2, which reads both
// CTAs' shared memory and writes each CTA's half of the accumulator into that CTA's tensor memory, so an SM reads
// only half of B per multiply-accumulate.  Both CTAs' loads report their bytes to the stage barrier of rank 0 (which
// expects the pair's total), a multicast tcgen05.commit frees the stage and publishes the accumulator in both CTAs.
// ------------------------------------------------------------------------------------------------------------
template <int CG>
__device__ __forceinline__ void mma_tf32_cg(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    if constexpr (CG == 1) {
        mma_tf32(d_tmem, adesc, bdesc, idesc, accumulate);
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
    }
}
// Arrive on the barrier at this shared-memory offset once every MMA issued so far has completed: in this CTA (CG 1),
// or in both CTAs of the pair (CG 2; the arrival is multicast, no data moves).
template <int CG>
__device__ __forceinline__ void mma_commit_cg(uint32_t bar) {
    if constexpr (CG == 1) {
        mma_commit(bar);
    } else {
        const uint16_t mask = 3;
        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                     ::"r"(bar), "h"(mask) : "memory");
    }
}
// Arrive on the barrier at the same offset in the CTA of rank `rank` of this cluster.
__device__ __forceinline__ void mbar_arrive_remote(uint32_t bar, uint32_t rank) {
    asm volatile(
        "{\n\t.reg .b32 ra;\n\t"
        "mapa.shared::cluster.u32 ra, %0, %1;\n\t"
        "mbarrier.arrive.release.cluster.shared::cluster.b64 _, [ra];\n\t}"
        ::"r"(bar), "r"(rank) : "memory");
}
// TMA load whose completion is reported to a barrier given by its cluster-wide address, which may lie in the other
// CTA of the pair (no multicast: the data goes to this CTA's shared memory only).
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const void* tmap, uint32_t bar_cluster, int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(tmap), "r"(bar_cluster), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
// One 3-D box from shared memory to a tensor (clipped at its extents); tracked by the issuing thread's bulk groups.
__device__ __forceinline__ void tma_store_3d(const void* tmap, uint32_t src, int c0, int c1, int c2) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4}], [%1];"
                 ::"l"(tmap), "r"(src), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ void bulk_stores_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Wait until at most N of the store groups this thread committed have still to read their shared memory.
template <int N>
__device__ __forceinline__ void bulk_stores_pending() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }

// Instantiated for what a plan uses, so that a launch carries only the code it runs (a single-wave launch meets it cold: 3-6 %
// on every record of this form, dense 2268 x 2256 -> 3944 76 -> 71 us).  MN: an operand is MN-major (otherwise the descriptors
// step by constants).  OUT: outputs leave by TMA stores.
template <int CG, bool MN, bool OUT>
__global__ void __launch_bounds__(kGemmThreads, 1)
tt_gemm_ps_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
                  const __grid_constant__ CUtensorMap tmap_y, const __grid_constant__ CUtensorMap tmap_r, const GemmArgs g) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_bar[kMaxStages];     // a stage's operands have landed
    __shared__ uint64_t empty_bar[kMaxStages];    // every multiply-accumulate that reads the stage has completed
    __shared__ uint64_t acc_full[2];              // an accumulator holds a finished tile
    __shared__ uint64_t acc_empty[2];             // the read-out warps (of both CTAs) have drained it
    __shared__ uint64_t last_full;                // the CTA's last tile is complete, and with it the pipeline idle
    __shared__ uint64_t res_full[8 * kMaxEpiBufs];   // per read-out warp and ring buffer: a residual block has landed
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ __align__(16) float s_bias[4][256];  // per tile under way: the bias of its columns

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    volatile int* abortp = &abort_flag;
    pdl_allow_next();
    const uint32_t rank = CG == 2 ? cluster_ctarank() : 0u;
    const int unit = (int)blockIdx.x / CG, n_units = (int)gridDim.x / CG;
    const int my_tiles = g.total_tiles > unit ? (g.total_tiles - unit + n_units - 1) / n_units : 0;
    const int tiles_per_batch = g.tiles_m * g.tiles_n;
    const int kt_n = g.k_tiles;

    const uint32_t tiles_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t stage_bytes = g.a_stage_bytes + g.b_stage_bytes;
    const bool a_mn = MN && g.a_mn != 0, b_mn = MN && g.b_mn != 0;
    const int b_rows = g.b_rows_cta;
    const int epi_warps = g.epi_warps;

    if (threadIdx.x == 32) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_a) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_b) : "memory");
        if (OUT) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_y) : "memory");
        if (g.res_tma) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_r) : "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < g.stages; ++s) {
            mbar_init(smem_u32(&full_bar[s]), 1u);
            mbar_init(smem_u32(&empty_bar[s]), 1u);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(smem_u32(&acc_full[a]), 1u);
            mbar_init(smem_u32(&acc_empty[a]), (uint32_t)(epi_warps * CG));
        }
        mbar_init(smem_u32(&last_full), 1u);
        if (g.res_tma) for (int b = 0; b < 8 * kMaxEpiBufs; ++b) mbar_init(smem_u32(&res_full[b]), 1u);
        abort_flag = 0;
        fence_mbar_init();
        fence_proxy_async_shared();
    }
    if (warp == 1) {
        if constexpr (CG == 1) {
            tmem_alloc(smem_u32(&tmem_slot), g.tmem_cols);
            tmem_relinquish();
        } else {
            // both CTAs of the pair allocate, with the same warp and the same destination offset
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(g.tmem_cols) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        }
    }
    tc_fence_before();
    __syncthreads();
    if constexpr (CG == 2) cluster_sync_all();           // the peer's barriers exist before anything arrives on them
    tc_fence_after();
    const uint32_t tmem_base = *(volatile uint32_t*)&tmem_slot;
    pdl_wait_prev();                                      // the set-up above touched no global memory

    auto decode = [&](int i, int& m0, int& n0, int& bz) {
        const int t = unit + i * n_units;
        bz = t / tiles_per_batch;
        const int r = t - bz * tiles_per_batch;
        int tm, tn;
        if (g.raster == 0) { tm = r % g.tiles_m; tn = r / g.tiles_m; }
        else               { tn = r % g.tiles_n; tm = r / g.tiles_n; }
        m0 = (tm * CG + (int)rank) * kHwTileM;
        n0 = tn * g.tile_n;
    };

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        const bool leader = elect_one();
        const uint32_t a_atom = (uint32_t)(kHwTileM * g.row_bytes), b_atom = (uint32_t)(b_rows * g.row_bytes);
        bool ok = true;
        uint32_t st = 0, ph = 0;
        long long issued = 0;
        for (int i = 0; i < my_tiles && ok; ++i) {
            int m0, n0, bz;
            decode(i, m0, n0, bz);
            const int a_bz = g.a_tma_batched ? bz : 0, b_bz = g.b_tma_batched ? bz : 0;
            const int nb0 = n0 + (int)rank * b_rows;      // CG 2: this CTA's half of the B rows
            for (int kt = 0, k0 = 0; kt < kt_n; ++kt, k0 += g.tile_k) {
                const bool got = mbar_wait(smem_u32(&empty_bar[st]), ph ^ 1u, abortp, g.status, 1u, g.wait_ns);
                if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
                if (leader) {
                    uint32_t bar = smem_u32(&full_bar[st]);
                    // (test facility: the first stage may be told to expect more than arrives, see tt_workload_test_stall)
                    if (rank == 0) mbar_expect_tx(bar, (uint32_t)CG * stage_bytes + (issued == 0 ? g.extra_tx : 0u));
                    if constexpr (CG == 2) bar = map_to_peer(bar, 0u);       // the pair's loads all report to rank 0
                    uint32_t dst = tiles_base + st * stage_bytes;
                    int kc = k0;
                    if (a_mn) load_mn_boxes(dst, &tmap_a, bar, m0, kHwTileM, k0, g.tile_k, a_bz);
                    else
#pragma unroll 1
                    for (int at = 0; at < g.n_atoms; ++at, dst += a_atom, kc += g.atom_k) {
                        if constexpr (CG == 2) tma_load_3d_pair(dst, &tmap_a, bar, kc, m0, a_bz);
                        else tma_load_3d(dst, &tmap_a, bar, kc, m0, a_bz);
                    }
                    dst = tiles_base + st * stage_bytes + g.a_stage_bytes;
                    kc = k0;
                    if (b_mn) load_mn_boxes(dst, &tmap_b, bar, nb0, b_rows, k0, g.tile_k, b_bz);
                    else
#pragma unroll 1
                    for (int at = 0; at < g.n_atoms; ++at, dst += b_atom, kc += g.atom_k) {
                        if constexpr (CG == 2) tma_load_3d_pair(dst, &tmap_b, bar, kc, nb0, b_bz);
                        else tma_load_3d(dst, &tmap_b, bar, kc, nb0, b_bz);
                    }
                }
                __syncwarp();
                ++issued;
                if (++st == (uint32_t)g.stages) { st = 0; ph ^= 1u; }
            }
        }
        if ((!ok || *abortp) && lane == 0) {
            // let copies in flight land before shared memory is given back (bounded)
            if (rank == 0) {
                const long long first = issued > g.stages ? issued - g.stages : 0;
                for (long long it = first; it < issued; ++it) {
                    const unsigned long long t0 = global_timer_ns();
                    while (!mbar_try_wait(smem_u32(&full_bar[it % g.stages]), (uint32_t)(it / g.stages) & 1u)) { if (global_timer_ns() - t0 > 2000000ull) break; }
                }
            } else {
                // this CTA's loads report to rank 0's barriers: give them time to land instead (the pair leaves
                // together, after rank 0 has seen the pair's bytes or given up on them)
                const unsigned long long t0 = global_timer_ns();
                while (global_timer_ns() - t0 < 200000ull) { }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer (of a pair: rank 0's) ----------------
        const bool leader = elect_one();
        uint32_t st = 0, ph = 0;
        bool ok = true;
        if (CG == 2 && rank != 0) {
            // rank 0 issues for the pair
        } else {
            const DescSteps da = desc_steps(a_mn, g.row_bytes, kHwTileM, g.tile_k, g.atom_k);
            const DescSteps db = desc_steps(b_mn, g.row_bytes, b_rows, g.tile_k, g.atom_k);
            const uint32_t a_lo0 = da.lo + ((tiles_base & 0x3FFFFu) >> 4);
            const uint32_t b_lo0 = db.lo + (((tiles_base + g.a_stage_bytes) & 0x3FFFFu) >> 4);
            const uint32_t stage_step = stage_bytes >> 4;
            const int k8n = g.atom_k >> 3;
            for (int i = 0; i < my_tiles && ok; ++i) {
                const uint32_t acc = (uint32_t)i & 1u, aph = ((uint32_t)i >> 1) & 1u;
                // the read-out of the tile that used this accumulator two tiles ago has finished
                const bool freed = CG == 2 ? mbar_wait_cluster(smem_u32(&acc_empty[acc]), aph ^ 1u, abortp, g.status, 12u, g.wait_ns)
                                           : mbar_wait(smem_u32(&acc_empty[acc]), aph ^ 1u, abortp, g.status, 12u, g.wait_ns);
                if (!__all_sync(0xffffffffu, freed)) { ok = false; break; }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + acc * (uint32_t)g.tile_n;
                for (int kt = 0; kt < kt_n; ++kt) {
                    const bool got = mbar_wait(smem_u32(&full_bar[st]), ph, abortp, g.status, 2u, g.wait_ns);
                    if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
                    tc_fence_after();
                    if (leader) {
                        uint32_t a_lo = a_lo0 + st * stage_step, b_lo = b_lo0 + st * stage_step;
                        uint32_t accumulate = kt > 0 ? 1u : 0u;
#pragma unroll 1
                        for (int at = 0; at < g.n_atoms; ++at, a_lo += da.atom, b_lo += db.atom) {
                            if (!MN && k8n == 4) {
#pragma unroll
                                for (uint32_t k8 = 0; k8 < 4; ++k8) {
                                    mma_tf32_cg<CG>(d_tmem, ((uint64_t)da.hi << 32) | (uint64_t)(a_lo + 2u * k8), ((uint64_t)da.hi << 32) | (uint64_t)(b_lo + 2u * k8), g.idesc,
                                                    k8 == 0 ? accumulate : 1u);
                                }
                                accumulate = 1u;
                            } else {
                                uint32_t a = a_lo, b = b_lo;
#pragma unroll 4
                                for (int k8 = 0; k8 < k8n; ++k8, a += da.k8, b += db.k8) {
                                    mma_tf32_cg<CG>(d_tmem, ((uint64_t)da.hi << 32) | (uint64_t)a, ((uint64_t)db.hi << 32) | (uint64_t)b, g.idesc, accumulate);
                                    accumulate = 1u;
                                }
                            }
                        }
                        mma_commit_cg<CG>(smem_u32(&empty_bar[st]));          // stage reusable once these MMAs have read it
                    }
                    __syncwarp();
                    if (++st == (uint32_t)g.stages) { st = 0; ph ^= 1u; }
                }
                if (ok && leader) mma_commit_cg<CG>(smem_u32(&acc_full[acc]));   // the tile's accumulator is complete
                if (ok && leader && i + 1 == my_tiles) mma_commit_cg<CG>(smem_u32(&last_full));
                __syncwarp();
            }
        }
    } else if (warp >= 10 - epi_warps || g.epi_late) {
        // ---------------- read-out: tensor memory -> bias, residual, activation -> global memory ----------------
        // A plan whose stages leave room for four read-out warps only gets the other four for the last tile, whose read-out
        // nothing hides: the pipeline's buffers are idle by then and take the staging blocks of all eight (dense 1854 x 680 ->
        // 1248 by CTA pairs, one tile each: 15.6 -> 13.8 us).
        const bool helper = warp < 10 - epi_warps;
        const int ew = helper ? 0 : warp - (10 - epi_warps);
        const int quad = warp & 3;                       // tensor-memory lane quadrant this warp may read
        int c_first = (ew >> 2) * 32, c_step = epi_warps * 8;            // the 32-column blocks of a tile that this warp takes
        EpiArgs e;
        e.y_ms = g.y_ms; e.y_ns = g.y_ns; e.M = g.M;
        e.lo = g.act == TT_ACT_NONE || g.act == TT_ACT_GELU_ERF ? -INFINITY : 0.f;
        e.hi = g.act == TT_ACT_RELU6 ? 6.f : INFINITY;
        e.gelu = g.act == TT_ACT_GELU_ERF;
        e.vec = (g.vec_store & 1) != 0;
        const bool transposed = g.y_ns == 1 && g.y_ms != 1;
        constexpr bool tma_out = OUT;
        const bool res_in = g.res_tma != 0;
        uint32_t ring = tiles_base + g.epi_off + (uint32_t)ew * g.epi_warp_bytes;
        int bufs = g.epi_bufs;
        const int per_tile = c_first < g.tile_n ? (g.tile_n - c_first + c_step - 1) / c_step : 0;    // blocks of a tile
        bool ok = true;
        // residual blocks are requested one ahead of their use: cursor of the next request
        int ri = 0, rc = c_first, rb = 0, rm0 = 0, rn0 = 0, rbz = 0;
        if (my_tiles > 0) decode(0, rm0, rn0, rbz);
        auto request_residual = [&]() {                  // lane 0; the buffer is free
            const uint32_t bar = smem_u32(&res_full[ew * kMaxEpiBufs + rb]);
            mbar_expect_tx(bar, 4096u);
            if (tma_out) tma_load_3d(ring + (uint32_t)rb * 4096u, &tmap_r, bar, rn0 + rc, rm0 + quad * 32, g.y_tma_batched ? rbz : 0);
            else tma_load_3d(ring + (uint32_t)rb * 4096u, &tmap_r, bar, rm0 + quad * 32, rn0 + rc, g.y_tma_batched ? rbz : 0);
        };
        auto advance_request = [&]() {
            if (++rb == bufs) rb = 0;
            rc += c_step;
            if (rc >= g.tile_n) { rc = c_first; if (++ri < my_tiles) decode(ri, rm0, rn0, rbz); }
        };
        int req_left = per_tile > 0 ? my_tiles : 0;      // (tiles; a warp without blocks requests nothing)
        if (res_in && req_left > 0) {
            if (lane == 0) request_residual();
            advance_request();
        }
        int buf = 0;                                     // ring position of the current block
        uint32_t rph = 0;                                // phase of the residual barriers at `buf`
        for (int i = helper ? max(0, my_tiles - 1) : 0; i < my_tiles; ++i) {
            int m0, n0, bz;
            decode(i, m0, n0, bz);
            const uint32_t acc = (uint32_t)i & 1u, aph = ((uint32_t)i >> 1) & 1u;
            const bool all_eight = g.epi_late && i + 1 == my_tiles;
            if (all_eight) { c_first = ((warp - 2) >> 2) * 32; c_step = 64; ring = tiles_base + (uint32_t)(warp - 2) * kLateRingBytes; bufs = 2; buf = 0; }
            const int m_first = m0 + quad * 32, m = m_first + lane;
            // the bias of this warp's blocks, staged while the tile is still being accumulated.  Warps that share columns write
            // the same values; four buffers, because a warp can be up to three tiles ahead of the slowest (whose arrival on an
            // accumulator the third needs)
            float* tile_bias = s_bias[i & 3];
            auto stage_bias = [&]() {
                for (int c = c_first; c < g.tile_n; c += c_step) tile_bias[c + lane] = (n0 + c + lane < g.N) ? __ldg(g.bias + n0 + c + lane) : 0.f;
                __syncwarp();
            };
            if (g.bias_mode == 2 && !helper) stage_bias();
            const float bias_row = (g.bias_mode == 1 && m < g.M) ? __ldg(g.bias + m) : 0.f;
            // (each read-out warp walks on its own: a barrier over the eight of them per tile cost batch_matmul NT
            // 3072 x 128 x 128 x 64 a tenth of its time, 73 us against 65 us)
            // (a helper has not followed the accumulators' phases: the last tile has a barrier of its own)
            ok = ok && mbar_wait(helper ? smem_u32(&last_full) : smem_u32(&acc_full[acc]), helper ? 0u : aph, abortp, g.status, 4u, g.wait_ns);
            if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
            tc_fence_after();
            if (g.bias_mode == 2 && helper) stage_bias();       // (not earlier: its buffer may have been an older tile's)
            e.ybase = g.y + (long long)bz * g.y_bs;
            e.rbase = g.residual ? g.residual + (long long)bz * g.y_bs : nullptr;
            const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16) + acc * (uint32_t)g.tile_n;
            uint32_t r[32];
            if (c_first < g.tile_n) tmem_ld32(t_row + (uint32_t)c_first, r);
            else if (lane == 0) {
                if (CG == 2) mbar_arrive_remote(smem_u32(&acc_empty[acc]), 0u);
                else mbar_arrive(smem_u32(&acc_empty[acc]));
            }
#pragma unroll 1
            for (int c0 = c_first; c0 < g.tile_n; c0 += c_step) {
                float v[32];
                const int nb = n0 + c0;
                const int cnt = min(g.N - nb, g.tile_n - c0);
                const uint32_t stg = ring + (uint32_t)buf * 4096u;
                if (res_in) {
                    // request the next block's residual: its buffer's last TMA store (if any) must have read it
                    if (ri < my_tiles) {
                        if (lane == 0) {
                            if (tma_out) { if (bufs == 2) bulk_stores_pending<0>(); else bulk_stores_pending<1>(); }
                            request_residual();
                        }
                        advance_request();
                    }
                } else if (tma_out) {
                    if (lane == 0) { if (bufs == 1) bulk_stores_pending<0>(); else bulk_stores_pending<1>(); }   // this buffer's last store has read it
                    __syncwarp();
                }
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
                if (c0 + c_step < g.tile_n) tmem_ld32(t_row + (uint32_t)(c0 + c_step), r);
                else {
                    // every value of this warp's part of the accumulator is in registers: hand it back to the MMA warp
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        if (CG == 2) mbar_arrive_remote(smem_u32(&acc_empty[acc]), 0u);
                        else mbar_arrive(smem_u32(&acc_empty[acc]));
                    }
                }
                if (g.bias_mode == 1) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] += bias_row;
                } else if (g.bias_mode == 2) {
#pragma unroll
                    for (int j = 0; j < 32; j += 4) {
                        const float4 b = *reinterpret_cast<const float4*>(tile_bias + c0 + j);
                        v[j] += b.x; v[j + 1] += b.y; v[j + 2] += b.z; v[j + 3] += b.w;
                    }
                }
                if (res_in) {
                    if (!mbar_wait(smem_u32(&res_full[ew * kMaxEpiBufs + buf]), rph, abortp, g.status, 17u, g.wait_ns)) ok = false;
                    ok = __all_sync(0xffffffffu, ok); // (after a lost block nothing more is stored; the next tile ends the walk)
                    if (tma_out) {
#pragma unroll
                        for (int j = 0; j < 32; j += 4) {
                            const float4 q = ld_shared_v4f(stg + (uint32_t)lane * 128u + ((uint32_t)((j >> 2) ^ (lane & 7)) << 4));
                            v[j] += q.x; v[j + 1] += q.y; v[j + 2] += q.z; v[j + 3] += q.w;
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] += ld_shared_f32(stg + (uint32_t)j * 128u + (uint32_t)lane * 4u);
                        __syncwarp();                    // the buffer may be requested again after the next block
                    }
                }
                if (tma_out || res_in || e.rbase == nullptr) {
                    if (e.gelu) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = gelu_erf(v[j]);
                    } else if (g.act != TT_ACT_NONE) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] = fminf(fmaxf(v[j], e.lo), e.hi);
                    }
                }
                if (!ok) continue;
                if (tma_out) {
#pragma unroll
                    for (int j = 0; j < 32; j += 4)
                        st_shared_v4(stg + (uint32_t)lane * 128u + ((uint32_t)((j >> 2) ^ (lane & 7)) << 4), v[j], v[j + 1], v[j + 2], v[j + 3]);
                    fence_proxy_async_shared();          // the lanes' stores -> visible to the TMA store
                    __syncwarp();
                    if (lane == 0) {
                        if (cnt > 0 && m_first < g.M) tma_store_3d(&tmap_y, stg, nb, m_first, g.y_tma_batched ? bz : 0);
                        bulk_stores_commit();
                    }
                } else if (cnt > 0) {                    // (warp-uniform)
                    const bool full = cnt >= 32 && m_first + 32 <= g.M && (e.vec || !transposed);
                    if (res_in || e.rbase == nullptr) {
                        if (full) epilogue_block<true, false>(v, e, m_first, nb, cnt, stg, lane, transposed);
                        else epilogue_block<false, false>(v, e, m_first, nb, cnt, stg, lane, transposed);
                    } else {
                        if (full) epilogue_block<true, true>(v, e, m_first, nb, cnt, stg, lane, transposed);
                        else epilogue_block<false, true>(v, e, m_first, nb, cnt, stg, lane, transposed);
                    }
                }
                if (tma_out || res_in) { if (++buf == bufs) { buf = 0; rph ^= 1u; } }
            }
        }
        if (tma_out && lane == 0) bulk_stores_pending<0>();      // shared memory stays until the last store has read it
        if (!ok && res_in && lane == 0) {
            // a residual block that was requested and not waited for (bounded)
            const unsigned long long t0 = global_timer_ns();
            while (global_timer_ns() - t0 < 200000ull) { }
        }
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    // a pair stays together until neither CTA touches the other's shared memory, barriers or tensor memory any more
    if constexpr (CG == 2) cluster_sync_all();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        if constexpr (CG == 1) tmem_dealloc(tmem_base, g.tmem_cols);
        else asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(g.tmem_cols) : "memory");
    }
}

// ------------------------------------------------------------------------------------------------------------
// DW_SIMT: depthwise conv + bias + activation.  One CTA = tile_c channels x tile_h x tile_w outputs of one image.
// The input halo tile is staged in shared memory with coalesced row reads; each thread then produces `items`
// consecutive outputs along the width and stores them with vec-wide stores.
// ------------------------------------------------------------------------------------------------------------
__global__ void tt_dwconv_kernel(const DwArgs d) {
    pdl_allow_next();
    pdl_wait_prev();
    extern __shared__ float dsm[];
    const int n = blockIdx.y;
    int t = blockIdx.x;
    const int tw = t % d.tiles_w; t /= d.tiles_w;
    const int th = t % d.tiles_h; t /= d.tiles_h;
    const int tc = t;
    const int c0 = tc * d.tile_c, p0 = th * d.tile_h, q0 = tw * d.tile_w;
    const int nc = min(d.tile_c, d.C - c0);
    const int in_hw = d.in_h * d.in_w;
    const int RS = d.R * d.S;
    float* s_in = dsm;                                   // [tile_c][in_h][in_w]
    float* s_w = dsm + (size_t)d.tile_c * in_hw;         // [tile_c][R*S]
    float* s_b = s_w + (size_t)d.tile_c * RS;            // [tile_c]
    const int ih0 = p0 * d.sh - d.ph, iw0 = q0 * d.sw - d.pw;

    for (int i = threadIdx.x; i < nc * in_hw; i += blockDim.x) {
        const int c = i / in_hw, rem = i - c * in_hw;
        const int r = rem / d.in_w, col = rem - r * d.in_w;
        const int ih = ih0 + r, iw = iw0 + col;
        float v = 0.f;
        if (ih >= 0 && ih < d.H && iw >= 0 && iw < d.W)
            v = __ldg(d.x + (((long long)n * d.C + c0 + c) * d.H + ih) * d.W + iw);
        s_in[i] = v;
    }
    for (int i = threadIdx.x; i < nc * RS; i += blockDim.x) s_w[i] = __ldg(d.w + (long long)c0 * RS + i);
    for (int i = threadIdx.x; i < nc; i += blockDim.x) s_b[i] = d.bias ? __ldg(d.bias + c0 + i) : 0.f;
    __syncthreads();

    const int groups_w = d.tile_w / d.items;             // tile_w is a multiple of items
    const int work = nc * d.tile_h * groups_w;
    for (int i = threadIdx.x; i < work; i += blockDim.x) {
        const int gwi = i % groups_w;
        const int rest = i / groups_w;
        const int r = rest % d.tile_h, c = rest / d.tile_h;
        const int p = p0 + r, q = q0 + gwi * d.items;
        if (p >= d.P || q >= d.Q) continue;
        float acc[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] = s_b[c];
        const float* wi = s_w + c * RS;
        const float* xi = s_in + c * in_hw + (r * d.sh) * d.in_w + gwi * d.items * d.sw;
        for (int fr = 0; fr < d.R; ++fr) {
            for (int fs = 0; fs < d.S; ++fs) {
                const float wv = wi[fr * d.S + fs];
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (j < d.items) acc[j] = fmaf(xi[fr * d.in_w + fs + j * d.sw], wv, acc[j]);
            }
        }
        float* yo = d.y + (((long long)n * d.C + c0 + c) * d.P + p) * d.Q + q;
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] = apply_act(acc[j], d.act);
        if (d.vec == 4 && q + d.items <= d.Q) {
#pragma unroll
            for (int j = 0; j < 8; j += 4)
                if (j < d.items) *reinterpret_cast<float4*>(yo + j) = make_float4(acc[j], acc[j + 1], acc[j + 2], acc[j + 3]);
        } else if (d.vec == 2 && q + d.items <= d.Q) {
#pragma unroll
            for (int j = 0; j < 8; j += 2)
                if (j < d.items) *reinterpret_cast<float2*>(yo + j) = make_float2(acc[j], acc[j + 1]);
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (j < d.items && q + j < d.Q) yo[j] = acc[j];
        }
    }
}

// ------------------------------------------------------------------------------------------------------------
// DW_SIMT, register-window form (3x3 and 5x5 filters, stride 1 or 2).  A thread owns a strip of ROWS output rows
// x 4 or 8 consecutive output columns of one channel.  It walks the (ROWS-1)*STRIDE + R input rows the strip needs
// once: of each row it fetches 3*STRIDE + R values (aligned 16-byte loads for the columns under the strip when the
// image rows allow it, 4-byte loads for the ragged edges; neighbouring strips' loads meet in L1) and feeds every
// output row whose window contains that input row, so an input value is read once per strip and no shared
// memory or barrier is involved.  Bound by HBM: the only DRAM traffic is x once, y once.
// ------------------------------------------------------------------------------------------------------------
template <int R, int STRIDE, int ROWS, int WIDTH>
__global__ void __launch_bounds__(256, WIDTH == 4 ? 6 : 4) tt_dwconv_window_kernel(const DwArgs d) {
    constexpr int NCOL = (WIDTH - 1) * STRIDE + R;        // input columns under a WIDTH-wide strip
    constexpr int IN_ROWS = (ROWS - 1) * STRIDE + R;
    constexpr int PAD = R / 2;                            // "same" padding: the launcher checks it
    constexpr int NV = (NCOL - PAD) / 4;                  // aligned 16-byte groups per window row
    pdl_allow_next();
    pdl_wait_prev();
    const int n = blockIdx.y;
    int t = blockIdx.x;
    const int tw = t % d.tiles_w; t /= d.tiles_w;
    const int th = t % d.tiles_h; t /= d.tiles_h;
    const int c0 = t * d.tile_c, p0 = th * d.tile_h, q0 = tw * d.tile_w;
    const int nc = min(d.tile_c, d.C - c0);
    const int groups_w = d.tile_w / WIDTH;
    const int groups_h = (d.tile_h + ROWS - 1) / ROWS;
    const int work = nc * groups_h * groups_w;
    for (int i = threadIdx.x; i < work; i += blockDim.x) {
        const int gwi = i % groups_w;
        const int rest = i / groups_w;
        const int gh = rest % groups_h, cl = rest / groups_h;
        const int p = p0 + gh * ROWS, q = q0 + gwi * WIDTH;
        if (p >= d.P || q >= d.Q || gh * ROWS >= d.tile_h) continue;
        const int c = c0 + cl;
        const float* __restrict__ xc = d.x + ((long long)n * d.C + c) * d.H * (long long)d.W;
        const float* __restrict__ wc = d.w + (long long)c * (R * R);
        float wv[R * R];
#pragma unroll
        for (int k = 0; k < R * R; ++k) wv[k] = __ldg(wc + k);
        const float b = d.bias ? __ldg(d.bias + c) : 0.f;
        float acc[ROWS][WIDTH];
#pragma unroll
        for (int ro = 0; ro < ROWS; ++ro)
#pragma unroll
            for (int j = 0; j < WIDTH; ++j) acc[ro][j] = b;
        const int ih0 = p * STRIDE - PAD, iw0 = q * STRIDE - PAD;
#pragma unroll
        for (int ri = 0; ri < IN_ROWS; ++ri) {
            const int ih = ih0 + ri;
            float v[NCOL];
#pragma unroll
            for (int j = 0; j < NCOL; ++j) v[j] = 0.f;
            if ((unsigned)ih < (unsigned)d.H) {
                const float* __restrict__ xr = xc + (long long)ih * d.W;
                if (d.vec_in) {
                    // window slots [PAD, PAD + 4*NV) lie under the strip and start on a 16-byte boundary; a group
                    // of four columns is inside the row or outside it as a whole (W % 4 == 0)
#pragma unroll
                    for (int k = 0; k < NV; ++k) {
                        const int col = iw0 + PAD + 4 * k;
                        if (col < d.W) {
                            const float4 f = __ldg(reinterpret_cast<const float4*>(xr + col));
                            v[PAD + 4 * k] = f.x; v[PAD + 4 * k + 1] = f.y; v[PAD + 4 * k + 2] = f.z; v[PAD + 4 * k + 3] = f.w;
                        }
                    }
#pragma unroll
                    for (int j = 0; j < NCOL; ++j) {
                        if (j >= PAD && j < PAD + 4 * NV) continue;
                        const int col = iw0 + j;
                        if ((unsigned)col < (unsigned)d.W) v[j] = __ldg(xr + col);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < NCOL; ++j) {
                        const int col = iw0 + j;
                        if ((unsigned)col < (unsigned)d.W) v[j] = __ldg(xr + col);
                    }
                }
            }
#pragma unroll
            for (int ro = 0; ro < ROWS; ++ro) {
                const int fr = ri - ro * STRIDE;              // compile-time after unrolling
                if (fr >= 0 && fr < R) {
#pragma unroll
                    for (int fs = 0; fs < R; ++fs)
#pragma unroll
                        for (int j = 0; j < WIDTH; ++j) acc[ro][j] = fmaf(v[j * STRIDE + fs], wv[fr * R + fs], acc[ro][j]);
                }
            }
        }
        float* __restrict__ yc = d.y + (((long long)n * d.C + c) * d.P + p) * (long long)d.Q + q;
#pragma unroll
        for (int ro = 0; ro < ROWS; ++ro) {
            if (p + ro >= d.P || gh * ROWS + ro >= d.tile_h) break;
            float* yo = yc + (long long)ro * d.Q;
#pragma unroll
            for (int j0 = 0; j0 < WIDTH; j0 += 4) {
                float o[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) o[j] = apply_act(acc[ro][j0 + j], d.act);
                if (d.vec == 4 && q + j0 + 4 <= d.Q) {
                    *reinterpret_cast<float4*>(yo + j0) = make_float4(o[0], o[1], o[2], o[3]);
                } else if (d.vec == 2 && q + j0 + 4 <= d.Q) {
                    *reinterpret_cast<float2*>(yo + j0) = make_float2(o[0], o[1]);
                    *reinterpret_cast<float2*>(yo + j0 + 2) = make_float2(o[2], o[3]);
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if (q + j0 + j < d.Q) yo[j0 + j] = o[j];
                }
            }
        }
    }
}

// The tiles of the persistent depthwise kernels: (channel group, image, row tile, column tile).  A CTA keeps its channel group, and
// with it the filters.  step > 0: CTA b has group b % groups and every step-th of its other coordinates, so that the CTAs work
// on neighbouring planes at any time; step = 0: consecutive ranges of all tiles, counted groups first (the launcher's choice).
struct DwTile { int ct, n, th, tw; };
struct DwWalk { DwTile first; int count, s_n, s_th, s_tw; };
__device__ __forceinline__ DwWalk dw_walk(const DwArgs& d) {
    DwWalk w;
    const int per_image = d.tiles_h * d.tiles_w, per_ct = d.N * per_image;
    int j;
    if (d.step) {
        const int groups = (d.C + d.tile_c - 1) / d.tile_c;
        j = (int)blockIdx.x / groups;
        w.first.ct = (int)blockIdx.x - j * groups;
        w.count = j < per_ct ? (per_ct - j + d.step - 1) / d.step : 0;
        w.s_n = d.step / per_image;
        const int rem = d.step - w.s_n * per_image;
        w.s_th = rem / d.tiles_w; w.s_tw = rem - w.s_th * d.tiles_w;
    } else {
        const int t0 = (int)((long long)d.total_tiles * blockIdx.x / gridDim.x);
        w.count = (int)((long long)d.total_tiles * (blockIdx.x + 1) / gridDim.x) - t0;
        w.first.ct = t0 / per_ct;
        j = t0 - w.first.ct * per_ct;
        w.s_n = per_image == 1 ? 1 : 0; w.s_th = per_image > 1 && d.tiles_w == 1 ? 1 : 0; w.s_tw = d.tiles_w > 1 ? 1 : 0;
    }
    w.first.n = j / per_image; j -= w.first.n * per_image;
    w.first.th = j / d.tiles_w; w.first.tw = j - w.first.th * d.tiles_w;
    return w;
}
__device__ __forceinline__ void dw_next(const DwArgs& d, const DwWalk& w, DwTile& t) {
    t.tw += w.s_tw; t.th += w.s_th; t.n += w.s_n;
    if (t.tw >= d.tiles_w) { t.tw -= d.tiles_w; ++t.th; }
    if (t.th >= d.tiles_h) { t.th -= d.tiles_h; ++t.n; }
    if (t.n >= d.N && d.step == 0) { t.n = 0; ++t.ct; }
}

// ------------------------------------------------------------------------------------------------------------
// DW_SIMT, TMA-staged persistent form (3x3 and 5x5 "same" filters, stride 1 or 2, image rows of 16-byte multiples).
// The image is one 3-D tensor (W, H, planes = N * C).  A tile is tile_c consecutive planes x tile_h x tile_w
// outputs; its input box [tile_c][in_h][box_w] starts 4 columns left of the tile (a 16-byte aligned coordinate) and
// PAD rows above it, and the TMA zero fill supplies the padding, so the compute loop has no bounds test on inputs.
// CTAs walk the tiles persistently with `stages` boxes in flight: no thread waits on a global load, which is what
// limits the register-window kernel.  Threads work on ROWS x WIDTH strips exactly as there, reading the window rows
// with aligned 16-byte shared-memory loads.  Same FMAs in the same order: bit-identical outputs.
// The instruction stream per output is what bounds this kernel next to the memory system, so everything that does
// not depend on the plane is hoisted: a thread keeps its strip position for the whole kernel, and the tiles are counted channels
// first, so that a CTA meets new filters once or twice, mostly once: they stay in registers where a thread has one plane, else in a shared-memory buffer ([tile_c][WP] floats: filter, bias, padding).
// A CTA has no more threads than a tile has strips, so more CTAs fit; the order of the lanes and the row pitch keep a warp's reads
// off the same banks.  240 x 28 x 28, 5x5, 256 images: 109 -> 85 us (HBM 59), bound by issue; 200 x 56 x 56, 5x5
// stride 2, 32 images: 31 -> 23 (15); 16 images of 240 x 28 x 28, 5x5: 10.5 -> 9.7.  Stride 2 is compiled for one CTA per SM: its
// strips need 95 registers, held to 64 they spilled (144 x 56 x 56, 3x3: 98 -> 92).
// ------------------------------------------------------------------------------------------------------------
template <int R, int STRIDE, int ROWS, int WIDTH>
__global__ void __launch_bounds__(256, STRIDE == 2 ? 1 : 0) tt_dwconv_tma_kernel(const __grid_constant__ CUtensorMap tmap_x, const DwArgs d) {
    constexpr int NCOL = (WIDTH - 1) * STRIDE + R;
    constexpr int IN_ROWS = (ROWS - 1) * STRIDE + R;
    constexpr int PAD = R / 2;
    constexpr int FIRST = 4 - PAD;                        // window slot 0 sits this many floats right of the strip's aligned base
    constexpr int NLD = (FIRST + NCOL + 3) / 4;           // aligned 16-byte loads per window row
    constexpr int WP = (R * R + 1 + 3) / 4 * 4;           // floats per plane in a weight buffer
    extern __shared__ uint8_t dw_raw[];
    __shared__ uint64_t full_bar[4];
    __shared__ int abort_flag;
    const uint32_t base = (smem_u32(dw_raw) + 127u) & ~127u;
    const uint32_t wst = base + (uint32_t)d.tma_stages * (uint32_t)d.stage_bytes;
    volatile int* abortp = &abort_flag;
    pdl_allow_next();
    if (threadIdx.x == 0) {
        for (int s = 0; s < d.tma_stages; ++s) mbar_init(smem_u32(&full_bar[s]), 1u);
        abort_flag = 0;
        fence_mbar_init();
        fence_proxy_async_shared();
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_x) : "memory");
    }
    __syncthreads();
    pdl_wait_prev();                                      // the set-up above touched no global memory
    const DwWalk walk = dw_walk(d);
    DwTile cur = walk.first;
    auto fill = [&](const DwTile& t, int s) {               // thread 0: request a tile's box into buffer s
        if (threadIdx.x != 0) return;
        const uint32_t bar = smem_u32(&full_bar[s]);
        mbar_expect_tx(bar, (uint32_t)(d.tile_c * d.in_h * d.box_w * 4));
        tma_load_3d(base + (uint32_t)s * (uint32_t)d.stage_bytes, &tmap_x, bar, t.tw * d.tile_w * STRIDE - 4,
                    t.th * d.tile_h * STRIDE - PAD, t.n * d.C + t.ct * d.tile_c);
    };
    DwTile ahead = cur;
    for (int i = 0; i < min(walk.count, d.tma_stages); ++i) { fill(ahead, i); dw_next(d, walk, ahead); }
    // a thread's strip position inside a plane is fixed for the whole kernel when a plane has at most blockDim strips
    // (the thread then walks planes cl_f, cl_f + cpp, ...); otherwise it also walks strips
    const int groups_w = d.tile_w / WIDTH;
    const int groups_h = (d.tile_h + ROWS - 1) / ROWS;
    const int spp = groups_h * groups_w;                  // strips per plane
    const bool fixed_pos = spp <= (int)blockDim.x;
    const int cpp = fixed_pos ? (int)blockDim.x / spp : 1;                  // planes per pass
    // neighbouring lanes take the strips of a row, then the plane's next strip row or (plane_next) the next plane's strips:
    // whichever spreads a warp's 16-byte reads over more of the banks
    int cl_f = 0, s_f = (int)threadIdx.x;
    if (fixed_pos && d.plane_next) {
        const int r = (int)threadIdx.x / groups_w;
        cl_f = r % cpp;
        s_f = r / cpp * groups_w + ((int)threadIdx.x - r * groups_w);
    } else if (fixed_pos) {
        cl_f = (int)threadIdx.x / spp;
        s_f = (int)threadIdx.x - cl_f * spp;
    }
    const int s_step = fixed_pos ? spp : (int)blockDim.x;                    // fixed: the strip loop runs once
    const bool active = cl_f < cpp && s_f < spp;
    const int gh_f = s_f / groups_w, gwi_f = s_f - gh_f * groups_w;
    const uint32_t plane_bytes = 4u * (uint32_t)(d.in_h * d.box_w);
    const long long plane_out = (long long)d.P * d.Q;
    const bool clamp = d.act == TT_ACT_RELU || d.act == TT_ACT_RELU6, gelu = d.act == TT_ACT_GELU_ERF;
    const float hi = d.act == TT_ACT_RELU6 ? 6.f : INFINITY;
    const bool keep = d.tile_c <= cpp;                    // one plane per thread: its filter stays in registers
    float wv[WP];
    int s = 0, have_ct = -1;
    uint32_t ph = 0;
    for (int i = 0; i < walk.count; ++i) {
        const int c0 = cur.ct * d.tile_c, ncl = min(d.tile_c, d.C - c0);
        if (cur.ct != have_ct) {                          // the same for every thread
            have_ct = cur.ct;
            if (keep) {
                if (cl_f < ncl) {
                    const float* w = d.w + (long long)(c0 + cl_f) * (R * R);
#pragma unroll
                    for (int k = 0; k < R * R; ++k) wv[k] = __ldg(w + k);
                    wv[R * R] = d.bias ? __ldg(d.bias + c0 + cl_f) : 0.f;
                }
            } else {                                      // (the barrier after the last tile has passed)
                for (int idx = (int)threadIdx.x; idx < ncl * WP; idx += (int)blockDim.x) {
                    const int cl = idx / WP, k = idx - cl * WP;
                    float v = 0.f;
                    if (k < R * R) v = __ldg(d.w + (long long)(c0 + cl) * (R * R) + k);
                    else if (k == R * R && d.bias) v = __ldg(d.bias + c0 + cl);
                    st_shared_f32(wst + 4u * (uint32_t)idx, v);
                }
                __syncthreads();
            }
        }
        // every thread waits for the box itself (all take the same decision: the same barrier and phase)
        if (!mbar_wait(smem_u32(&full_bar[s]), ph, abortp, d.status, 9u, d.wait_ns)) break;
        const int pl0 = cur.n * d.C + c0, p0 = cur.th * d.tile_h, q0 = cur.tw * d.tile_w;
        const uint32_t stage = base + (uint32_t)s * (uint32_t)d.stage_bytes;
        for (int sidx = s_f; active && sidx < spp; sidx += s_step) {
            int gh = gh_f, gwi = gwi_f;
            if (sidx != s_f) { gh = sidx / groups_w; gwi = sidx - gh * groups_w; }
            const int p = p0 + gh * ROWS, q = q0 + gwi * WIDTH;
            if (p >= d.P || q >= d.Q || gh * ROWS >= d.tile_h) continue;
            const int nrows = min(ROWS, min(d.P - p, d.tile_h - gh * ROWS));
            const bool whole = q + WIDTH <= d.Q;
            // the strip's window rows: box row gh*ROWS*STRIDE + ri, from the aligned float WIDTH*gwi*STRIDE on
            const uint32_t soff = stage + 4u * (uint32_t)((gh * ROWS * STRIDE) * d.box_w + WIDTH * gwi * STRIDE);
            float* __restrict__ y0 = d.y + ((long long)pl0 * d.P + p) * (long long)d.Q + q;
#pragma unroll 1
            for (int cl = cl_f; cl < ncl; cl += cpp) {
                if (!keep) {
#pragma unroll
                    for (int k = 0; k < WP / 4; ++k) {
                        const float4 f = ld_shared_v4f(wst + 4u * (uint32_t)(cl * WP + 4 * k));
                        wv[4 * k] = f.x; wv[4 * k + 1] = f.y; wv[4 * k + 2] = f.z; wv[4 * k + 3] = f.w;
                    }
                }
                float acc[ROWS][WIDTH];
#pragma unroll
                for (int ro = 0; ro < ROWS; ++ro)
#pragma unroll
                    for (int j = 0; j < WIDTH; ++j) acc[ro][j] = wv[R * R];
                const uint32_t row0 = soff + (uint32_t)cl * plane_bytes;
#pragma unroll
                for (int ri = 0; ri < IN_ROWS; ++ri) {
                    float u[4 * NLD];
#pragma unroll
                    for (int k = 0; k < NLD; ++k) {
                        const float4 f = ld_shared_v4f(row0 + 4u * (uint32_t)(ri * d.box_w + 4 * k));
                        u[4 * k] = f.x; u[4 * k + 1] = f.y; u[4 * k + 2] = f.z; u[4 * k + 3] = f.w;
                    }
#pragma unroll
                    for (int ro = 0; ro < ROWS; ++ro) {
                        const int fr = ri - ro * STRIDE;          // compile-time after unrolling
                        if (fr >= 0 && fr < R) {
#pragma unroll
                            for (int fs = 0; fs < R; ++fs)
#pragma unroll
                                for (int j = 0; j < WIDTH; ++j) acc[ro][j] = fmaf(u[FIRST + j * STRIDE + fs], wv[fr * R + fs], acc[ro][j]);
                        }
                    }
                }
                float* __restrict__ yc = y0 + (long long)cl * plane_out;
#pragma unroll
                for (int ro = 0; ro < ROWS; ++ro) {
                    if (ro >= nrows) break;
                    if (clamp) {
#pragma unroll
                        for (int j = 0; j < WIDTH; ++j) acc[ro][j] = fminf(fmaxf(acc[ro][j], 0.f), hi);
                    } else if (gelu) {
#pragma unroll
                        for (int j = 0; j < WIDTH; ++j) acc[ro][j] = gelu_erf(acc[ro][j]);
                    }
                    float* yo = yc + (long long)ro * d.Q;
                    if (whole && d.vec == 4) {
#pragma unroll
                        for (int j = 0; j < WIDTH; j += 4)
                            *reinterpret_cast<float4*>(yo + j) = make_float4(acc[ro][j], acc[ro][j + 1], acc[ro][j + 2], acc[ro][j + 3]);
                    } else if (whole && d.vec == 2) {
#pragma unroll
                        for (int j = 0; j < WIDTH; j += 2) *reinterpret_cast<float2*>(yo + j) = make_float2(acc[ro][j], acc[ro][j + 1]);
                    } else {
#pragma unroll
                        for (int j = 0; j < WIDTH; ++j)
                            if (q + j < d.Q) yo[j] = acc[ro][j];
                    }
                }
            }
        }
        __syncthreads();                                  // everyone is done with this box
        if (i + d.tma_stages < walk.count) { fill(ahead, s); dw_next(d, walk, ahead); }
        dw_next(d, walk, cur);
        if (++s == d.tma_stages) { s = 0; ph ^= 1u; }
    }
    // after a tripped wait: let the boxes still in flight land before the shared memory is given back (bounded)
    if (threadIdx.x == 0 && *abortp) {
        for (int b = 0; b < d.tma_stages; ++b) {
            const unsigned long long t0 = global_timer_ns();
            while (!mbar_try_wait(smem_u32(&full_bar[b]), 0u) && !mbar_try_wait(smem_u32(&full_bar[b]), 1u)) {
                if (global_timer_ns() - t0 > 2000000ull) break;
            }
        }
    }
}

// ------------------------------------------------------------------------------------------------------------
// DW_SIMT, run-staged persistent form (3x3 and 5x5 "same" filters, stride 1 or 2, image rows that are no 16-byte multiples, which
// fit no TMA box).  Consecutive planes of an image, or consecutive rows of one plane, are one run of floats: a bulk copy brings it
// in from the 16-byte boundary before it (up to three floats at the tensor's end by cp.async).  Its rows lie packed, so a thread
// takes one output column x ROWS rows and neighbouring lanes neighbouring columns: 4-byte reads without bank conflicts inside a
// row, coalesced stores.  A window column outside the image is a predicate that holds for the strip, a window row outside it is
// read from a row of zeros.  Same products in the same order as the other forms.
// Instruction issue bounds it next to the memory system, so a thread keeps its column, and its channel's filter in registers: the
// tiles are counted channels first, a CTA takes a consecutive range of them and meets a new filter once or twice.
// Even rows: a thread takes two columns, read as pairs; with stride 1 their products are paired too (half the issue slots).
// 256 images, against the register-window form's best record: 480 x 14 x 14, 5x5: 134 -> 57 us (HBM 30); 384 x 14 x 14, 3x3: 61 -> 33
// (24); 576 x 14 x 14, 3x3 stride 2: 53 -> 29 (22); 960 x 7 x 7, 3x3: 44 -> 30 (15); 64 images of 144 x 55 x 55, 3x3: 77 -> 54 (34).
// ------------------------------------------------------------------------------------------------------------
template <int R, int STRIDE, int ROWS, int WIDTH>
__global__ void __launch_bounds__(256, R == 5 && STRIDE == 1 && WIDTH == 2 ? 2 : 3) tt_dwconv_run_kernel(const DwArgs d) {
    constexpr int IN_ROWS = (ROWS - 1) * STRIDE + R;
    constexpr int PAD = R / 2;
    // two columns: window columns are read in pairs from an even one on, each of them inside the image or outside as a whole
    constexpr int LEFT = WIDTH == 2 ? 2 : PAD, FIRST = LEFT - PAD;
    constexpr int NLD = WIDTH == 2 ? (FIRST + STRIDE + R + 1) / 2 : R;
    const int lanes_q = (d.Q + WIDTH - 1) / WIDTH;        // threads of one strip row
    extern __shared__ __align__(128) float dw_floats[];
    __shared__ uint64_t full_bar[4];
    __shared__ int abort_flag;
    const int stage_f = d.stage_bytes / 4, zero_f = d.tma_stages * stage_f;      // after the buffers: the row of zeros
    const uint32_t base = smem_u32(dw_floats);
    volatile int* abortp = &abort_flag;
    pdl_allow_next();
    if (threadIdx.x == 0) {
        // the run's request and the copies of thread 0, or (x not on 16 bytes) of every thread
        for (int s = 0; s < d.tma_stages; ++s) mbar_init(smem_u32(&full_bar[s]), d.vec_in ? 2u : blockDim.x + 1u);
        abort_flag = 0;
        fence_mbar_init();
        fence_proxy_async_shared();
    }
    for (int i = (int)threadIdx.x; i < d.W; i += (int)blockDim.x) dw_floats[zero_f + i] = 0.f;
    __syncthreads();
    pdl_wait_prev();                                      // the set-up above touched no global memory
    const int HW = d.H * d.W;
    const long long all = (long long)d.N * d.C * HW;
    const bool whole = d.tiles_h == 1;                    // tiles of whole planes; otherwise of a band of one plane
    const DwWalk walk = dw_walk(d);
    DwTile cur = walk.first;
    // the run's first float and first image row
    auto start_of = [&](const DwTile& t, int& row0) {
        row0 = whole ? 0 : max(0, t.th * d.tile_h * STRIDE - PAD);
        return ((long long)t.n * d.C + t.ct * d.tile_c) * HW + row0 * d.W;
    };
    auto fill = [&](const DwTile& t, int s) {
        if (d.vec_in && threadIdx.x != 0) return;
        int row0;
        const long long start = start_of(t, row0), first = start & ~3LL;
        const long long end = start + (whole ? min(d.tile_c, d.C - t.ct * d.tile_c) * HW
                                             : (min(d.H, t.th * d.tile_h * STRIDE - PAD + d.in_h) - row0) * d.W);
        const uint32_t bar = smem_u32(&full_bar[s]), dst = base + (uint32_t)s * (uint32_t)d.stage_bytes;
        if (threadIdx.x == 0) {
            const long long split = d.vec_in ? min((end + 3) & ~3LL, all & ~3LL) : first;      // [first, split) in one copy
            const uint32_t bytes = split > first ? (uint32_t)(split - first) * 4u : 0u;
            mbar_expect_tx(bar, bytes);
            if (bytes) bulk_load(dst, d.x + first, bytes, bar);
            if (d.vec_in) for (long long e = max(split, first); e < end; ++e) cp_async_4(dst + 4u * (uint32_t)(e - first), d.x + e);
        }
        if (!d.vec_in) for (long long e = start + (int)threadIdx.x; e < end; e += (int)blockDim.x) cp_async_4(dst + 4u * (uint32_t)(e - first), d.x + e);
        cp_async_arrive(bar);
    };
    DwTile ahead = cur;
    for (int i = 0; i < min(walk.count, d.tma_stages); ++i) { fill(ahead, i); dw_next(d, walk, ahead); }
    // This thread's column q of strip row gh (and gh + strip_rows, ...) of plane pl.  A unit is one strip row of one plane: Q columns.
    // Narrow images put `units_per_warp` of them side by side in a warp, either consecutive ones or ones `unit_far` apart,
    // whichever spreads the reads over more banks; wide ones run on through the warps.
    int pl, gh0, q;
    bool active;
    {
        const int units = d.tile_c * d.strip_rows;
        int u;
        if (d.units_per_warp) {
            const int lane = (int)threadIdx.x & 31, warp = (int)threadIdx.x >> 5, slot = lane / lanes_q;
            q = lane - slot * lanes_q;
            u = d.unit_far ? warp + slot * d.unit_far : warp * d.units_per_warp + slot;
            active = slot < d.units_per_warp && u < units;
        } else {
            u = (int)threadIdx.x / lanes_q; q = (int)threadIdx.x - u * lanes_q;
            active = u < units;
        }
        pl = u / d.strip_rows; gh0 = u - pl * d.strip_rows;
    }
    q *= WIDTH;
    const int col0 = q * STRIDE - LEFT;
    bool in_col[NLD];
#pragma unroll
    for (int k = 0; k < NLD; ++k) in_col[k] = (unsigned)(col0 + k * WIDTH) < (unsigned)d.W;
    const bool pair_out = WIDTH == 2 && d.Q % 2 == 0 && d.vec >= 2;      // d.vec: what y's alignment allows
    const bool clamp = d.act == TT_ACT_RELU || d.act == TT_ACT_RELU6, gelu = d.act == TT_ACT_GELU_ERF;
    const float hi = d.act == TT_ACT_RELU6 ? 6.f : INFINITY;
    float wv[R * R], bias = 0.f;
    int s = 0, have_ct = -1;
    uint32_t ph = 0;
    for (int i = 0; i < walk.count; ++i) {
        const int c = cur.ct * d.tile_c + pl;             // this thread's channel
        const bool mine = active && c < d.C;
        if (cur.ct != have_ct && mine) {
#pragma unroll
            for (int k = 0; k < R * R; ++k) wv[k] = __ldg(d.w + (long long)c * (R * R) + k);
            if (d.bias) bias = __ldg(d.bias + c);
        }
        have_ct = cur.ct;
        if (!mbar_wait(smem_u32(&full_bar[s]), ph, abortp, d.status, 9u, d.wait_ns)) break;
        int row0;
        const int shift = (int)(start_of(cur, row0) & 3LL);
        const int p0 = cur.th * d.tile_h, p_end = min(d.P, p0 + d.tile_h);
        const int x0 = s * stage_f + shift + pl * HW - row0 * d.W + col0;      // image row 0 of this thread's first window column
        float* __restrict__ y0 = d.y + (((long long)cur.n * d.C + c) * d.P) * d.Q + q;
        if (mine) {
#pragma unroll 1
            for (int p = p0 + gh0 * ROWS; p < p_end; p += d.strip_rows * ROWS) {
                float2 acc[ROWS];                         // .y: the second column
#pragma unroll
                for (int ro = 0; ro < ROWS; ++ro) acc[ro] = make_float2(bias, bias);
                const int ih0 = p * STRIDE - PAD;
                int at = x0 + ih0 * d.W;
#pragma unroll
                for (int ri = 0; ri < IN_ROWS; ++ri) {
                    const int r = (unsigned)(ih0 + ri) < (unsigned)d.H ? at : zero_f + col0;
                    at += d.W;
                    float v[NLD * WIDTH];
#pragma unroll
                    for (int k = 0; k < NLD; ++k) {
                        if constexpr (WIDTH == 2) {
                            const float2 f = in_col[k] ? *reinterpret_cast<const float2*>(dw_floats + r + 2 * k) : make_float2(0.f, 0.f);
                            v[2 * k] = f.x; v[2 * k + 1] = f.y;
                        } else v[k] = in_col[k] ? dw_floats[r + k] : 0.f;
                    }
#pragma unroll
                    for (int ro = 0; ro < ROWS; ++ro) {
                        const int fr = ri - ro * STRIDE;  // compile-time after unrolling
                        if (fr >= 0 && fr < R) {
#pragma unroll
                            for (int fs = 0; fs < R; ++fs) {
                                const float w = wv[fr * R + fs];
                                if constexpr (WIDTH == 1) acc[ro].x = fmaf(v[fs], w, acc[ro].x);
                                else if constexpr (STRIDE == 1) acc[ro] = fma_pair(make_float2(v[FIRST + fs], v[FIRST + fs + 1]), make_float2(w, w), acc[ro]);
                                else {
                                    acc[ro].x = fmaf(v[FIRST + fs], w, acc[ro].x);
                                    acc[ro].y = fmaf(v[FIRST + fs + STRIDE], w, acc[ro].y);
                                }
                            }
                        }
                    }
                }
                if (clamp) {
#pragma unroll
                    for (int ro = 0; ro < ROWS; ++ro) {
                        acc[ro].x = fminf(fmaxf(acc[ro].x, 0.f), hi);
                        if (WIDTH == 2) acc[ro].y = fminf(fmaxf(acc[ro].y, 0.f), hi);
                    }
                } else if (gelu) {
#pragma unroll
                    for (int ro = 0; ro < ROWS; ++ro) {
                        acc[ro].x = gelu_erf(acc[ro].x);
                        if (WIDTH == 2) acc[ro].y = gelu_erf(acc[ro].y);
                    }
                }
                float* __restrict__ yo = y0 + p * d.Q;
#pragma unroll
                for (int ro = 0; ro < ROWS; ++ro) {
                    if (p + ro >= p_end) break;
                    if (pair_out) *reinterpret_cast<float2*>(yo + ro * d.Q) = acc[ro];
                    else {
                        yo[ro * d.Q] = acc[ro].x;
                        if (WIDTH == 2 && q + 1 < d.Q) yo[ro * d.Q + 1] = acc[ro].y;
                    }
                }
            }
        }
        __syncthreads();                                  // everyone is done with this run
        if (i + d.tma_stages < walk.count) { fill(ahead, s); dw_next(d, walk, ahead); }
        dw_next(d, walk, cur);
        if (++s == d.tma_stages) { s = 0; ph ^= 1u; }
    }
    cp_async_wait_all();
    // after a tripped wait: let the runs still in flight land before the shared memory is given back (bounded)
    if (threadIdx.x == 0 && *abortp) {
        for (int b = 0; b < d.tma_stages; ++b) {
            const unsigned long long t0 = global_timer_ns();
            while (!mbar_try_wait(smem_u32(&full_bar[b]), 0u) && !mbar_try_wait(smem_u32(&full_bar[b]), 1u)) {
                if (global_timer_ns() - t0 > 2000000ull) break;
            }
        }
    }
}

// ------------------------------------------------------------------------------------------------------------
// ROW_SIMT: softmax(scale * x) per row; `lanes_per_row` threads of one warp share a row.
// ------------------------------------------------------------------------------------------------------------
__global__ void tt_softmax_kernel(const RowArgs a) {
    pdl_allow_next();
    pdl_wait_prev();
    const int lpr = a.lanes_per_row;
    const int sub = threadIdx.x % lpr;
    const long long row = (long long)blockIdx.x * a.rows_per_cta + threadIdx.x / lpr;
    const bool live = row < a.rows;
    const float* xr = a.x + (live ? row : 0) * (long long)a.cols;
    float* yr = a.y + (live ? row : 0) * (long long)a.cols;
    const int vec = a.vec;
    float mx = -INFINITY;
    if (live) {
        for (int j = sub * vec; j < a.cols; j += lpr * vec)
            for (int e = 0; e < vec; ++e) mx = fmaxf(mx, a.scale * __ldg(xr + j + e));
    }
    for (int o = lpr >> 1; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float sum = 0.f;
    if (live) {
        for (int j = sub * vec; j < a.cols; j += lpr * vec)
            for (int e = 0; e < vec; ++e) sum += expf(a.scale * __ldg(xr + j + e) - mx);
    }
    for (int o = lpr >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (live) {
        const float inv = 1.f / sum;
        for (int j = sub * vec; j < a.cols; j += lpr * vec) {
            float o4[4];
            for (int e = 0; e < vec; ++e) o4[e] = expf(a.scale * __ldg(xr + j + e) - mx) * inv;
            if (vec == 4) *reinterpret_cast<float4*>(yr + j) = make_float4(o4[0], o4[1], o4[2], o4[3]);
            else if (vec == 2) *reinterpret_cast<float2*>(yr + j) = make_float2(o4[0], o4[1]);
            else yr[j] = o4[0];
        }
    }
}

// ROW_SIMT, register-resident form: every lane keeps its share of the row (up to NV 16-byte groups) in registers,
// so x is read from memory once and each exponential is computed once.  Rows of up to lanes_per_row * 4 * NV columns
// whose length is a multiple of 4 and whose pointers are 16-byte aligned; other rows take the two kernels around it.
template <int NV>
__global__ void __launch_bounds__(cached_threads(NV)) tt_softmax_cached_kernel(const RowArgs a) {
    pdl_allow_next();
    pdl_wait_prev();
    const int lpr = a.lanes_per_row;
    const int sub = threadIdx.x % lpr;
    const long long row = (long long)blockIdx.x * a.rows_per_cta + threadIdx.x / lpr;
    const bool live = row < a.rows;
    const float4* xr = reinterpret_cast<const float4*>(a.x + (live ? row : 0) * (long long)a.cols);
    float4* yr = reinterpret_cast<float4*>(a.y + (live ? row : 0) * (long long)a.cols);
    const int groups = a.cols >> 2;
    float4 v[NV];
    float mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const int gidx = sub + i * lpr;
        if (live && gidx < groups) {
            v[i] = __ldg(xr + gidx);
            v[i].x *= a.scale; v[i].y *= a.scale; v[i].z *= a.scale; v[i].w *= a.scale;
            mx = fmaxf(mx, fmaxf(fmaxf(v[i].x, v[i].y), fmaxf(v[i].z, v[i].w)));
        }
    }
    for (int o = lpr >> 1; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const int gidx = sub + i * lpr;
        if (live && gidx < groups) {
            v[i].x = expf(v[i].x - mx); v[i].y = expf(v[i].y - mx); v[i].z = expf(v[i].z - mx); v[i].w = expf(v[i].w - mx);
            sum += (v[i].x + v[i].y) + (v[i].z + v[i].w);
        }
    }
    for (int o = lpr >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const float inv = 1.f / sum;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const int gidx = sub + i * lpr;
        if (live && gidx < groups) yr[gidx] = make_float4(v[i].x * inv, v[i].y * inv, v[i].z * inv, v[i].w * inv);
    }
}

// ROW_SIMT for ragged rows (the length is no multiple of 4, so rows begin anywhere inside a 16-byte group): a warp owns
// `chunk` consecutive rows, whose values are a multiple of four (even rows in twos, others in fours), so that their bytes begin on a
// 16-byte boundary and fill whole groups.
// One bulk copy brings them to shared memory, the lanes read them value by value (NV per lane, kept in registers), write
// the results over them, and one bulk copy takes them back: memory sees whole lines only.  Warps do not meet.
// Next to memory the instructions per value bind (4-byte accesses; the exponential alone is half a dozen), so NV is the
// exact number of values per lane up to 32 and only the last of them is guarded.  (Even counts only, the last two guarded: 5 to
// 13 % slower up to 8 values, 45.8 -> 49.3 us for rows of 197 with 7; 5 % at 13 and 25; the same at 16 and 32.)
// 151296 rows of 197 columns: 136 us in three passes of 4-byte accesses from memory, 57 us with guards on every value,
// 38 us this way (6.3 TB/s; floor 36 us).
constexpr int kRaggedExact = 32;                         // values per lane up to which there is an instantiation for each count
template <int NV>
__global__ void __launch_bounds__(ragged_threads(NV)) tt_softmax_ragged_kernel(const RowArgs a, int chunk) {
    extern __shared__ __align__(16) float sm_rows[];
    __shared__ uint64_t landed[32];
    pdl_allow_next();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t bar = smem_u32(&landed[warp]);
    if (lane == 0) {
        mbar_init(bar, 1u);
        fence_proxy_async_shared();
    }
    __syncwarp();
    pdl_wait_prev();
    const long long row0 = ((long long)blockIdx.x * (blockDim.x >> 5) + warp) * chunk;
    if (row0 >= a.rows) return;
    const int rows = (int)min((long long)chunk, a.rows - row0);
    float* buf = sm_rows + (size_t)warp * chunk * a.cols;
    const float* x = a.x + row0 * a.cols;
    float* y = a.y + row0 * a.cols;
    const int n = rows * a.cols;
    const bool whole = rows == chunk;                    // the last rows of the tensor may be no whole groups
    if (whole) {
        if (lane == 0) {
            mbar_expect_tx(bar, 4u * (uint32_t)n);
            bulk_load(smem_u32(buf), x, 4u * (uint32_t)n, bar);
        }
        // the copy reads this launch's own x: it lands within microseconds or not at all; the limit only keeps a lost one from spinning
        const unsigned long long t0 = global_timer_ns();
        while (!mbar_try_wait(bar, 0u)) if (global_timer_ns() - t0 > a.wait_ns) { if (lane == 0) atomicCAS(a.status, 0u, (unsigned)TT_ERR_TIMEOUT); return; }
    } else {
        for (int i = lane; i < n; i += 32) buf[i] = __ldg(x + i);
        __syncwarp();
    }
    const int lpr = a.lanes_per_row, sub = lane % lpr, per_pass = 32 / lpr;
    for (int r0 = 0; r0 < rows; r0 += per_pass) {
        const int r = r0 + lane / lpr;
        const bool live = r < rows;
        float* row = buf + (live ? r : 0) * a.cols;
        float v[NV];
        float mx = -INFINITY;
        const int guard = NV <= kRaggedExact ? NV - 1 : 0;   // values from here on may lie past the end of the row
        row += sub;
        const int left = a.cols - sub;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            v[i] = i < guard || i * lpr < left ? row[i * lpr] * a.scale : -INFINITY;
            mx = fmaxf(mx, v[i]);
        }
        for (int o = lpr >> 1; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        float sum = 0.f;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            v[i] = expf(v[i] - mx);
            sum += i < guard || i * lpr < left ? v[i] : 0.f;
        }
        for (int o = lpr >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        const float inv = 1.f / sum;
        if (live) {
#pragma unroll
            for (int i = 0; i < NV; ++i)
                if (i < guard || i * lpr < left) row[i * lpr] = v[i] * inv;
        }
    }
    if (whole) {
        fence_proxy_async_shared();                      // the lanes' stores -> visible to the bulk copy
        __syncwarp();
        if (lane == 0) {
            bulk_store(y, smem_u32(buf), 4u * (uint32_t)n);
            bulk_stores_read();
        }
    } else {
        __syncwarp();
        for (int i = lane; i < n; i += 32) y[i] = buf[i];
    }
}

// A kernel that does nothing, for the launch floor: launched with a record's grid, block size, shared memory,
// cluster shape and dependent-launch attribute, its time is what a launch of that record costs before any work.
__global__ void tt_floor_kernel() {
    pdl_allow_next();
    pdl_wait_prev();
}

// ------------------------------------------------------------------------------------------------------------
// Launchers (called from tt_device.cu)
// ------------------------------------------------------------------------------------------------------------
// Two CTAs fit one SM when each takes at most half of its shared memory (228 KB, of which 1 KB per CTA is the
// system's, plus the kernel's static part) and half of its 512 tensor-memory columns.
static bool gemm_two_per_sm(int smem_bytes, int tmem_cols) { return smem_bytes <= 112 * 1024 && tmem_cols <= 256; }

typedef void (*GemmKernel)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const GemmArgs, const ChainParam<false>);
// (compensated products from tensor memory have one CTA per SM)
#define TT_GEMM_FORMS(CTAS, CL, X3_TMEM) {tt_gemm_tc_kernel<CTAS, kFormTma, CL>, tt_gemm_tc_kernel<CTAS, kFormMn, CL>, tt_gemm_tc_kernel<CTAS, kFormIm2col, CL>, \
    tt_gemm_tc_kernel<CTAS, kFormGather, CL>, tt_gemm_tc_kernel<CTAS, kFormX3, CL>, X3_TMEM, tt_gemm_tc_kernel<CTAS, kFormIm2colRun, CL>, \
    tt_gemm_tc_kernel<CTAS, kFormRaw, CL>}
static const GemmKernel kGemmKernels[2][2][8] = {
    {TT_GEMM_FORMS(1, false, (tt_gemm_tc_kernel<1, kFormX3Tmem, false>)), TT_GEMM_FORMS(1, true, (tt_gemm_tc_kernel<1, kFormX3Tmem, true>))},
    {TT_GEMM_FORMS(2, false, nullptr), TT_GEMM_FORMS(2, true, nullptr)}};
#undef TT_GEMM_FORMS

static int gemm_form(const GemmArgs& g) {
    if (g.x3) return g.x3_bufs > 0 ? kFormX3Tmem : kFormX3;
    if (g.a_mode == OPM_IM2COL || g.b_mode == OPM_IM2COL) return g.slab_tma == 2 ? kFormIm2colRun : kFormIm2col;
    const bool a = g.a_mode == OPM_TMA || g.a_mode == OPM_TMA_MN, b = g.b_mode == OPM_TMA || g.b_mode == OPM_TMA_MN;
    if (!a || !b) return g.a_mode == OPM_RAW || g.b_mode == OPM_RAW ? kFormRaw : kFormGather;
    return g.a_mode == OPM_TMA && g.b_mode == OPM_TMA ? kFormTma : kFormMn;
}

// Which instantiation a plan runs; its shared-memory limit is raised once per device.  Which build (two CTAs per SM) is the
// record's choice (ctas_per_sm), resolved by the legaliser.
static cudaError_t gemm_kernel_for(const GemmArgs& g, int smem_bytes, GemmKernel* out) {
    static OncePerDevice raised[2][2][8];
    const int two = g.two_per_sm && gemm_two_per_sm(smem_bytes, g.tmem_cols), form = gemm_form(g), cl = g.cluster > 0;
    *out = kGemmKernels[two][cl][form];
    return raised[two][cl][form]([&] { return cudaFuncSetAttribute(*out, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit); });
}

// A launch of the one-tile form, `layers` of them along grid.z where that is more than the plan's batch.
template <bool CHAIN>
static cudaError_t launch_one_tile(void (*kern)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const GemmArgs, const ChainParam<CHAIN>),
                                   const tt_apply_info& I, int smem_bytes, int layers, const GemmArgs& g, const ChainParam<CHAIN>& chain,
                                   const void* tmap_a, const void* tmap_b, const void* tmap_x, cudaStream_t st) {
    CUtensorMap ta, tb, tx;
    memcpy(&ta, tmap_a, sizeof ta);
    memcpy(&tb, tmap_b, sizeof tb);
    memcpy(&tx, tmap_x, sizeof tx);
    dim3 grid(I.grid_x, I.grid_y, layers > 1 ? layers : I.grid_z);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = dim3(kGemmThreads, 1, 1); cfg.dynamicSmemBytes = (size_t)smem_bytes; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n_attr = 0;
    // the kernel's set-up may overlap the tail of the kernel before it in the stream (it waits before its first
    // global access); captured into a graph this becomes a programmatic dependency edge
    attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
    ++n_attr;
    if (g.cluster) {
        // the splits of one output tile (grid.y) form a thread-block cluster
        attr[n_attr].id = cudaLaunchAttributeClusterDimension;
        attr[n_attr].val.clusterDim.x = 1; attr[n_attr].val.clusterDim.y = (unsigned)g.cluster; attr[n_attr].val.clusterDim.z = 1;
        ++n_attr;
    }
    cfg.attrs = attr; cfg.numAttrs = (unsigned)n_attr;
    return cudaLaunchKernelEx(&cfg, kern, ta, tb, tx, g, chain);
}

cudaError_t launch_gemm(const tt_apply_info& I, int smem_bytes, const GemmArgs& g, const void* tmap_a, const void* tmap_b, const void* tmap_x,
                        cudaStream_t st) {
    GemmKernel kern;
    const cudaError_t e = gemm_kernel_for(g, smem_bytes, &kern);
    if (e != cudaSuccess) return e;
    return launch_one_tile<false>(kern, I, smem_bytes, 1, g, ChainParam<false>{}, tmap_a, tmap_b, tmap_x, st);
}

// The same with what a chained pass adds (both operands K-major by TMA, one CTA per SM).  tmap_x, tmap_z: the weights of a group's
// second and third layer.
cudaError_t launch_gemm_chain(const tt_apply_info& I, int smem_bytes, const GemmArgs& g, const ChainArgs& c, const void* tmap_a, const void* tmap_b,
                              const void* tmap_x, const void* tmap_z, cudaStream_t st) {
    static OncePerDevice raised;
    const auto alone = tt_gemm_tc_kernel<1, kFormTma, false, true>, cluster = tt_gemm_tc_kernel<1, kFormTma, true, true>;
    const cudaError_t ready = raised([&] {
        const cudaError_t e = cudaFuncSetAttribute(alone, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit);
        return e != cudaSuccess ? e : cudaFuncSetAttribute(cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit);
    });
    if (ready != cudaSuccess) return ready;
    ChainParam<true> p;
    memcpy(&p.tmap_z, tmap_z, sizeof p.tmap_z);
    p.a = c;
    return launch_one_tile<true>(g.cluster ? cluster : alone, I, smem_bytes, c.group, g, p, tmap_a, tmap_b, tmap_x, st);
}

typedef void (*PsKernel)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, const GemmArgs);
static const PsKernel kPs[3][2] = {{tt_gemm_ps_kernel<1, false, false>, tt_gemm_ps_kernel<1, false, true>},
                                   {tt_gemm_ps_kernel<1, true, false>, tt_gemm_ps_kernel<1, true, true>},
                                   {tt_gemm_ps_kernel<2, false, false>, tt_gemm_ps_kernel<2, false, true>}};

// The persistent form: one CTA (or one pair of CTAs, as a cluster of two) per SM.
cudaError_t launch_gemm_ps(const tt_apply_info& I, const GemmArgs& g, const TmapPair& maps, cudaStream_t st) {
    static OncePerDevice raised;
    const cudaError_t ready = raised([] {
        cudaError_t e = cudaSuccess;
        for (const PsKernel kern : {kPs[0][0], kPs[0][1], kPs[1][0], kPs[1][1], kPs[2][0], kPs[2][1]})
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit);
        return e;
    });
    if (ready != cudaSuccess) return ready;
    int dev = 0, sm_count = 0;
    cudaGetDevice(&dev);
    const cudaError_t counted = cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev);
    if (counted != cudaSuccess) return counted;
    CUtensorMap ta, tb, ty, tr;
    memcpy(&ta, maps.a, sizeof ta);
    memcpy(&tb, maps.b, sizeof tb);
    const int cg = g.cta_group == 2 ? 2 : 1;
    const long long units = std::min<long long>(g.total_tiles, sm_count / cg);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(units * cg), 1, 1); cfg.blockDim = dim3(kGemmThreads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)I.smem_bytes; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n_attr = 0;
    attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
    ++n_attr;
    if (cg == 2) {
        attr[n_attr].id = cudaLaunchAttributeClusterDimension;
        attr[n_attr].val.clusterDim.x = 2; attr[n_attr].val.clusterDim.y = 1; attr[n_attr].val.clusterDim.z = 1;
        ++n_attr;
    }
    cfg.attrs = attr; cfg.numAttrs = (unsigned)n_attr;
    memcpy(&ty, maps.y, sizeof ty);
    memcpy(&tr, maps.r, sizeof tr);
    return cudaLaunchKernelEx(&cfg, kPs[cg == 2 ? 2 : (g.a_mn || g.b_mn ? 1 : 0)][g.epi_tma ? 1 : 0], ta, tb, ty, tr, g);
}

// Can a cluster of a plan's CTAs be resident at all?
cudaError_t gemm_cluster_fits(const GemmArgs& g, int smem_bytes, int* fits) {
    GemmKernel kern;
    cudaError_t e = gemm_kernel_for(g, smem_bytes, &kern);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(1, (unsigned)g.cluster, 1); cfg.blockDim = dim3(kGemmThreads, 1, 1); cfg.dynamicSmemBytes = (size_t)smem_bytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1; attr[0].val.clusterDim.y = (unsigned)g.cluster; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
    if (e != cudaSuccess) return e;
    *fits = n > 0;
    return cudaSuccess;
}

cudaError_t launch_floor(const tt_apply_info& I, int smem_bytes, int cluster, cudaStream_t st) {
    static OncePerDevice raised;
    const cudaError_t ready = raised([] { return cudaFuncSetAttribute(tt_floor_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit); });
    if (ready != cudaSuccess) return ready;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(I.grid_x, I.grid_y, I.grid_z); cfg.blockDim = dim3(I.threads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem_bytes; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    int n_attr = 0;
    attr[n_attr].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n_attr].val.programmaticStreamSerializationAllowed = 1;
    ++n_attr;
    if (cluster) {
        attr[n_attr].id = cudaLaunchAttributeClusterDimension;
        attr[n_attr].val.clusterDim.x = 1; attr[n_attr].val.clusterDim.y = (unsigned)cluster; attr[n_attr].val.clusterDim.z = 1;
        ++n_attr;
    }
    cfg.attrs = attr; cfg.numAttrs = (unsigned)n_attr;
    return cudaLaunchKernelEx(&cfg, tt_floor_kernel);
}

// Launch with programmatic stream serialization (the kernels wait before their first global access): in a stream or
// a captured graph the kernel's launch latency and set-up hide behind its predecessor's tail.
template <typename... KArgs, typename... Args>
static cudaError_t launch_serialized(void (*kern)(KArgs...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, Args&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = dim3(threads, 1, 1); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

// CTAs per channel group; 0: consecutive ranges.  Whole planes are runs of memory of their own and go by ranges, which use every CTA.
// Bands of planes (two tiles and more a plane) lose the memory's locality that way (256 images of 144 x 56 x 56, 3x3: 173 us
// against 154), so there the CTAs keep to neighbouring planes, unless whole groups leave more than an eighth of them idle.
static int dw_step(int ctas, int groups, long long per_group) {
    const long long m = std::min<long long>(ctas / groups, per_group);
    if (m < 1) return 0;
    const long long rounds = (per_group + m - 1) / m;
    return 8 * groups * per_group >= 7 * rounds * ctas ? (int)m : 0;
}

// Calls f with the instantiation that a staged plan runs.
template <typename F>
static cudaError_t with_dw_staged(const DwArgs& dw, F&& f) {
#define TT_DWT_BOX(RR, SS, RO, WI) \
    if (dw.R == RR && dw.sh == SS && dw.window_rows == RO && dw.items == WI) return f(tt_dwconv_tma_kernel<RR, SS, RO, WI>);
#define TT_DWT_RUN(RR, SS, RO) \
    if (dw.R == RR && dw.sh == SS && dw.window_rows == RO && dw.items == 1) return f(tt_dwconv_run_kernel<RR, SS, RO, 1>); \
    if (dw.R == RR && dw.sh == SS && dw.window_rows == RO && dw.items == 2) return f(tt_dwconv_run_kernel<RR, SS, RO, 2>);
#define TT_DWT_FILTER(RR, SS) \
    if (!dw.runs) { \
        TT_DWT_BOX(RR, SS, 1, 4) TT_DWT_BOX(RR, SS, 2, 4) TT_DWT_BOX(RR, SS, 4, 4) TT_DWT_BOX(RR, SS, 1, 8) TT_DWT_BOX(RR, SS, 2, 8) \
    } else { TT_DWT_RUN(RR, SS, 2) TT_DWT_RUN(RR, SS, 4) TT_DWT_RUN(RR, SS, 7) }
    TT_DWT_FILTER(3, 1) TT_DWT_FILTER(3, 2) TT_DWT_FILTER(5, 1) TT_DWT_FILTER(5, 2)
    if (!dw.runs) { TT_DWT_BOX(5, 1, 7, 4) TT_DWT_BOX(5, 2, 7, 4) }
#undef TT_DWT_FILTER
#undef TT_DWT_RUN
#undef TT_DWT_BOX
    return cudaErrorInvalidValue;
}

// When a record is applied: the grid of persistent CTAs, never more than the device holds at once (registers may allow fewer than
// shared memory does; asking costs more than a launch), and the tiles' order.
cudaError_t plan_dw_staged(tt_apply_info& I, DwArgs& dw) {
    int dev = 0, per_sm = 0, sm_count = 0;
    cudaGetDevice(&dev);
    cudaError_t e = cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = with_dw_staged(dw, [&](auto* kern) {
            const cudaError_t raised = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit);
            return raised != cudaSuccess ? raised : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, I.threads, (size_t)I.smem_bytes);
        });
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorLaunchOutOfResources;
    const int groups = (dw.C + dw.tile_c - 1) / dw.tile_c;
    I.grid_x = (int)std::min<long long>(I.grid_x, (long long)sm_count * per_sm);
    dw.step = dw.tiles_h * dw.tiles_w > 1 ? dw_step(I.grid_x, groups, (long long)dw.N * dw.tiles_h * dw.tiles_w) : 0;
    if (dw.step) I.grid_x = dw.step * groups;
    return cudaSuccess;
}

cudaError_t launch_dw_staged(const tt_apply_info& I, const DwArgs& dw, const void* tmap_x, cudaStream_t st) {
    const dim3 grid(I.grid_x, 1, 1);
    return with_dw_staged(dw, [&](auto* kern) {
        if constexpr (std::is_invocable_v<decltype(kern), const CUtensorMap, const DwArgs>) {
            CUtensorMap tx;
            memcpy(&tx, tmap_x, sizeof tx);
            return launch_serialized(kern, grid, (unsigned)I.threads, (size_t)I.smem_bytes, st, tx, dw);
        } else {
            return launch_serialized(kern, grid, (unsigned)I.threads, (size_t)I.smem_bytes, st, dw);
        }
    });
}

cudaError_t launch_dw(const tt_apply_info& I, const DwArgs& dw, cudaStream_t st) {
    static OncePerDevice raised;
    const cudaError_t ready = raised([] { return cudaFuncSetAttribute(tt_dwconv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit); });
    if (ready != cudaSuccess) return ready;
    dim3 grid(I.grid_x, I.grid_y, 1);
    if (dw.window_rows > 0) {
        // register-window kernels: one instantiation per (filter size, stride, output rows per thread)
#define TT_DW_CASE(RR, SS, RO, WD) \
        if (dw.R == RR && dw.sh == SS && dw.window_rows == RO && dw.items == WD) return launch_serialized(tt_dwconv_window_kernel<RR, SS, RO, WD>, grid, (unsigned)I.threads, 0, st, dw);
        TT_DW_CASE(3, 1, 1, 4) TT_DW_CASE(3, 1, 2, 4) TT_DW_CASE(3, 1, 4, 4)
        TT_DW_CASE(3, 2, 1, 4) TT_DW_CASE(3, 2, 2, 4) TT_DW_CASE(3, 2, 4, 4)
        TT_DW_CASE(5, 1, 1, 4) TT_DW_CASE(5, 1, 2, 4) TT_DW_CASE(5, 1, 4, 4)
        TT_DW_CASE(5, 2, 1, 4) TT_DW_CASE(5, 2, 2, 4) TT_DW_CASE(5, 2, 4, 4)
        TT_DW_CASE(3, 1, 1, 8) TT_DW_CASE(3, 1, 2, 8) TT_DW_CASE(3, 2, 1, 8) TT_DW_CASE(3, 2, 2, 8)
        TT_DW_CASE(5, 1, 1, 8) TT_DW_CASE(5, 1, 2, 8) TT_DW_CASE(5, 2, 1, 8) TT_DW_CASE(5, 2, 2, 8)
#undef TT_DW_CASE
        return cudaErrorInvalidValue;
    }
    return launch_serialized(tt_dwconv_kernel, grid, (unsigned)I.threads, (size_t)I.smem_bytes, st, dw);
}

template <int NV>
static cudaError_t launch_row_ragged(const tt_apply_info& I, const RowArgs& row, cudaStream_t st) {
    static OncePerDevice raised;
    const cudaError_t ready = raised([] { return cudaFuncSetAttribute(tt_softmax_ragged_kernel<NV>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRowSmem); });
    if (ready != cudaSuccess) return ready;
    return launch_serialized(tt_softmax_ragged_kernel<NV>, dim3((unsigned)I.grid_x, 1, 1), (unsigned)I.threads, (size_t)I.smem_bytes, st, row, row.chunk);
}
typedef cudaError_t (*RaggedLauncher)(const tt_apply_info&, const RowArgs&, cudaStream_t);
template <int... I>
static RaggedLauncher ragged_launcher(int per_lane, std::integer_sequence<int, I...>) {
    static const RaggedLauncher exact[] = {launch_row_ragged<I + 1>...};
    return exact[per_lane - 1];
}

cudaError_t launch_row(const tt_apply_info& I, const RowArgs& row, cudaStream_t st) {
    if (row.cached > 0) {
        const dim3 grid(I.grid_x, 1, 1);
        if (row.cached == 1) return launch_serialized(tt_softmax_cached_kernel<1>, grid, (unsigned)I.threads, 0, st, row);
        if (row.cached == 2) return launch_serialized(tt_softmax_cached_kernel<2>, grid, (unsigned)I.threads, 0, st, row);
        if (row.cached <= 4) return launch_serialized(tt_softmax_cached_kernel<4>, grid, (unsigned)I.threads, 0, st, row);
        if (row.cached <= 8) return launch_serialized(tt_softmax_cached_kernel<8>, grid, (unsigned)I.threads, 0, st, row);
        return launch_serialized(tt_softmax_cached_kernel<kCachedMost>, grid, (unsigned)I.threads, 0, st, row);
    } else if (row.chunk > 0) {
        const int per_lane = (row.cols + row.lanes_per_row - 1) / row.lanes_per_row;
        if (per_lane <= kRaggedExact) return ragged_launcher(per_lane, std::make_integer_sequence<int, kRaggedExact>{})(I, row, st);
        if (per_lane <= 48) return launch_row_ragged<48>(I, row, st);
        return launch_row_ragged<kRaggedMost>(I, row, st);
    }
    const unsigned grid = (unsigned)((row.rows + row.rows_per_cta - 1) / row.rows_per_cta);
    return launch_serialized(tt_softmax_kernel, dim3(grid, 1, 1), (unsigned)(row.rows_per_cta * row.lanes_per_row), 0, st, row);
}

}  // namespace tt
