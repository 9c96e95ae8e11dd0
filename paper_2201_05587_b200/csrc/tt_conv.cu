// conv2d with the reduction walked by blocks of 32 channels and, inside a block, tap by tap (records with k_order = 1).
//
// kind::tf32 wants the reduction index contiguous in shared memory, an NCHW image has the pixels contiguous.  Expanding the
// im2col operand costs one shared-memory access per element and tap; here every input value is turned around ONCE per
// 32-channel block and tile, into a pixel-major slab (one 128-byte line of 32 channels per position, swizzled like a TMA
// tile), and the operand of tap (r, s) is that slab read a constant number of lines further on: only the start address of
// the descriptor changes.
//
// The columns of the contraction are the output positions of the whole batch, numbered
//     n = (image * hp + row) * wp + column,
// with wp and hp so much larger than the output that a tap which reaches past the edge of an image row (or of an image) lands
// on positions that hold zeros: the right padding of a row is the left padding of the next, and the rows between two images
// pad both.  Columns that are no outputs are computed and dropped.  Tiles cross rows and images, so a batch of 7 x 7 images
// fills tiles as well as one of 56 x 56 (overhead (wp * hp) / (P * Q): 1.31 and 1.04 for a padded 3x3).
// A stride > 1 splits the image by the parity of its padded coordinates: taps of one parity class read one sub-image
// ("plane") at unit stride, and the reduction walks (channel block, plane, tap of the plane).
//
// Filters (re-packed to [filter][channel block][tap in walk order][32], a small kernel per weight pointer) ride the 128 rows of
// the accumulator and arrive by TMA, up to taps_per_stage taps of 16 KB per pipeline stage.
// Warps: 0 TMA, 1 MMA issuer + tensor-memory owner, 2-9 bring the slab in, 10-13 read out.
//
// CTAs walk tiles with two accumulators, so that a tile is read out while the next one is multiplied; the slab has two
// buffers and the loads of a block run while the block before it is multiplied.  The slab warps load from global memory
// straight into registers (32 channels of 32 positions in flight per warp) and store 16 bytes per lane without conflicts: no
// staging buffer, no alignment asked of the image rows.
// Where all tiles are resident at once there is nothing to overlap with: then the slab warps help to read out, and a cluster of
// CTAs (the record's cta_group) may share a tile's channel blocks: each leaves the blocks of its accumulator that another CTA
// finishes in scratch memory, and every CTA adds up its blocks, in CTA order, after the cluster's barrier.
//
// Bound by shared memory in the multiply phase: a tap moves its filters in and out (2 * 128 lines of 128 bytes), its columns
// and its share of the slab, 500 cycles measured for 192 columns that take the tensor core 384.  The rest is the prologue
// (launch, first slab and filters: 2 us) and the read-out of the last tile (2.3 us, all CTAs storing at once).
// Measured, before (one tile per CTA and image, TMA-staged slab) and now: 3x3 128 -> 128 at 28 x 28, batch 32, 20.8 -> 17.4 us;
// 3x3 512 -> 512 at 7 x 7 with residual, batch 32, 53.6 (expanded im2col) -> 23.7 us; 3x3 32 -> 248 at 56 x 56, batch 5,
// 16.6 -> 11.3 us.
#include <cuda_runtime.h>
#include <cuda.h>
#include <algorithm>
#include <cstring>
#include "tt_ptx.cuh"

namespace tt {

constexpr int kPmSlabWarps = 8;
constexpr int kPmEpiWarps = 4;
constexpr int kPmThreads = 32 * (2 + kPmSlabWarps + kPmEpiWarps);
constexpr int kPmPitch = 36;                             // floats per staged row: 16-byte accesses stay conflict-free
constexpr uint32_t kPmBlockBytes = 32 * kPmPitch * 4;
static_assert(kPmBlockBytes == kPmEpiBlockBytes, "the legaliser plans with the same staging block");

// u / d and the remainder for u >= 0; magic = floor(2^32 / d) (2^32 - 1 for d = 1) leaves the quotient at most one short.
__device__ __forceinline__ int div_magic(int u, int d, unsigned magic, int& rem) {
    int q = (int)__umulhi((unsigned)u, magic);
    rem = u - q * d;
    if (rem >= d) { ++q; rem -= d; }
    return q;
}

__global__ void __launch_bounds__(kPmThreads, 1)
tt_conv_pm_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ ConvPmArgs g) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t full_bar[kMaxStages];     // a stage's filters (up to taps_per_stage taps) have landed
    __shared__ uint64_t empty_bar[kMaxStages];    // the multiply-accumulates that read them have completed
    __shared__ uint64_t pm_full[2];               // a slab buffer has been written
    __shared__ uint64_t pm_empty[2];              // every multiply-accumulate that reads it has completed
    __shared__ uint64_t acc_full[2];              // an accumulator holds a finished tile
    __shared__ uint64_t acc_empty[2];             // it has been read out
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    volatile int* abortp = &abort_flag;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int split = g.split;
    const int crank = (int)blockIdx.y;                    // (a cluster is a column of the grid)
    const int unit = (int)blockIdx.x, n_units = (int)gridDim.x;
    const int my_tiles = g.total_tiles > unit ? (g.total_tiles - unit + n_units - 1) / n_units : 0;
    const bool single = g.total_tiles <= n_units;         // all tiles resident at once: no tile follows another on this CTA
    const int cb0 = crank * g.blocks / split, cb1 = (crank + 1) * g.blocks / split;   // this CTA's channel blocks
    const int RS = g.R * g.S, tps = g.taps_per_stage;
    const uint32_t stage_bytes = (uint32_t)tps * kPmTapBytes;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t slab0 = base + g.slab_off;

    if (threadIdx.x == 32) asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_w) : "memory");
    if (threadIdx.x == 0) {
        for (int s = 0; s < g.stages; ++s) { mbar_init(smem_u32(&full_bar[s]), 1u); mbar_init(smem_u32(&empty_bar[s]), 1u); }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&pm_full[b]), (uint32_t)kPmSlabWarps);
            mbar_init(smem_u32(&pm_empty[b]), 1u);
            mbar_init(smem_u32(&acc_full[b]), 1u);
            mbar_init(smem_u32(&acc_empty[b]), (uint32_t)kPmEpiWarps);
        }
        abort_flag = 0;
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
    // filters that nobody is writing (constant weights, re-packed by an earlier call) may be fetched before the kernel in
    // front has finished; everything else waits for it (the slab warps once they have worked out their first addresses)
    const bool slab_warp = warp >= 2 && warp < 2 + kPmSlabWarps;
    if (!slab_warp && (warp != 0 || !g.early_filters)) asm volatile("griddepcontrol.wait;" ::: "memory");
    auto decode = [&](int i, int& m0, int& n0) {
        const int t = unit + i * n_units;
        int tm, tn;
        if (g.raster == 0) { tm = t % g.tiles_m; tn = t / g.tiles_m; }
        else               { tn = t % g.tiles_n; tm = t / g.tiles_n; }
        m0 = tm * kHwTileM;
        n0 = tn * g.tile_n;
    };
    bool ok = true;

    // Warps 0 and 1 leave their loops to one thread: a vote over the warp for every wait and a re-convergence per stage made
    // the issue of a stage a serial chain of 600 cycles (a tap of 192 columns takes the tensor core 384).
    if (warp == 0) {
        // ---------------- filters ----------------
        if (elect_one()) {
            uint32_t st = 0, ph = 0;
            long long issued = 0;
            for (int i = 0; i < my_tiles && ok; ++i) {
                int m0, n0;
                decode(i, m0, n0);
                for (int cb = cb0, kt = cb0 * RS; cb < cb1 && ok; ++cb) {
                    for (int pl = 0; pl < g.n_planes && ok; ++pl) {
                        const int taps = g.planes[pl].nr * g.planes[pl].ns;
                        for (int t = 0; t < taps; t += tps) {
                            const int n = min(tps, taps - t);
                            const uint32_t bar = smem_u32(&full_bar[st]);
                            if (!mbar_wait(smem_u32(&empty_bar[st]), ph ^ 1u, abortp, g.status, 1u, g.wait_ns)) { ok = false; break; }
                            // (test facility: the first stage may be told to expect more than arrives, see tt_workload_test_stall)
                            mbar_expect_tx(bar, (uint32_t)n * kPmTapBytes + (issued == 0 && crank == 0 ? g.extra_tx : 0u));
                            uint32_t dst = base + st * stage_bytes;
                            for (int k = 0; k < n; ++k, dst += kPmTapBytes, ++kt) tma_load_3d(dst, &tmap_w, bar, kt * 32, m0, 0);
                            ++issued;
                            if (++st == (uint32_t)g.stages) { st = 0; ph ^= 1u; }
                        }
                    }
                }
            }
            if (!ok || *abortp) {
                // let copies in flight land before shared memory is given back (bounded)
                for (long long it = issued > g.stages ? issued - g.stages : 0; it < issued; ++it) {
                    const unsigned long long t0 = global_timer_ns();
                    while (!mbar_try_wait(smem_u32(&full_bar[it % g.stages]), (uint32_t)(it / g.stages) & 1u)) { if (global_timer_ns() - t0 > 2000000ull) break; }
                }
            }
        }
        __syncwarp();
        if (g.early_filters) asm volatile("griddepcontrol.wait;" ::: "memory");   // (a kernel ends only after the one in front of it)
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if (elect_one()) {
            const uint64_t d0 = make_desc(0u, 128);
            const uint32_t d_hi = (uint32_t)(d0 >> 32), d_lo = (uint32_t)d0;
            uint32_t st = 0, ph = 0, buf = 0, bph = 0;
            uint32_t ready = 0;                           // the filters of stage st have been seen to be there
            for (int i = 0; i < my_tiles && ok; ++i) {
                const uint32_t acc = (uint32_t)i & 1u, aph = ((uint32_t)i >> 1) & 1u;
                if (!mbar_wait(smem_u32(&acc_empty[acc]), aph ^ 1u, abortp, g.status, 12u, g.wait_ns)) { ok = false; break; }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + acc * (uint32_t)g.tile_n;
                uint32_t accumulate = 0u;
                for (int cb = cb0; cb < cb1 && ok; ++cb) {
                    for (int pl = 0; pl < g.n_planes && ok; ++pl) {
                        const ConvPlane P = g.planes[pl];
                        if (!mbar_wait(smem_u32(&pm_full[buf]), bph, abortp, g.status, 7u, g.wait_ns)) { ok = false; break; }
                        // first line of the slab that the plane's first tap reads
                        const uint32_t b_first = slab0 + buf * g.slab_bytes + (uint32_t)(P.f0 * g.wp + P.e0 - g.shift_min) * 128u;
                        const int taps = P.nr * P.ns;
                        int c = 0;
                        uint32_t b_row = b_first;
                        for (int t = 0; t < taps; t += tps) {
                            if (!ready && !mbar_wait(smem_u32(&full_bar[st]), ph, abortp, g.status, 2u, g.wait_ns)) { ok = false; break; }
                            tc_fence_after();
                            const uint32_t freed = smem_u32(&empty_bar[st]);
                            uint32_t a = d_lo + (((base + st * stage_bytes) & 0x3FFFFu) >> 4);
                            if (++st == (uint32_t)g.stages) { st = 0; ph ^= 1u; }
                            ready = mbar_test_wait(smem_u32(&full_bar[st]), ph);      // (answered while the products below are issued)
                            const int n = min(tps, taps - t);
#pragma unroll 1
                            for (int k = 0; k < n; ++k, a += kPmTapBytes >> 4) {
                                const uint32_t b = d_lo + (((b_row + (uint32_t)c * 128u) & 0x3FFFFu) >> 4);
#pragma unroll
                                for (uint32_t k8 = 0; k8 < 4; ++k8)
                                    mma_tf32(d_tmem, ((uint64_t)d_hi << 32) | (uint64_t)(a + 2u * k8), ((uint64_t)d_hi << 32) | (uint64_t)(b + 2u * k8), g.idesc, k8 == 0 ? accumulate : 1u);
                                accumulate = 1u;
                                if (++c == P.ns) { c = 0; b_row += (uint32_t)g.wp * 128u; }
                            }
                            mma_commit(freed);
                        }
                        if (ok) mma_commit(smem_u32(&pm_empty[buf]));
                        if (++buf == (uint32_t)g.slab_bufs) { buf = 0; bph ^= 1u; }
                    }
                }
                if (ok) mma_commit(smem_u32(&acc_full[acc]));
            }
        }
        __syncwarp();
    } else if (slab_warp) {
        // ---------------- slab: 32 positions x 32 channels at a time, lanes walk positions ----------------
        const int sw = warp - 2;
        uint32_t buf = 0, bph = 0;
        bool waited = false;                             // for the kernel in front
        for (int i = 0; i < my_tiles && ok; ++i) {
            int m0, n0;
            decode(i, m0, n0);
            for (int cb = cb0; cb < cb1 && ok; ++cb) {
                const int c_left = g.C - cb * 32;        // channels of the block that exist (the rest reads as zero)
                for (int pl = 0; pl < g.n_planes && ok; ++pl) {
                    const int pa = g.planes[pl].a, pb = g.planes[pl].b;
                    bool free = false;
                    for (int p0 = sw * 32; p0 < g.slab_lines; p0 += kPmSlabWarps * 32) {
                        const int p = p0 + lane;
                        const int u = n0 + g.shift_min + p;
                        int rem, j;
                        const int img = div_magic(max(u, 0), g.image_pitch, g.magic_image, rem);
                        const int row = div_magic(rem, g.wp, g.magic_wp, j);
                        const int y = row * g.sh + pa, x = j * g.sw + pb;
                        const bool valid = u >= 0 && img < g.images && y < g.H && x < g.W && p < g.slab_lines;
                        const float* src = g.x + (((long long)img * g.C + cb * 32) * g.H + y) * (long long)g.W + x;
                        float v[32];
                        const long long plane = (long long)g.H * g.W;
                        if (!waited) { asm volatile("griddepcontrol.wait;" ::: "memory"); waited = true; }
                        if (c_left >= 32) {
#pragma unroll
                            for (int c = 0; c < 32; ++c) v[c] = valid ? __ldg(src + c * plane) : 0.f;
                        } else {
#pragma unroll
                            for (int c = 0; c < 32; ++c) v[c] = valid && c < c_left ? __ldg(src + c * plane) : 0.f;
                        }
                        // (the loads above are in flight while the buffer's last readers finish)
                        if (!free) {
                            free = mbar_wait(smem_u32(&pm_empty[buf]), bph ^ 1u, abortp, g.status, 8u, g.wait_ns);
                            if (!__all_sync(0xffffffffu, free)) { ok = false; break; }
                        }
                        if (p < g.slab_lines) {
                            const uint32_t line = slab0 + buf * g.slab_bytes + 128u * (uint32_t)p;
#pragma unroll
                            for (int q = 0; q < 8; ++q)
                                st_shared_v4(line + ((((uint32_t)q) ^ ((line >> 7) & 7u)) << 4), v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                        }
                    }
                    if (ok && !free) ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&pm_empty[buf]), bph ^ 1u, abortp, g.status, 8u, g.wait_ns));
                    fence_proxy_async_shared();          // generic-proxy stores -> visible to the tensor core's reads
                    __syncwarp();
                    if (ok && lane == 0) mbar_arrive(smem_u32(&pm_full[buf]));
                    if (++buf == (uint32_t)g.slab_bufs) { buf = 0; bph ^= 1u; }
                }
            }
        }
        if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
    }
    // ---------------- read-out ----------------
    // One 32 x 32 block at a time: tensor memory -> (sum over the cluster) -> bias, activation -> a staging block in shared
    // memory, from which the lanes write one filter's 32 positions after the other.  A lane keeps its position.
    const bool reader = warp >= 2 + kPmSlabWarps || (single && warp >= 2);
    const int quad = warp & 3;                           // tensor-memory lane quadrant this warp may read
    const int per_quad = single ? (kPmSlabWarps + kPmEpiWarps) / 4 : 1, mine = single ? (warp - 2) >> 2 : 0;
    const int blocks_n = (g.tile_n + 31) >> 5;
    const float lo = g.act == TT_ACT_NONE || g.act == TT_ACT_GELU_ERF ? -INFINITY : 0.f;
    const float hi = g.act == TT_ACT_RELU6 ? 6.f : INFINITY;
    const long long PQ = (long long)g.P * g.Q;
    auto stage_block = [&](uint32_t at, const float (&v)[32]) {
#pragma unroll
        for (int j = 0; j < 32; j += 4) st_shared_v4(at + (uint32_t)(lane * kPmPitch + j) * 4u, v[j], v[j + 1], v[j + 2], v[j + 3]);
    };
    // where this lane's position of block b goes (false: nowhere), counted from the tensor's start at filter 0
    auto position = [&](int n0, int b, long long& off) {
        const int n = n0 + b * 32 + lane;
        int rem, q;
        const int img = div_magic(n, g.image_pitch, g.magic_image, rem);
        const int p = div_magic(rem, g.wp, g.magic_wp, q);
        off = (long long)img * g.M * PQ + (long long)p * g.Q + q;
        return q < g.Q && p < g.P && img < g.images && b * 32 + lane < g.tile_n;
    };
    // the residual of a block: 32 filters at this lane's position, requested before the accumulator is waited for
    auto load_residual = [&](float (&w)[32], int m_first, int n0, int b) {
        long long off;
        const bool out = position(n0, b, off);
        const float* res = g.residual + off + (long long)m_first * PQ;
        const int rows = g.M - m_first;
#pragma unroll
        for (int r = 0; r < 32; ++r, res += PQ) w[r] = out && r < rows ? __ldg(res) : 0.f;
    };
    // bias and activation on a block of pre-activation values (lane = filter), then out, adding the residual on the way
    auto finish_block = [&](float (&v)[32], const float (&w)[32], int m_first, int n0, int b, float bias, uint32_t stg) {
        long long off;
        const bool out = position(n0, b, off);
        const int rows = g.M - m_first;
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] += bias;
        if (g.residual == nullptr) {
            if (g.act == TT_ACT_GELU_ERF) {
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = gelu_erf(v[j]);
            } else if (g.act != TT_ACT_NONE) {
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = fminf(fmaxf(v[j], lo), hi);
            }
        }
        __syncwarp();                                    // (the staging block's previous values have been read)
        stage_block(stg, v);
        __syncwarp();
        float* y = g.y + off + (long long)m_first * PQ;
        const uint32_t from = stg + (uint32_t)lane * 4u;
        if (g.residual != nullptr) {
            // (the activation's branch stays outside the unrolled loops: code that runs once per launch is read from the L2, and
            // 32 inlined copies of GELU to jump over cost 5 us)
            float t[32];
#pragma unroll
            for (int r = 0; r < 32; ++r) t[r] = ld_shared_f32(from + (uint32_t)(r * kPmPitch) * 4u) + w[r];
            if (g.act == TT_ACT_GELU_ERF) {
#pragma unroll
                for (int r = 0; r < 32; ++r) t[r] = gelu_erf(t[r]);
            } else {
#pragma unroll
                for (int r = 0; r < 32; ++r) t[r] = fminf(fmaxf(t[r], lo), hi);
            }
            if (out) {
#pragma unroll
                for (int r = 0; r < 32; ++r, y += PQ) if (r < rows) *y = t[r];
            }
        } else if (rows >= 32) {
            if (out) {
#pragma unroll
                for (int r = 0; r < 32; ++r, y += PQ) *y = ld_shared_f32(from + (uint32_t)(r * kPmPitch) * 4u);
            }
        } else if (out) {
            for (int r = 0; r < rows; ++r, y += PQ) *y = ld_shared_f32(from + (uint32_t)(r * kPmPitch) * 4u);
        }
    };
    if (split == 1) {
        if (reader) {
            // (all tiles resident: the pipeline's shared memory is idle by now and takes the staging blocks of twelve warps)
            const uint32_t stg = single ? base + (uint32_t)(warp - 2) * kPmBlockBytes : base + g.epi_off + (uint32_t)(warp - 2 - kPmSlabWarps) * kPmBlockBytes;
            for (int i = 0; i < my_tiles && ok; ++i) {
                int m0, n0;
                decode(i, m0, n0);
                const uint32_t acc = (uint32_t)i & 1u, aph = ((uint32_t)i >> 1) & 1u;
                const int m_first = m0 + quad * 32;
                const float bias = g.bias && m_first + lane < g.M ? __ldg(g.bias + m_first + lane) : 0.f;
                float w[32];
                if (g.residual && mine < blocks_n) load_residual(w, m_first, n0, mine);
                ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&acc_full[acc]), aph, abortp, g.status, 4u, g.wait_ns));
                if (!ok) break;
                tc_fence_after();
                const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16) + acc * (uint32_t)g.tile_n;
#pragma unroll 1
                for (int b = mine; b < blocks_n; b += per_quad) {
                    uint32_t r[32];
                    float v[32];
                    tmem_ld32(t_row + (uint32_t)(b * 32), r);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
                    if (!single && b + 1 == blocks_n) {
                        // every value is in registers: hand the accumulator back to the MMA warp
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&acc_empty[acc]));
                    }
                    if (m_first < g.M) finish_block(v, w, m_first, n0, b, bias, stg);
                    if (g.residual && b + per_quad < blocks_n) load_residual(w, m_first, n0, b + per_quad);
                }
            }
        }
    } else {
        // Every CTA of the cluster reads out the blocks b with b % split == its rank, and leaves the others to their CTAs: in scratch
        // memory, as the registers lie, 512 contiguous bytes per four columns.  That goes through the L2.  Loads from the other CTAs' shared
        // memory came to 10 bytes a cycle and SM (a tile of 256 columns in fours: 12300 cycles for 96 KB and the stores); this way
        // 512 -> 512 at 7 x 7, batch 32, takes 23.7 us instead of 25.2, 208 -> 120 at 56 x 56, stride 2, 4 images, 15.4 instead of 17.6.
        int m0 = 0, n0 = 0;
        if (my_tiles > 0) decode(0, m0, n0);
        const int m_first = m0 + quad * 32;
        const uint32_t t_row = tmem_base + ((uint32_t)(quad * 32) << 16);
        const int own = crank + mine * split, own_step = per_quad * split;       // the own blocks, dealt to the warps of a quadrant
        const auto part_of = [&](int cta, int b) { return reinterpret_cast<float4*>(g.partial) + (((long long)(unit * split + cta) * blocks_n + b) * 4 + quad) * 256 + lane; };
        // A quadrant whose 32 filters are all beyond the layer's has nothing to pass on, and no traffic to slow the others with: 480 -> 24 at
        // 7 x 7, 12 images, 12.0 -> 11.1 us, 256 -> 40 at 14 x 14, 16 images, 11.4 -> 10.9.
        const bool sums = reader && my_tiles > 0 && m_first < g.M;
        float w[32];
        float bias = 0.f;
        if (reader && my_tiles > 0) {
            bias = g.bias && m_first + lane < g.M ? __ldg(g.bias + m_first + lane) : 0.f;
            if (g.residual && sums && own < blocks_n) load_residual(w, m_first, n0, own);
            ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&acc_full[0]), 0u, abortp, g.status, 4u, g.wait_ns));
            if (ok) tc_fence_after();
            if (ok && sums) {
#pragma unroll 1
                for (int b = mine; b < blocks_n; b += per_quad) {
                    if (b % split == crank) continue;
                    uint32_t r[32];
                    tmem_ld32(t_row + (uint32_t)(b * 32), r);
                    tmem_wait_ld();
                    float4* to = part_of(crank, b);
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        __stcg(to + j * 32, make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]), __uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3])));
                }
            }
        }
        if (!ok) *abortp = 1;
        cluster_sync_all();                              // (executed by every thread, also after a tripped wait)
        if (sums && ok) {
            const uint32_t stg = base + (uint32_t)(warp - 2) * kPmBlockBytes;       // (the pipeline's shared memory is idle)
#pragma unroll 1
            for (int b = own; b < blocks_n; b += own_step) {
                uint32_t r[32];
                float v[32];
                tmem_ld32(t_row + (uint32_t)(b * 32), r);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 32; ++j) v[j] = 0.f;
#pragma unroll 1
                for (int p = 0; p < split; ++p) {        // in CTA order, this CTA's own part where its turn comes
                    if (p == crank) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) v[j] += __uint_as_float(r[j]);
                    } else {
                        const float4* from = part_of(p, b);
                        float4 q[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j) q[j] = __ldcg(from + j * 32);
#pragma unroll
                        for (int j = 0; j < 8; ++j) { v[4 * j] += q[j].x; v[4 * j + 1] += q[j].y; v[4 * j + 2] += q[j].z; v[4 * j + 3] += q[j].w; }
                    }
                }
                finish_block(v, w, m_first, n0, b, bias, stg);
                if (g.residual && b + own_step < blocks_n) load_residual(w, m_first, n0, b + own_step);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, g.tmem_cols);
    }
}

// Filters [kout][C][R*S] -> [kout][block of 32 channels][tap in walk order][channel in block], zero beyond C.  One thread per
// output element; reads walk the channels of a tap (stride R*S), writes are contiguous.
struct TapOrder { unsigned char tap[64]; };
__global__ void tt_repack_filters_kernel(const float* __restrict__ w, float* __restrict__ out, int kout, int C, int RS, int CB, const TapOrder order) {
    const long long per_filter = (long long)CB * RS * 32;
    const long long total = (long long)kout * per_filter;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
        const long long f = i / per_filter;
        const int rem = (int)(i - f * per_filter);
        const int ci = rem & 31, t2 = rem >> 5;
        const int cb = t2 / RS, tap = order.tap[t2 - cb * RS];
        const int c = cb * 32 + ci;
        out[i] = c < C ? __ldg(w + (f * C + c) * RS + tap) : 0.f;
    }
    // The convolution behind this kernel waits for it; the one behind that may fetch its filters as soon as the first has started,
    // which is when the blocks here have left: what they wrote has to be in place by then, for copy engines too.
    asm volatile("fence.proxy.async.global;" ::: "memory");
    __threadfence();
}

cudaError_t launch_repack(const float* w, float* out, const ConvPmArgs& g, cudaStream_t st) {
    // the order in which the kernel walks the taps: plane by plane, row by row
    TapOrder order;
    memset(&order, 0, sizeof order);
    int t = 0;
    for (int pl = 0; pl < g.n_planes; ++pl) {
        const ConvPlane& p = g.planes[pl];
        for (int r = 0; r < p.nr; ++r) for (int s = 0; s < p.ns; ++s) order.tap[t++] = (unsigned char)((p.r0 + r * g.sh) * g.S + p.s0 + s * g.sw);
    }
    const long long total = (long long)g.M * g.blocks * g.R * g.S * 32;
    const int grid = (int)std::min<long long>((total + 255) / 256, kSms * 8);
    tt_repack_filters_kernel<<<grid, 256, 0, st>>>(w, out, g.M, g.C, g.R * g.S, g.blocks, order);
    return cudaGetLastError();
}

static cudaError_t raise_smem_limit() {
    static OncePerDevice once;
    return once([] { return cudaFuncSetAttribute(tt_conv_pm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit); });
}

static void launch_config(const tt_apply_info& I, const ConvPmArgs& g, cudaLaunchConfig_t* cfg, cudaLaunchAttribute (&attr)[2]) {
    cfg->gridDim = dim3((unsigned)I.grid_x, (unsigned)I.grid_y, 1); cfg->blockDim = dim3(kPmThreads, 1, 1);
    cfg->dynamicSmemBytes = (size_t)I.smem_bytes;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1; attr[0].val.clusterDim.y = (unsigned)g.split; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg->attrs = g.split > 1 ? attr : attr + 1;
    cfg->numAttrs = g.split > 1 ? 2 : 1;
}

// Can a cluster of the plan's CTAs be resident at all?
cudaError_t conv_pm_cluster_fits(const tt_apply_info& I, const ConvPmArgs& g, int* fits) {
    cudaError_t e = raise_smem_limit();
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[2];
    launch_config(I, g, &cfg, attr);
    cfg.numAttrs = 1;                                    // (the cluster dimension alone)
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, tt_conv_pm_kernel, &cfg);
    *fits = n > 0;
    return e;
}

cudaError_t launch_conv_pm(const tt_apply_info& I, const ConvPmArgs& g, const void* tmap_w, cudaStream_t st) {
    const cudaError_t e = raise_smem_limit();
    if (e != cudaSuccess) return e;
    CUtensorMap tw;
    memcpy(&tw, tmap_w, sizeof tw);
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr[2];
    launch_config(I, g, &cfg, attr);
    cfg.stream = st;
    return cudaLaunchKernelEx(&cfg, tt_conv_pm_kernel, tw, g);
}

}  // namespace tt
