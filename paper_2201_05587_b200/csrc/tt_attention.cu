// Attention inside a chained pass: scores = Q K^T, row softmax, context = P V, three layers of a chain in one launch.
//
// At batch 1 the three launches are latency and nothing else (12 heads of 128 x 128 x 64: 12 or 24 CTAs, 3.6 + 1.6 + 5.4 us of
// which the products take a tenth).  Here a CTA takes kAttnRows query rows of one head through all three: the scores stay in
// tensor memory and registers between the products, and all three outputs are written as the separate layers write them.  The
// arithmetic is that of their records to the bit: as many accumulators as a record has splits or accumulators, added up in its
// order, and row sums in the order of the softmax record's lanes.
//
// The accumulators have 128 rows, of which kAttnRows are used: with 32, 12 heads of 128 rows spread over 48 SMs, and the rows' work
// (exponentials, 2 x 4 bytes written per score) is what is serial here, not the products.  The A tiles (queries, probabilities) hold
// those 32 rows only; the tensor core reads the unused rows from whatever follows them in shared memory and their results are
// never read.
//
// Latency is the bound: 5.3 us from the end of the projections to its own, of which 2 are the launch and the first loads, the rest
// one product, one softmax and one product after the other; of 12-layer encoders on 128 tokens it takes 81 us off 511.
//
// Warps: 0, 4, 8, 12 softmax (they may read lanes 0-31 of tensor memory; each takes every fourth 32-column block of the keys),
// 1 TMA, 2 MMA issuer + tensor-memory owner, the others write scores and probabilities to memory from their shared-memory tiles
// while the softmax goes on.  The probabilities' tile is the second product's K-major operand as it lies; the values' tile is
// MN-major.
#include <cuda_runtime.h>
#include <cuda.h>
#include <cstring>
#include "tt_ptx.cuh"

namespace tt {

constexpr int kAttnThreads = 512;
constexpr int kAttnSoftmaxWarps = 4, kAttnStoreWarps = 10;
constexpr uint32_t kAttnAtom = kAttnRows * 128u;         // bytes of a 32-column block of a tile of kAttnRows rows

// Builds: FAR, more than 128 keys (two blocks of 32 a softmax warp), and the order of the sums: rows of 16 or 32 lanes, of 8, or ORDER_ANY,
// records of several accumulators, single values a lane or rows of 4 lanes too.  A launch meets a cold instruction cache, and code costs
// it where nothing of it is run: 0.5 us what ORDER_ANY adds (the 12-layer encoder on 128 tokens 385 -> 391 us, on 256 525 -> 531), 0.3 FAR
// (381).  80 or 128 registers and 512 threads: no CTA that needs tensor memory, too, fits beside one that has not got its columns yet.
enum AttnOrder { ORDER_WIDE = 0, ORDER_EIGHT = 1, ORDER_ANY = 2 };

// One product: its steps of 8 of the reduction go into the accumulators of its record, `pitch` columns apart: `per` steps to each in
// turn (a record with splits), or dealt one by one (per = 0).
template <int ORDER, typename Issue>
__device__ __forceinline__ void attn_steps(uint32_t col, uint32_t pitch, int accs, int per, int steps, Issue issue) {
    if (ORDER == ORDER_ANY && accs > 1) {
#pragma unroll 1
        for (int a = 0; a < accs; ++a, col += pitch) {
            const int first = per > 0 ? a * per : a, end = per > 0 ? min(steps, first + per) : steps;
#pragma unroll 1
            for (int k8 = first; k8 < end; k8 += per > 0 ? 1 : accs) issue(col, k8, k8 != first ? 1u : 0u);
        }
        return;
    }
    for (int k8 = 0; k8 < steps; ++k8) issue(col, k8, k8 > 0 ? 1u : 0u);
}
// ... and 32 of its columns, read out in accumulator order.
template <int ORDER>
__device__ __forceinline__ void attn_read(uint32_t col, uint32_t pitch, int accs, float (&v)[32]) {
    uint32_t r[32];
    tmem_ld32(col, r);
    tmem_wait_ld();
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
    if constexpr (ORDER == ORDER_ANY) {
#pragma unroll 1
        for (int a = 1; a < accs; ++a) {
            tmem_ld32(col + (uint32_t)a * pitch, r);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] += __uint_as_float(r[j]);
        }
    }
}

// The sum of a row as 4 * m lanes come to it (m = 1, 2, 4, 8): lane l's share is the sum of values l, l + 4 m, ... of the line, the
// shares are added in halves, l and l + 2 m first.  The line holds 8 groups of four values, or 16 (`far`).
template <bool FAR, int ORDER>
__device__ __forceinline__ float attn_row_sum(uint32_t line, bool far, int m) {
    const auto add = [](float4& a, const float4& b) { a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; };
    const auto at = [&](int q) { return ld_shared_v4f(line + 16u * (uint32_t)q); };
    float4 x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = at(q);
    if (ORDER == ORDER_EIGHT) m = 2;
    if (ORDER == ORDER_EIGHT || (ORDER == ORDER_ANY && m < 4)) {
        // (m = 2: two shares of every second group; m = 1: one of all)
        const auto odd = [&](const float4& v) { if (m == 1) add(x[0], v); else add(x[1], v); };
        if (m == 1) add(x[0], x[1]);
#pragma unroll
        for (int q = 2; q < 8; q += 2) { add(x[0], x[q]); odd(x[q + 1]); }
#pragma unroll 1
        for (int q = 8; q < (FAR && far ? 16 : 8); q += 2) { add(x[0], at(q)); odd(at(q + 1)); }
        if (m == 2) add(x[0], x[1]);
    } else {
        if (FAR && far && m == 8) {
#pragma unroll
            for (int q = 0; q < 8; ++q) add(x[q], at(q + 8));
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) add(x[q], x[q + 4]);           // m = 8: the first halves; m = 4: a share's second group
        if (FAR && far && m == 4) {
#pragma unroll
            for (int q = 8; q < 16; ++q) add(x[q & 3], at(q));
        }
        add(x[0], x[2]); add(x[1], x[3]); add(x[0], x[1]);
    }
    return (x[0].x + x[0].z) + (x[0].y + x[0].w);
}

// Named barriers: 1 the softmax warps, 2 and 3 the softmax and the storing warps (a tile is in shared memory).
__device__ __forceinline__ void attn_meet(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void attn_report(int id, int threads) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory"); }

template <bool FAR, int ORDER>
__global__ void __launch_bounds__(kAttnThreads, 1)
tt_attention_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                    const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ AttnArgs g) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t qk_bar, v_bar;                    // operands have landed
    __shared__ uint64_t s_bar, o_bar;                     // the scores', the context's accumulator is complete
    __shared__ uint64_t p_bar;                            // the probabilities' tile is written
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ float s_max[kAttnSoftmaxWarps][32];

    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
    volatile int* abortp = &abort_flag;
    pdl_allow_next();
    const int head = (int)blockIdx.x / g.tiles_m, m0 = ((int)blockIdx.x - head * g.tiles_m) * kAttnRows;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t q_s = base, p_s = base + g.p_off, k_s = base + g.k_off, v_s = base + g.v_off;
    const uint32_t sc_s = k_s;                            // the scores' tile takes the keys' place once they have been multiplied
    if (threadIdx.x == 32) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_q) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_k) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmap_v) : "memory");
    }
    if (threadIdx.x == 0) {
        for (uint64_t* b : {&qk_bar, &v_bar, &s_bar, &o_bar}) mbar_init(smem_u32(b), 1u);
        mbar_init(smem_u32(&p_bar), (uint32_t)kAttnSoftmaxWarps);
        abort_flag = 0;
        fence_mbar_init();
        fence_proxy_async_shared();
    }
    if (warp == 2) {
        tmem_alloc(smem_u32(&tmem_slot), g.tmem_cols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *(volatile uint32_t*)&tmem_slot;
    if (g.ahead.bytes[0] != 0u && threadIdx.x == 96) prefetch_ahead(g.ahead, blockIdx.x, gridDim.x);
    pdl_wait_prev();

    const bool softmax_warp = (warp & 3) == 0;
    if (warp == 1) {
        // ---------------- TMA ----------------
        if (elect_one()) {
            const uint32_t qb = smem_u32(&qk_bar), vb = smem_u32(&v_bar);
            const uint32_t k_atom = (uint32_t)g.n16 * 128u, v_box = (uint32_t)g.n8 * 128u;
            mbar_expect_tx(qb, (uint32_t)g.d_atoms * (kAttnAtom + k_atom) + g.extra_tx);      // (test facility: tt_workload_test_stall)
            for (int at = 0; at < g.d_atoms; ++at) {
                tma_load_3d(q_s + (uint32_t)at * kAttnAtom, &tmap_q, qb, at * 32, m0, head);
                tma_load_3d(k_s + (uint32_t)at * k_atom, &tmap_k, qb, at * 32, 0, head);
            }
            mbar_expect_tx(vb, (uint32_t)g.v_boxes * v_box);
            for (int b = 0; b < g.v_boxes; ++b) tma_load_3d(v_s + (uint32_t)b * v_box, &tmap_v, vb, b * 32, 0, head);
            // shared memory stays until the copies have landed, also when somebody gave up (bounded)
            for (const uint32_t bar : {qb, vb}) {
                const unsigned long long t0 = global_timer_ns();
                while (!mbar_try_wait(bar, 0u)) if (global_timer_ns() - t0 > g.wait_ns) break;
            }
        }
        __syncwarp();
    } else if (warp == 2) {
        // ---------------- MMA issuer ----------------
        if (elect_one()) {
            const uint64_t d0 = make_desc(0u, 128);
            const uint32_t hi = (uint32_t)(d0 >> 32), lo = (uint32_t)d0;
            bool ok = mbar_wait(smem_u32(&qk_bar), 0u, abortp, g.status, 2u, g.wait_ns);
            if (ok) {
                tc_fence_after();
                const uint32_t a0 = lo + ((q_s & 0x3FFFFu) >> 4), b0 = lo + ((k_s & 0x3FFFFu) >> 4), b_atom = (uint32_t)g.n16 * 8u;
                attn_steps<ORDER>(tmem_base, (uint32_t)g.n_blocks * 32u, g.s_accs, g.s_per, g.d_steps, [&](uint32_t d, int k8, uint32_t accumulate) {
                    const uint32_t at = (uint32_t)k8 >> 2, in = 2u * ((uint32_t)k8 & 3u);
                    mma_tf32(d, ((uint64_t)hi << 32) | (uint64_t)(a0 + at * (kAttnAtom >> 4) + in), ((uint64_t)hi << 32) | (uint64_t)(b0 + at * b_atom + in), g.idesc_s, accumulate);
                });
                mma_commit(smem_u32(&s_bar));
                ok = mbar_wait(smem_u32(&v_bar), 0u, abortp, g.status, 2u, g.wait_ns) && mbar_wait(smem_u32(&p_bar), 0u, abortp, g.status, 3u, g.wait_ns);
            }
            if (ok) {
                tc_fence_after();
                const uint64_t v0 = make_desc_mn(0u, (uint32_t)g.n8 * 128u);
                const uint32_t v_hi = (uint32_t)(v0 >> 32);
                const uint32_t a0 = lo + ((p_s & 0x3FFFFu) >> 4);
                const uint32_t b0 = (uint32_t)v0 + ((v_s & 0x3FFFFu) >> 4);
                attn_steps<ORDER>(tmem_base + (uint32_t)g.o_col, (uint32_t)g.v_boxes * 32u, g.o_accs, g.o_per, g.n8 >> 3, [&](uint32_t d, int k8, uint32_t accumulate) {
                    const uint32_t a = a0 + ((uint32_t)k8 >> 2) * (kAttnAtom >> 4) + 2u * ((uint32_t)k8 & 3u);
                    mma_tf32(d, ((uint64_t)hi << 32) | (uint64_t)a, ((uint64_t)v_hi << 32) | (uint64_t)(b0 + 64u * (uint32_t)k8), g.idesc_o, accumulate);
                });
                mma_commit(smem_u32(&o_bar));
            }
        }
        __syncwarp();
    } else if (softmax_warp) {
        // ---------------- softmax: a lane has one query row, a warp every fourth block of 32 keys ----------------
        const int sw = warp >> 2, row = m0 + lane;
        constexpr int kBlocks = FAR ? 2 : 1;             // blocks a warp can have
        const uint32_t line = (uint32_t)lane * 128u, swz = (uint32_t)(lane & 7);
        float v[kBlocks][32];
        float mx = -INFINITY;
        bool ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&s_bar), 0u, abortp, g.status, 4u, g.wait_ns));
        tc_fence_after();
        if (ok) {
#pragma unroll
            for (int i = 0; i < kBlocks; ++i) {
                const int blk = sw + i * kAttnSoftmaxWarps;
                if (blk >= g.n_blocks) break;            // (warp-uniform)
                attn_read<ORDER>(tmem_base + (uint32_t)(blk * 32), (uint32_t)g.n_blocks * 32u, g.s_accs, v[i]);
#pragma unroll
                for (int j = 0; j < 32; j += 4)
                    st_shared_v4(sc_s + (uint32_t)blk * kAttnAtom + line + ((((uint32_t)j >> 2) ^ swz) << 4), v[i][j], v[i][j + 1], v[i][j + 2], v[i][j + 3]);
                const int left = g.n - blk * 32;
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    v[i][j] = j < left ? __fmul_rn(v[i][j], g.scale) : -INFINITY;
                    mx = fmaxf(mx, v[i][j]);
                }
            }
        }
        attn_report(2, 32 * (kAttnSoftmaxWarps + kAttnStoreWarps));
        s_max[sw][lane] = mx;
        attn_meet(1, 32 * kAttnSoftmaxWarps);
        mx = fmaxf(fmaxf(s_max[0][lane], s_max[1][lane]), fmaxf(s_max[2][lane], s_max[3][lane]));
        // The row's sum in the order of the softmax record's lanes: theirs are groups of four values, whose sums go to the row's line (zeros
        // where the row has no more of them), ...
        const uint32_t sums = base + g.x_off + (uint32_t)lane * kAttnSumLine;
        const bool far = FAR && g.n_blocks > kAttnSoftmaxWarps;
#pragma unroll
        for (int i = 0; i < kBlocks; ++i) {
            const int blk = sw + i * kAttnSoftmaxWarps;
            if (i > 0 && !far) break;
            float t[8] = {};
            if (blk < g.n_blocks) {
#pragma unroll
                for (int j = 0; j < 32; ++j) v[i][j] = expf(v[i][j] - mx);
#pragma unroll
                for (int j = 0; j < 8; ++j) t[j] = (v[i][4 * j] + v[i][4 * j + 1]) + (v[i][4 * j + 2] + v[i][4 * j + 3]);
                if (ORDER == ORDER_ANY && !g.lane_groups) {
#pragma unroll
                    for (int j = 0; j < 32; j += 4)
                        st_shared_v4(p_s + (uint32_t)blk * kAttnAtom + line + ((((uint32_t)j >> 2) ^ swz) << 4), v[i][j], v[i][j + 1], v[i][j + 2], v[i][j + 3]);
                }
            }
            st_shared_v4(sums + (uint32_t)blk * 32u, t[0], t[1], t[2], t[3]);
            st_shared_v4(sums + (uint32_t)blk * 32u + 16u, t[4], t[5], t[6], t[7]);
        }
        attn_meet(1, 32 * kAttnSoftmaxWarps);
        if (ORDER == ORDER_ANY && !g.lane_groups) {
            // ... or single values, every lane's 4 m apart: the warps add them up, four lanes' at a time
#pragma unroll 1
            for (int q = sw; q < 8; q += kAttnSoftmaxWarps) {
                float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
                for (int u = q < g.lanes4 ? q : g.n_blocks * 8; u < g.n_blocks * 8; u += g.lanes4) {
                    const float4 e = ld_shared_v4f(p_s + (uint32_t)(u >> 3) * kAttnAtom + line + ((((uint32_t)u & 7u) ^ swz) << 4));
                    t.x += e.x; t.y += e.y; t.z += e.z; t.w += e.w;
                }
                st_shared_v4(sums + (uint32_t)q * 16u, t.x, t.y, t.z, t.w);
            }
            attn_meet(1, 32 * kAttnSoftmaxWarps);
        }
        const float inv = 1.f / attn_row_sum<FAR, ORDER>(sums, far && g.lane_groups, g.lanes4);
#pragma unroll
        for (int i = 0; i < kBlocks; ++i) {
            const int blk = sw + i * kAttnSoftmaxWarps;
            if (blk >= g.n_blocks) break;
#pragma unroll
            for (int j = 0; j < 32; j += 4)
                st_shared_v4(p_s + (uint32_t)blk * kAttnAtom + line + ((((uint32_t)j >> 2) ^ swz) << 4), v[i][j] * inv, v[i][j + 1] * inv, v[i][j + 2] * inv, v[i][j + 3] * inv);
        }
        fence_proxy_async_shared();                      // the lanes' stores -> visible to the tensor core's reads
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&p_bar));
        attn_report(3, 32 * (kAttnSoftmaxWarps + kAttnStoreWarps));
        // context: 32 columns a warp
        ok = __all_sync(0xffffffffu, ok && mbar_wait(smem_u32(&o_bar), 0u, abortp, g.status, 4u, g.wait_ns));
        tc_fence_after();
        if (!ok) {
            // wherever a wait gave up, this one has too: the run of all three layers (the first one's status word has it from the wait)
            if (lane == 0) for (unsigned* word : g.status_more) atomicCAS(word, 0u, (unsigned)TT_ERR_TIMEOUT | (20u << 8));
        } else if (sw * 32 < g.dv) {
            float r[32];
            attn_read<ORDER>(tmem_base + (uint32_t)(g.o_col + sw * 32), (uint32_t)g.v_boxes * 32u, g.o_accs, r);
            if (row < g.m) {
                float* y = g.ctx + ((long long)head * g.m + row) * g.dv + sw * 32;
                const int left = g.dv - sw * 32;         // (a multiple of 4)
#pragma unroll
                for (int j = 0; j < 32; j += 4) {
                    if (j >= left) break;
                    if (g.ctx_vec) *reinterpret_cast<float4*>(y + j) = make_float4(r[j], r[j + 1], r[j + 2], r[j + 3]);
                    else for (int e = 0; e < 4; ++e) y[j + e] = r[j + e];
                }
            }
        }
    } else {
        // ---------------- scores and probabilities: shared-memory tiles -> rows in memory ----------------
        const int w = warp - 1 - (warp >> 2);             // 3 5 6 7 9 10 11 13 14 15 -> 2 3 4 5 6 7 8 9 10 11
        const int rows = min(kAttnRows, g.m - m0);
        const long long first = ((long long)head * g.m + m0) * g.n;
        for (int pass = 0; pass < 2; ++pass) {
            attn_meet(2 + pass, 32 * (kAttnSoftmaxWarps + kAttnStoreWarps));
            if (*abortp) continue;                       // (a tripped wait: the barriers are kept, nothing is stored)
            const uint32_t tile = pass ? p_s : sc_s;
            float* y = (pass ? g.probs : g.scores) + first;
            for (int r = w - 2; r < rows; r += kAttnStoreWarps) {
                const uint32_t line = tile + (uint32_t)r * 128u, swz = (uint32_t)(r & 7);
                float* yr = y + (long long)r * g.n;
                if (pass ? g.probs_vec : g.scores_vec) {
                    for (int c = lane * 4; c < g.n; c += 128)
                        *reinterpret_cast<float4*>(yr + c) = ld_shared_v4f(line + (uint32_t)(c >> 5) * kAttnAtom + ((((uint32_t)(c & 31) >> 2) ^ swz) << 4));
                } else {
                    for (int c = lane; c < g.n; c += 32)
                        yr[c] = ld_shared_f32(line + (uint32_t)(c >> 5) * kAttnAtom + ((((uint32_t)lane >> 2) ^ swz) << 4) + 4u * (uint32_t)(lane & 3));
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, g.tmem_cols);
    }
}

cudaError_t launch_attention(const AttnArgs& g, int heads, const void* tmap_q, const void* tmap_k, const void* tmap_v, cudaStream_t st) {
    typedef void (*Kernel)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const AttnArgs);
    static const Kernel kernels[] = {tt_attention_kernel<false, ORDER_WIDE>, tt_attention_kernel<true, ORDER_WIDE>, tt_attention_kernel<false, ORDER_EIGHT>,
                                     tt_attention_kernel<true, ORDER_EIGHT>, tt_attention_kernel<true, ORDER_ANY>};
    static OncePerDevice raised[5];
    const bool any = g.s_accs > 1 || g.o_accs > 1 || !g.lane_groups || g.lanes4 < 2;
    const int build = any ? 4 : 2 * (g.lanes4 == 2) + (g.n > 128);
    const Kernel kern = kernels[build];
    const cudaError_t ready = raised[build]([&] { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit); });
    if (ready != cudaSuccess) return ready;
    CUtensorMap tq, tk, tv;
    memcpy(&tq, tmap_q, sizeof tq);
    memcpy(&tk, tmap_k, sizeof tk);
    memcpy(&tv, tmap_v, sizeof tv);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(heads * g.tiles_m), 1, 1); cfg.blockDim = dim3(kAttnThreads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)g.smem_bytes; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, tq, tk, tv, g);
}

}  // namespace tt
