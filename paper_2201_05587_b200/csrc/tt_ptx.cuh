// PTX wrappers shared by the kernels: barriers, TMA, tensor memory, the tensor core, shared and distributed shared memory.
#pragma once
#include <cuda_runtime.h>
#include <cuda.h>
#include <atomic>
#include <cstdint>
#include "tt_internal.h"

namespace tt {

// Host side: what a launcher sets up on a device before its first launch there (a kernel's shared-memory limit).  Threads may make
// their first calls at once; two that do both set up, which is harmless, and neither launches before it has.
class OncePerDevice {
public:
    template <typename F>
    cudaError_t operator()(F&& set_up) {
        int dev = 0;
        cudaGetDevice(&dev);
        const uint64_t bit = 1ull << (dev & 63);
        if (done_.load(std::memory_order_acquire) & bit) return cudaSuccess;
        const cudaError_t e = set_up();
        if (e == cudaSuccess) done_.fetch_or(bit, std::memory_order_release);
        return e;
    }
private:
    std::atomic<uint64_t> done_{0};
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Raise the byte count the barrier's current phase expects, without arriving on it.
__device__ __forceinline__ void mbar_expect_tx_only(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}
// Non-blocking test of a barrier phase.
__device__ __forceinline__ uint32_t mbar_test_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}
__device__ __forceinline__ unsigned long long global_timer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait.  Returns false when the CTA is aborting (this wait or another one expired).
static __device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag, unsigned* status,
                                            unsigned where, unsigned long long limit_ns) {
    const unsigned long long t0 = global_timer_ns();
    unsigned spins = 0;
    for (;;) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((++spins & 31u) == 0u) {
            if (*abort_flag) return false;
            if (global_timer_ns() - t0 > limit_ns) {
                *abort_flag = 1;
                atomicCAS(status, 0u, (unsigned)TT_ERR_TIMEOUT | (where << 8));
                return false;
            }
        }
    }
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, unsigned* status,
                                          unsigned where, unsigned long long limit_ns) {
    if (mbar_try_wait(bar, parity)) return true;         // the common case costs one instruction
    return mbar_wait_slow(bar, parity, abort_flag, status, where, limit_ns);
}

// Programmatic dependent launch.  A kernel launched with programmatic stream serialization may become resident while
// its predecessor in the stream is still running; it must wait here before its first access to global memory.  The
// kernel after it is allowed to do the same from this kernel's entry on.  (Without the launch attribute both
// instructions do nothing.)
__device__ __forceinline__ void pdl_allow_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait_prev() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// CTA `cta` of `ctas` asks for its share of what the launches behind this one will read (one thread; nothing waits for it).
__device__ __forceinline__ void prefetch_ahead(const Ahead& a, unsigned cta, unsigned ctas) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const unsigned share = ((a.bytes[i] + ctas - 1u) / ctas + 127u) & ~127u;
        const unsigned first = cta * share;
        if (first >= a.bytes[i]) continue;
        const unsigned end = min(first + share, a.bytes[i]);
#pragma unroll 1
        for (unsigned o = first; o < end; o += 16384u)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(static_cast<const char*>(a.p[i]) + o), "r"(min(16384u, end - o)) : "memory");
    }
}

// One lane of a converged warp (the same lane every time): it issues the warp's asynchronous instructions.
__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(pred));
    return pred != 0u;
}

__device__ __forceinline__ void fence_proxy_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const void* tmap, uint32_t bar, int c0, int c1, int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(tmap), "r"(bar), "r"(c0), "r"(c1), "r"(c2) : "memory");
}

// An MN-major operand tile: one box [tile_k][32 rows] after the other.
__device__ __forceinline__ void load_mn_boxes(uint32_t dst, const void* tmap, uint32_t bar, int row0, int rows, int k0, int tile_k, int bz) {
#pragma unroll 1
    for (int r = 0; r < rows; r += 32, dst += (uint32_t)tile_k * 128u) tma_load_3d(dst, tmap, bar, row0 + r, k0, bz);
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const void* tmap, uint32_t bar, int c0, int c1, int c2, int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(tmap), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t slot_smem, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot_smem), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]^T, one 128 x N x 8 TF32 step.
__device__ __forceinline__ void mma_tf32(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// The same with A in tensor memory: row i in lane i, one 32-bit column per reduction index.
__device__ __forceinline__ void mma_tf32_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// All 8-wide reduction steps of one pipeline stage into one accumulator: ATOMS swizzle atoms of K8 steps each.
// Inside an atom a step advances both descriptors by 2 (32 bytes); the next atom starts a_atom / b_atom later.
template <int ATOMS, int K8>
__device__ __forceinline__ void issue_steps(uint32_t d_tmem, uint32_t d_hi, uint32_t a_lo, uint32_t b_lo, uint32_t a_atom,
                                            uint32_t b_atom, uint32_t idesc, uint32_t accumulate) {
#pragma unroll
    for (int at = 0; at < ATOMS; ++at) {
#pragma unroll
        for (int k8 = 0; k8 < K8; ++k8) {
            mma_tf32(d_tmem, ((uint64_t)d_hi << 32) | (uint64_t)(a_lo + (uint32_t)at * a_atom + 2u * (uint32_t)k8),
                     ((uint64_t)d_hi << 32) | (uint64_t)(b_lo + (uint32_t)at * b_atom + 2u * (uint32_t)k8), idesc,
                     (at == 0 && k8 == 0) ? accumulate : 1u);
        }
    }
}
// The same when an operand is MN-major: any number of steps, each operand with its own stride (k8_a, k8_b) per step inside
// an atom of k8_n steps.
__device__ __forceinline__ void issue_steps_any(uint32_t d_tmem, uint32_t a_hi, uint32_t b_hi, uint32_t a_lo, uint32_t b_lo, uint32_t k8_a,
                                                uint32_t k8_b, uint32_t a_atom, uint32_t b_atom, int atoms, int k8_n, uint32_t idesc,
                                                uint32_t accumulate) {
#pragma unroll 1
    for (int at = 0; at < atoms; ++at, a_lo += a_atom, b_lo += b_atom) {
        uint32_t a = a_lo, b = b_lo;
#pragma unroll 4
        for (int k8 = 0; k8 < k8_n; ++k8, a += k8_a, b += k8_b) {
            mma_tf32(d_tmem, ((uint64_t)a_hi << 32) | (uint64_t)a, ((uint64_t)b_hi << 32) | (uint64_t)b, idesc, accumulate);
            accumulate = 1u;
        }
    }
}

// Arrive on an mbarrier once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor of a K-major tile whose rows are `row_bytes` long and hardware-swizzled with
// the span of one row: start address >> 4 in bits 0-13, leading byte offset >> 4 in bits 16-29 (not used by
// swizzled K-major tiles; set to 1), stride byte offset (distance between 8-row groups) >> 4 in bits 32-45,
// constant 0b001 in bits 46-48, swizzle mode in bits 61-63 (2 = 128 B, 4 = 64 B, 6 = 32 B).
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, int row_bytes) {
    const uint64_t swz = row_bytes == 128 ? 2ull : (row_bytes == 64 ? 4ull : 6ull);
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= 1ull << 16;
    d |= (uint64_t)((8u * (uint32_t)row_bytes) >> 4) << 32;
    d |= 1ull << 46;
    d |= swz << 61;
    return d;
}

// The same for an MN-major tile: the row index of the operand is the contiguous one in memory (the pixels of a 1x1
// convolution, the columns of an NN batch_matmul's second operand), so a TMA box of 32 rows x tile_k is [k][32 rows] lines of
// 128 bytes.  kind::tf32 reads that form with the 128-byte swizzle of 32-byte atoms (mode 1: the 32-byte chunk index is XORed
// with the line index modulo 4; read out of the tensor core with an indexed tile): four lines make an atom of 512 bytes
// (stride byte offset), and the next 32 rows begin a box further on (leading byte offset).
__device__ __forceinline__ uint64_t make_desc_mn(uint32_t saddr, uint32_t box_bytes) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)(box_bytes >> 4) << 16;
    d |= (uint64_t)(512u >> 4) << 32;
    d |= 1ull << 46;
    d |= 1ull << 61;
    return d;
}
// How far a descriptor's start address (in 16-byte units) moves per 8-wide reduction step and per swizzle atom of K.
struct DescSteps { uint32_t lo, hi, k8, atom; };
__device__ __forceinline__ DescSteps desc_steps(bool mn, int row_bytes, int rows, int tile_k, int atom_k) {
    DescSteps s;
    const uint64_t d = mn ? make_desc_mn(0u, (uint32_t)tile_k * 128u) : make_desc(0u, row_bytes);
    s.lo = (uint32_t)d; s.hi = (uint32_t)(d >> 32);
    s.k8 = mn ? 64u : 2u;                                // eight lines of 128 bytes; 32 bytes along a line
    s.atom = mn ? 64u * (uint32_t)(atom_k >> 3) : (uint32_t)(rows * row_bytes) >> 4;
    return s;
}

// GELU in its erf form, 0.5 x (1 + erf(x / sqrt 2)).  erf through the rational approximation 7.1.26 of Abramowitz and
// Stegun (absolute error below 1.5e-7, far inside what a TF32 product carries): a dozen instructions instead of
// the library routine's, which matters in a read-out that is a long serial instruction stream per thread.
__device__ __forceinline__ float gelu_erf(float x) {
    const float z = fabsf(x) * 0.70710678118654752440f;
    const float t = __fdividef(1.f, fmaf(0.3275911f, z, 1.f));
    float poly = fmaf(1.061405429f, t, -1.453152027f);
    poly = fmaf(poly, t, 1.421413741f);
    poly = fmaf(poly, t, -0.284496736f);
    poly = fmaf(poly, t, 0.254829592f);
    const float erf_abs = 1.f - poly * t * __expf(-z * z);
    return 0.5f * x * (1.f + copysignf(erf_abs, x));
}

__device__ __forceinline__ float apply_act(float v, int act) {
    switch (act) {
        case TT_ACT_RELU: return fmaxf(v, 0.f);
        case TT_ACT_RELU6: return fminf(fmaxf(v, 0.f), 6.f);
        case TT_ACT_GELU_ERF: return gelu_erf(v);
        default: return v;
    }
}

__device__ __forceinline__ void st_shared_v4(uint32_t addr, float a, float b, float c, float d) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}
__device__ __forceinline__ void st_shared_f32(uint32_t addr, float a) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(a) : "memory");
}
__device__ __forceinline__ void st_shared_u32(uint32_t addr, uint32_t a) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(addr), "r"(a) : "memory");
}
__device__ __forceinline__ float ld_shared_f32(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t ld_shared_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint4 ld_shared_v4u(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
// two fp32 products and sums in one instruction, each rounded as fmaf rounds
__device__ __forceinline__ float2 fma_pair(float2 a, float2 b, float2 c) {
    float2 r;
    asm("{\n\t.reg .b64 a, b, c;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
        "fma.rn.f32x2 c, a, b, c;\n\tmov.b64 {%0, %1}, c;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
__device__ __forceinline__ void cp_async_16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_4(uint32_t dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
// arrives on the barrier once the thread's copies so far have landed
__device__ __forceinline__ void cp_async_arrive(uint32_t bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Thread-block cluster primitives (split-K over a cluster: the splits of one output tile are the CTAs of a cluster
// and exchange their partial tiles through distributed shared memory).
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t map_to_peer(uint32_t saddr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
    return r;
}
__device__ __forceinline__ float4 ld_shared_v4f(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
// One band of this CTA's staged partial tile -> the same band's slot in a peer's reduction area; the bytes are counted
// on the peer's barrier (both destination addresses are shared::cluster addresses of the same peer).
__device__ __forceinline__ void bulk_copy_to_peer(uint32_t dst_caddr, uint32_t src_saddr, uint32_t bytes, uint32_t bar_caddr) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst_caddr), "r"(src_saddr), "r"(bytes), "r"(bar_caddr) : "memory");
}
// Wait until every bulk copy this thread issued has been written at its destination.
__device__ __forceinline__ void bulk_copies_done() {
    asm volatile("cp.async.bulk.commit_group;\n\tcp.async.bulk.wait_group 0;" ::: "memory");
}

// Untiled copies between global and shared memory (16-byte aligned, whole multiples of 16 bytes).
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, uint32_t src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n\tcp.async.bulk.commit_group;" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
}
// Wait until the stores this thread issued have read their shared memory.
__device__ __forceinline__ void bulk_stores_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// 32 lanes x 32 consecutive 32-bit columns: thread i of the warp receives lane (base + i).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr) : "memory");
}

// ... and back: thread i of the warp writes 8 consecutive columns of lane (base + i).
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float (&v)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"r"(taddr), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}
// Bounded wait on a barrier that CTAs of the cluster arrive on (acquire at cluster scope).
static __device__ __noinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort_flag, unsigned* status,
                                               unsigned where, unsigned long long limit_ns) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    const unsigned long long t0 = global_timer_ns();
    unsigned spins = 0;
    for (;;) {
        if (mbar_try_wait_cluster(bar, parity)) return true;
        if ((++spins & 31u) == 0u) {
            if (*abort_flag) return false;
            if (global_timer_ns() - t0 > limit_ns) {
                *abort_flag = 1;
                atomicCAS(status, 0u, (unsigned)TT_ERR_TIMEOUT | (where << 8));
                return false;
            }
        }
    }
}

__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
}  // namespace tt
