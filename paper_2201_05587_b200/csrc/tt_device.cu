// Device-facing half of the C ABI: binding a legalised record to a workload (workspace, tensor maps), running,
// the device-timed evaluator (Section 4.3 of the paper), the native grid tuner that fills pools.
#include <cuda_runtime.h>
#include <cuda.h>
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cstring>
#include <mutex>
#include <unordered_map>
#include <vector>
#include "tt_internal.h"

namespace tt {

cudaError_t launch_gemm(const tt_apply_info& I, int smem_bytes, const GemmArgs& g, const void* tmap_a, const void* tmap_b, const void* tmap_x,
                        cudaStream_t st);
cudaError_t launch_gemm_chain(const tt_apply_info& I, int smem_bytes, const GemmArgs& g, const ChainArgs& c, const void* tmap_a, const void* tmap_b,
                              const void* tmap_x, const void* tmap_z, cudaStream_t st);
cudaError_t launch_attention(const AttnArgs& g, int heads, const void* tmap_q, const void* tmap_k, const void* tmap_v, cudaStream_t st);
cudaError_t launch_dw(const tt_apply_info& I, const DwArgs& dw, cudaStream_t st);
cudaError_t plan_dw_staged(tt_apply_info& I, DwArgs& dw);
cudaError_t launch_dw_staged(const tt_apply_info& I, const DwArgs& dw, const void* tmap_x, cudaStream_t st);
cudaError_t launch_row(const tt_apply_info& I, const RowArgs& row, cudaStream_t st);
cudaError_t gemm_cluster_fits(const GemmArgs& g, int smem_bytes, int* fits);
cudaError_t launch_repack(const float* w, float* out, const ConvPmArgs& g, cudaStream_t st);
cudaError_t launch_conv_pm(const tt_apply_info& I, const ConvPmArgs& g, const void* tmap_w, cudaStream_t st);
cudaError_t conv_pm_cluster_fits(const tt_apply_info& I, const ConvPmArgs& g, int* fits);
cudaError_t launch_floor(const tt_apply_info& I, int smem_bytes, int cluster, cudaStream_t st);
cudaError_t launch_gemm_ps(const tt_apply_info& I, const GemmArgs& g, const TmapPair& maps, cudaStream_t st);

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver entry point is looked up through the runtime, so the library links against cudart only and loads
// on machines without a driver.
EncodeTiledFn encode_fn() {
    static const EncodeTiledFn fn = [] {                 // (looked up by one thread, the others wait for it)
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            return reinterpret_cast<EncodeTiledFn>(p);
        cudaGetLastError();
        return EncodeTiledFn(nullptr);
    }();
    return fn;
}

bool device_present() {
    int n = 0;
    if (cudaGetDeviceCount(&n) != cudaSuccess) { cudaGetLastError(); return false; }
    return n > 0;
}

// K-major operand [batch][rows][K] -> 3-D tensor map, box = [atom_k, box_rows, 1], swizzle span = one box row.
tt_status encode_operand(void* out, const float* base, int K, int rows, int batch, long long rs, long long bs,
                         bool batched, int atom_k, int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return TT_ERR_CUDA;
    if ((reinterpret_cast<uintptr_t>(base) & 15u) != 0) return TT_ERR_INVALID_ARG;
    const cuuint64_t nb = batched ? (cuuint64_t)batch : 1;
    cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, nb};
    cuuint64_t strides[2] = {(cuuint64_t)rs * 4, (cuuint64_t)(batched ? bs : (long long)rows * rs) * 4};
    cuuint32_t box[3] = {(cuuint32_t)atom_k, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    const int row_bytes = atom_k * 4;
    const CUtensorMapSwizzle swz = row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                 : row_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
    CUresult r = fn(reinterpret_cast<CUtensorMap*>(out), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base),
                    dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? TT_OK : TT_ERR_CUDA;
}

// Row-contiguous operand [batch][K][rows] (element (row, k) at k * ks + row) -> 3-D tensor map, box = [32 rows, box_k, 1]: the
// 128-byte lines of an MN-major tile, swizzled in 32-byte atoms as kind::tf32 reads them.
tt_status encode_operand_mn(void* out, const float* base, int rows, int K, int batch, long long ks, long long bs, bool batched, int box_k) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return TT_ERR_CUDA;
    if ((reinterpret_cast<uintptr_t>(base) & 15u) != 0) return TT_ERR_INVALID_ARG;
    const cuuint64_t nb = batched ? (cuuint64_t)batch : 1;
    cuuint64_t dims[3] = {(cuuint64_t)rows, (cuuint64_t)K, nb};
    cuuint64_t strides[2] = {(cuuint64_t)ks * 4, (cuuint64_t)(batched ? bs : (long long)K * ks) * 4};
    cuuint32_t box[3] = {32, (cuuint32_t)box_k, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(reinterpret_cast<CUtensorMap*>(out), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims,
                    strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? TT_OK : TT_ERR_CUDA;
}

// Ragged rows [rows][K] in groups of four, which are multiples of 16 bytes: box = [box_k + 4, box_rows] of the groups' lines, no swizzle.
tt_status encode_operand_raw(void* out, const float* base, int K, int rows, int box_k, int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return TT_ERR_CUDA;
    cuuint64_t dims[3] = {4 * (cuuint64_t)K, (cuuint64_t)(rows / 4), 1};
    cuuint64_t strides[2] = {16 * (cuuint64_t)K, 16 * (cuuint64_t)K * (cuuint64_t)(rows / 4)};
    cuuint32_t box[3] = {(cuuint32_t)box_k + 4, (cuuint32_t)box_rows, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(reinterpret_cast<CUtensorMap*>(out), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims,
                    strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? TT_OK : TT_ERR_CUDA;
}

// A matrix [batch][rows][cols] (rows `pitch` elements apart) in 32 x 32 blocks: the read-out's stores and residual loads.
tt_status encode_blocks(void* out, const float* base, int cols, int rows, int batch, long long pitch, long long bs, bool batched, bool swizzled) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return TT_ERR_CUDA;
    const cuuint64_t nb = batched ? (cuuint64_t)batch : 1;
    cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, nb};
    cuuint64_t strides[2] = {(cuuint64_t)pitch * 4, (cuuint64_t)(batched ? bs : (long long)rows * pitch) * 4};
    cuuint32_t box[3] = {32, 32, 1};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(reinterpret_cast<CUtensorMap*>(out), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims,
                    strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzled ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? TT_OK : TT_ERR_CUDA;
}

// NCHW image -> 4-D tensor map (W, H, C, N) without swizzle; box = [W + gap, in_rows, box_ch, 1].  A load that
// starts `gap` columns left of the image and at any (also negative) row gets zeros for everything outside.
tt_status encode_image(void* out, const float* base, int W, int H, int C, int N, int box_w, int box_h, int box_c) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return TT_ERR_CUDA;
    if ((reinterpret_cast<uintptr_t>(base) & 15u) != 0) return TT_ERR_INVALID_ARG;
    cuuint64_t dims[4] = {(cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)C, (cuuint64_t)N};
    cuuint64_t strides[3] = {(cuuint64_t)W * 4, (cuuint64_t)W * H * 4, (cuuint64_t)W * H * C * 4};
    cuuint32_t box[4] = {(cuuint32_t)box_w, (cuuint32_t)box_h, (cuuint32_t)box_c, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    CUresult r = fn(reinterpret_cast<CUtensorMap*>(out), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float*>(base), dims,
                    strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? TT_OK : TT_ERR_CUDA;
}

// Depthwise input as a 3-D tensor (W, H, planes = N * C), box = [box_w, in_h, tile_c], no swizzle.
tt_status encode_planes(void* out, const float* base, int W, int H, long long planes, int box_w, int box_h, int box_c) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return TT_ERR_CUDA;
    if ((reinterpret_cast<uintptr_t>(base) & 15u) != 0) return TT_ERR_INVALID_ARG;
    cuuint64_t dims[3] = {(cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)planes};
    cuuint64_t strides[2] = {(cuuint64_t)W * 4, (cuuint64_t)W * H * 4};
    cuuint32_t box[3] = {(cuuint32_t)box_w, (cuuint32_t)box_h, (cuuint32_t)box_c};
    cuuint32_t estr[3] = {1, 1, 1};
    CUresult r = fn(reinterpret_cast<CUtensorMap*>(out), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims,
                    strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? TT_OK : TT_ERR_CUDA;
}

const void* pick(const tt_tensors* t, int which) { return which == 0 ? t->x : t->w; }

// The events of chained passes.  A pass borrows its events and gives them back when it has been enqueued: a wait refers to
// what was recorded when it was issued, so an event may be recorded again at once.  At most kKept stay for the next pass on
// each device, the rest are destroyed; any thread may borrow.
class EventLoan {
public:
    explicit EventLoan(size_t most) {
        taken_.reserve(most);
        if (cudaGetDevice(&dev_) != cudaSuccess || dev_ >= kDevices) dev_ = -1;
    }
    ~EventLoan() {
        if (taken_.empty()) return;
        std::lock_guard<std::mutex> hold(lock());
        for (cudaEvent_t e : taken_) {
            if (n_kept()[dev_] < kKept) kept()[dev_][n_kept()[dev_]++] = e;
            else cudaEventDestroy(e);
        }
    }
    EventLoan(const EventLoan&) = delete;
    EventLoan& operator=(const EventLoan&) = delete;
    cudaEvent_t get() {
        if (dev_ < 0 || taken_.size() == taken_.capacity()) return nullptr;
        cudaEvent_t e = nullptr;
        {
            std::lock_guard<std::mutex> hold(lock());
            if (n_kept()[dev_] > 0) e = kept()[dev_][--n_kept()[dev_]];
        }
        if (!e && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) { cudaGetLastError(); return nullptr; }
        taken_.push_back(e);
        return e;
    }
private:
    static constexpr int kDevices = 64;
    static constexpr size_t kKept = 128;
    typedef cudaEvent_t Kept[kKept];
    static std::mutex& lock() { static std::mutex m; return m; }
    static Kept* kept() { static Kept k[kDevices]; return k; }
    static size_t* n_kept() { static size_t n[kDevices]; return n; }
    int dev_ = -1;
    std::vector<cudaEvent_t> taken_;
};

}  // namespace

// Forget what the workspace holds of re-packed filters, and the workspaces that passes captured under the record in force read.
static void forget_filters(tt_workload* w) {
    for (void* p : w->kept) cudaFree(p);
    w->kept.clear();
    w->repacked_for = nullptr; w->repacked_in = 0; w->captured_read = w->captured_fill = false;
}

void release_device(tt_workload* w) {
    forget_filters(w);
    if (w->workspace) cudaFree(w->workspace);
    if (w->exchange) cudaFree(w->exchange);
    w->exchange = nullptr; w->exchange_bytes = 0;
    if (w->status_word) cudaFree(w->status_word);
    if (w->ktab_dev) cudaFree(w->ktab_dev);
    w->ktab_dev = nullptr; w->ktab_bytes = 0;
    for (int i = 0; i < 5; ++i) if (w->hbuf[i]) cudaFree(w->hbuf[i]);
    w->workspace = nullptr; w->workspace_bytes = 0; w->status_word = nullptr;
    for (int i = 0; i < 5; ++i) { w->hbuf[i] = nullptr; w->hbytes[i] = 0; }
    cudaGetLastError();
}

tt_status bind_device(tt_workload* w) try {
    if (!device_present()) return TT_ERR_CUDA;
    if (w->family == TT_FAMILY_GEMM_TC && w->plan.g.cluster) {
        // a cluster whose CTAs cannot be resident together can never launch: an invalid pair, not a device error
        int fits = 0;
        if (gemm_cluster_fits(w->plan.g, w->plan.run_smem, &fits) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
        if (!fits) return TT_ERR_RESOURCE;
    }
    if (w->family == TT_FAMILY_GEMM_TC && w->plan.repack && w->plan.pm.split > 1) {
        int fits = 0;
        if (conv_pm_cluster_fits(w->plan.info, w->plan.pm, &fits) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
        if (!fits) return TT_ERR_RESOURCE;
    }
    if (w->family == TT_FAMILY_DW_SIMT && w->plan.dw.tma_stages > 0) {
        const cudaError_t e = plan_dw_staged(w->plan.info, w->plan.dw);
        if (e != cudaSuccess) { cudaGetLastError(); return e == cudaErrorLaunchOutOfResources ? TT_ERR_RESOURCE : TT_ERR_CUDA; }
    }
    forget_filters(w);
    const size_t need = (size_t)w->plan.info.workspace_bytes;
    if (need > w->workspace_bytes) {
        if (w->workspace) cudaFree(w->workspace);
        w->workspace = nullptr; w->workspace_bytes = 0;
        if (cudaMalloc(&w->workspace, need) != cudaSuccess) { cudaGetLastError(); return TT_ERR_OOM; }
        w->workspace_bytes = need;
    }
    const size_t exchange = (size_t)w->plan.info.exchange_kib * 1024;
    if (exchange > w->exchange_bytes) {
        if (w->exchange) cudaFree(w->exchange);
        w->exchange = nullptr; w->exchange_bytes = 0;
        if (cudaMalloc(&w->exchange, exchange) != cudaSuccess) { cudaGetLastError(); return TT_ERR_OOM; }
        w->exchange_bytes = exchange;
    }
    if (need > 0 && !w->plan.repack) {
        // arrival counters start at zero; each launch leaves them at zero again
        const size_t off = (size_t)w->plan.partial_bytes;
        if (cudaMemset(static_cast<char*>(w->workspace) + off, 0, need - off) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
    }
    if (!w->status_word) {
        if (cudaMalloc(reinterpret_cast<void**>(&w->status_word), 512) != cudaSuccess) { cudaGetLastError(); return TT_ERR_OOM; }
        if (cudaMemset(w->status_word, 0, 512) != cudaSuccess) return TT_ERR_CUDA;
    }
    if (w->family == TT_FAMILY_GEMM_TC && (w->plan.g.a_mode == OPM_IM2COL || w->plan.g.b_mode == OPM_IM2COL)) {
        // reduction-index table of the applied record: byte offset of (c, r, s) inside the slab, channel counted
        // from 0 (the kernel rebases it per chunk); indices past K point at the last channel, whose products meet
        // zero-filled filter values
        const GemmArgs& g = w->plan.g;
        const int kpad = g.k_tiles * g.tile_k, RS = g.R * g.S;
        std::vector<int> tab((size_t)kpad);
        for (int k = 0; k < kpad; ++k) {
            if (k < g.K) {
                const int c = k / RS, rem = k - c * RS, fr = rem / g.S, fs = rem - fr * g.S;
                tab[k] = 4 * (c * g.slab_chpitch + fr * g.slab_wp + fs);
            } else {
                tab[k] = 4 * ((g.C - 1) * g.slab_chpitch);
            }
        }
        const size_t bytes = (size_t)kpad * 4;
        if (bytes > w->ktab_bytes) {
            if (w->ktab_dev) cudaFree(w->ktab_dev);
            w->ktab_dev = nullptr; w->ktab_bytes = 0;
            if (cudaMalloc(reinterpret_cast<void**>(&w->ktab_dev), bytes) != cudaSuccess) { cudaGetLastError(); return TT_ERR_OOM; }
            w->ktab_bytes = bytes;
        }
        if (cudaMemcpy(w->ktab_dev, tab.data(), bytes, cudaMemcpyHostToDevice) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
    }
    w->tmaps.clear();
    return TT_OK;
} TT_NO_THROW

static tt_status tensor_maps_for(tt_workload* w, const GemmArgs& g, const void* a_ptr, const void* b_ptr, const TmapPair** out, int plan = 0) {
    const void* y_ptr = g.epi_tma ? g.y : nullptr;
    const void* r_ptr = g.res_tma ? g.residual : nullptr;
    // a pass calls a kernel's layers in the same order every time: the search begins behind the last hit
    const size_t n_maps = w->tmaps.size();
    for (size_t i = 0, at = w->tmap_next; i < n_maps; ++i, ++at) {
        if (at >= n_maps) at = 0;
        const TmapPair& e = w->tmaps[at];
        if (e.plan == plan && e.a_ptr == a_ptr && e.b_ptr == b_ptr && e.y_ptr == y_ptr && e.r_ptr == r_ptr) { w->tmap_next = at + 1; *out = &e; return TT_OK; }
    }
    TmapPair e;
    std::memset(&e, 0, sizeof e);
    e.plan = plan; e.a_ptr = a_ptr; e.b_ptr = b_ptr; e.y_ptr = y_ptr; e.r_ptr = r_ptr;
    // A gathered operand keeps an all-zero map in its parameter slot; the kernel never issues a TMA load on it.
    tt_status st = TT_OK;
    if (g.a_mode == OPM_TMA)
        st = encode_operand(e.a, static_cast<const float*>(a_ptr), g.K, g.M, g.batch, g.a_rs, g.a_bs, g.a_tma_batched != 0,
                            g.atom_k, kHwTileM);
    if (st != TT_OK) return st;
    if (g.b_mode == OPM_TMA)
        st = encode_operand(e.b, static_cast<const float*>(b_ptr), g.K, g.N, g.batch, g.b_rs, g.b_bs, g.b_tma_batched != 0,
                            g.atom_k, g.b_rows_cta);
    if (st != TT_OK) return st;
    if (g.a_mode == OPM_RAW) st = encode_operand_raw(e.a, static_cast<const float*>(a_ptr), g.K, g.a_rows_all, g.tile_k, kHwTileM / 4);
    if (st == TT_OK && g.b_mode == OPM_RAW) st = encode_operand_raw(e.b, static_cast<const float*>(b_ptr), g.K, g.b_rows_all, g.tile_k, g.tile_n / 4);
    if (st != TT_OK) return st;
    if (g.a_mode == OPM_TMA_MN)
        st = encode_operand_mn(e.a, static_cast<const float*>(a_ptr), g.M, g.K, g.batch, g.a_ks, g.a_bs, g.a_tma_batched != 0,
                               g.tile_k);
    if (st != TT_OK) return st;
    if (g.b_mode == OPM_TMA_MN)
        st = encode_operand_mn(e.b, static_cast<const float*>(b_ptr), g.N, g.K, g.batch, g.b_ks, g.b_bs, g.b_tma_batched != 0,
                               g.tile_k);
    if (st != TT_OK) return st;
    // the output (and the residual) in blocks: along the tile's columns, or, for a residual of outputs that are contiguous
    // along its rows, transposed
    if (y_ptr) st = encode_blocks(e.y, static_cast<const float*>(y_ptr), g.N, g.M, g.batch, g.y_ms, g.y_bs, g.y_tma_batched != 0, true);
    if (st == TT_OK && r_ptr)
        st = g.epi_tma ? encode_blocks(e.r, static_cast<const float*>(r_ptr), g.N, g.M, g.batch, g.y_ms, g.y_bs, g.y_tma_batched != 0, true)
                       : encode_blocks(e.r, static_cast<const float*>(r_ptr), g.M, g.N, g.batch, g.y_ns, g.y_bs, g.y_tma_batched != 0, false);
    if (st != TT_OK) return st;
    if (g.slab_tma == 1) {
        const float* img = static_cast<const float*>(g.a_mode == OPM_IM2COL ? a_ptr : b_ptr);
        if ((reinterpret_cast<uintptr_t>(img) & 15u) != 0) return TT_ERR_INVALID_ARG;   // images must be 16-byte aligned
        st = encode_image(e.x, img, g.W, g.H, g.C, g.batch, g.slab_wp, g.slab_in_rows, g.slab_box_ch);
        if (st != TT_OK) return st;
    }
    if (w->tmaps.size() >= 4096) w->tmaps.clear();
    w->tmaps.push_back(e);
    *out = &w->tmaps.back();
    return TT_OK;
}

// Tap-major convolution: the filters are brought into walk order first, once per weight pointer and applied record where
// the caller has promised that they are constant.  A capture only records the re-pack, and what it records runs whenever the
// pass is replayed.  So a copy made inside a capture serves that capture alone; a copy that a captured pass was told to read is
// kept for it, and a call for other weights goes to a workspace of its own; and calls under the promise leave a workspace that a
// captured pass fills.
static tt_status filters_for(tt_workload* w, const void* weights, cudaStream_t st, bool* repacked_now) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    unsigned long long capture = 0;
    if (cudaStreamGetCaptureInfo(st, &status, &capture) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
    if (status != cudaStreamCaptureStatusActive) capture = 0;
    *repacked_now = false;
    if (w->constant_weights && w->repacked_for == weights && (w->repacked_in == 0 || w->repacked_in == capture)) {
        if (capture != 0 && w->repacked_in == 0) w->captured_read = true;
        return TT_OK;
    }
    if (w->captured_read || (w->constant_weights && capture == 0 && w->captured_fill)) {
        void* fresh = nullptr;
        w->kept.reserve(w->kept.size() + 1);
        cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;       // (an allocation belongs to no capture)
        cudaThreadExchangeStreamCaptureMode(&mode);
        const cudaError_t e = cudaMalloc(&fresh, w->workspace_bytes);
        cudaThreadExchangeStreamCaptureMode(&mode);
        if (e != cudaSuccess) { cudaGetLastError(); return TT_ERR_OOM; }
        w->kept.push_back(w->workspace);
        w->workspace = fresh;
        w->captured_read = w->captured_fill = false;
    }
    w->repacked_for = nullptr;
    if (launch_repack(static_cast<const float*>(weights), static_cast<float*>(w->workspace), w->plan.pm, st) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
    if (w->constant_weights) w->repacked_for = weights;
    w->repacked_in = capture;
    if (capture != 0) w->captured_fill = true;
    *repacked_now = true;
    return TT_OK;
}

static tt_status launch_tap_major(tt_workload* w, const tt_tensors* t, cudaStream_t st) {
    const Plan& p = w->plan;
    bool repacked_now = false;
    tt_status s = filters_for(w, t->w, st, &repacked_now);
    if (s != TT_OK) return s;
    const TmapPair* maps = nullptr;
    s = tensor_maps_for(w, p.g, w->workspace, nullptr, &maps);
    if (s != TT_OK) return s;
    ConvPmArgs c = p.pm;
    c.x = static_cast<const float*>(t->x); c.y = static_cast<float*>(t->y);
    c.bias = w->sh.has_bias ? static_cast<const float*>(t->bias) : nullptr;
    c.residual = w->sh.has_residual ? static_cast<const float*>(t->residual) : nullptr;
    c.partial = static_cast<float*>(w->exchange);
    c.status = w->status_word; c.wait_ns = w->wait_ns; c.extra_tx = w->extra_tx;
    c.early_filters = w->constant_weights && !repacked_now;
    if (launch_conv_pm(p.info, c, maps->a, st) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
    return TT_OK;
}

// What a launch of a chained pass does beside its own layer: further layers of the same plan on the same x (their tensors), and
// the weights it brings into the L2 for the launches behind it.  chained: a launch of the pass does, and then all its dense layers
// take the kernel that can: two builds in turn meet a cold instruction cache (12-layer encoder 380 us with one, 391 with both).
struct Beside {
    bool chained = false;
    const tt_tensors* more[2] = {nullptr, nullptr};
    int n_more = 0;
    Ahead ahead{};
};

// The form of the one-tile kernel that does more than its layer.
static bool chain_form(const tt_workload* w, const Plan& p) {
    return w->op == TT_OP_DENSE && !w->sh.has_residual && !p.g.persistent && !p.g.x3 && p.g.a_mode == OPM_TMA && p.g.b_mode == OPM_TMA && !p.g.two_per_sm &&
           p.info.workspace_bytes == 0;
}

static tt_status launch_with(tt_workload* w, const tt_tensors* t, void* stream, const Beside& beside);

tt_status launch(tt_workload* w, const tt_tensors* t, void* stream) { return launch_with(w, t, stream, Beside{}); }

static tt_status launch_with(tt_workload* w, const tt_tensors* t, void* stream, const Beside& beside) try {
    if (!w || !t) return TT_ERR_INVALID_ARG;
    if (!w->plan.applied) return TT_ERR_NOT_APPLIED;
    if (!t->x || !t->y) return TT_ERR_INVALID_ARG;
    if (w->op != TT_OP_SOFTMAX && !t->w) return TT_ERR_INVALID_ARG;
    if (w->sh.has_bias && !t->bias) return TT_ERR_INVALID_ARG;
    if (w->sh.has_residual && !t->residual) return TT_ERR_INVALID_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaSuccess;
    const Plan& p = beside.n_more > 0 ? w->group[beside.n_more - 1] : w->plan;
    if (w->family == TT_FAMILY_GEMM_TC) {
        if (p.repack) return launch_tap_major(w, t, st);
        GemmArgs g = p.g;
        const void* a_ptr = pick(t, p.a_tensor);
        const void* b_ptr = pick(t, p.b_tensor);
        g.a = static_cast<const float*>(a_ptr);
        g.b = static_cast<const float*>(b_ptr);
        g.y = static_cast<float*>(t->y);
        g.bias = w->sh.has_bias ? static_cast<const float*>(t->bias) : nullptr;
        g.residual = w->sh.has_residual ? static_cast<const float*>(t->residual) : nullptr;
        g.partial = static_cast<float*>(w->workspace);
        g.counters = reinterpret_cast<unsigned*>(static_cast<char*>(w->workspace) + p.partial_bytes);
        g.status = w->status_word;
        if ((reinterpret_cast<uintptr_t>(t->y) & 15u) != 0 ||
            (g.residual && (reinterpret_cast<uintptr_t>(g.residual) & 15u) != 0)) g.vec_store = g.epi_tma = g.res_tma = 0;
        if (!g.residual) g.res_tma = 0;
        if (g.bias && (reinterpret_cast<uintptr_t>(g.bias) & 15u) == 0) g.vec_store |= 2;
        g.ktab_dev = w->ktab_dev;
        g.wait_ns = w->wait_ns;
        g.extra_tx = w->extra_tx;
        g.w_operand = 0;
        if (w->constant_weights && !g.persistent && (w->op == TT_OP_DENSE || w->op == TT_OP_CONV2D)) {
            if (p.a_tensor == 1 && g.a_mode == OPM_TMA) g.w_operand = 1;
            else if (p.b_tensor == 1 && g.b_mode == OPM_TMA) g.w_operand = 2;
        }
        // A row-contiguous operand that does not start on 16 bytes cannot come by TMA: it is gathered into a K-major tile (which
        // takes no more room than the MN-major one).  Images with rows of 16-byte multiples are asked for that in every form.
        if (!g.persistent && (w->op != TT_OP_CONV2D || w->sh.w % 4 != 0)) {
            if (g.a_mode == OPM_TMA_MN && (reinterpret_cast<uintptr_t>(a_ptr) & 15u) != 0) { g.a_mode = OPM_GATHER_ROWS; g.idesc &= ~(1u << 15); }
            if (g.b_mode == OPM_TMA_MN && (reinterpret_cast<uintptr_t>(b_ptr) & 15u) != 0) { g.b_mode = OPM_GATHER_ROWS; g.idesc &= ~(1u << 16); }
        }
        if (g.a_mode == OPM_RAW && (reinterpret_cast<uintptr_t>(a_ptr) & 15u) != 0) g.a_mode = OPM_GATHER_K;
        if (g.b_mode == OPM_RAW && (reinterpret_cast<uintptr_t>(b_ptr) & 15u) != 0) g.b_mode = OPM_GATHER_K;
        if (g.slab_tma == 2 && (reinterpret_cast<uintptr_t>(t->x) & 15u) != 0) g.slab_tma = 0;
        const TmapPair* maps = nullptr;
        if (beside.chained && chain_form(w, p)) {
            ChainArgs c{};
            c.group = 1 + beside.n_more;
            c.w_member = p.a_tensor == 1 ? 1 : 2;
            c.ahead = beside.ahead;
            unsigned char more[2][128] = {};             // (copies: what a further member's maps add to the cache may move the others)
            for (int i = 0; i < beside.n_more; ++i) {
                const tt_tensors* o = beside.more[i];
                const tt_status s = tensor_maps_for(w, g, pick(o, p.a_tensor), pick(o, p.b_tensor), &maps, beside.n_more);
                if (s != TT_OK) return s;
                std::memcpy(more[i], p.a_tensor == 1 ? maps->a : maps->b, 128);
                c.bias_more[i] = w->sh.has_bias ? static_cast<const float*>(o->bias) : nullptr;
                c.y_more[i] = static_cast<float*>(o->y);
            }
            const tt_status s = tensor_maps_for(w, g, a_ptr, b_ptr, &maps, beside.n_more);
            if (s != TT_OK) return s;
            e = launch_gemm_chain(p.info, p.run_smem, g, c, maps->a, maps->b, more[0], more[1], st);
        } else {
            const tt_status s = tensor_maps_for(w, g, a_ptr, b_ptr, &maps);
            if (s != TT_OK) return s;
            e = g.persistent ? launch_gemm_ps(p.info, g, *maps, st) : launch_gemm(p.info, p.run_smem, g, maps->a, maps->b, maps->x, st);
        }
    } else if (w->family == TT_FAMILY_DW_SIMT) {
        DwArgs d = p.dw;
        d.x = static_cast<const float*>(t->x); d.w = static_cast<const float*>(t->w);
        d.bias = w->sh.has_bias ? static_cast<const float*>(t->bias) : nullptr;
        d.y = static_cast<float*>(t->y);
        if ((reinterpret_cast<uintptr_t>(t->y) & 15u) != 0) d.vec = 1;
        if ((reinterpret_cast<uintptr_t>(t->x) & 15u) != 0) d.vec_in = 0;
        if (d.tma_stages > 0) {
            // the image's tensor map, cached per input pointer like the contraction's maps
            const TmapPair* maps = nullptr;
            if (!d.runs) {
                for (const TmapPair& m : w->tmaps) if (m.a_ptr == t->x) { maps = &m; break; }
                if (!maps) {
                    TmapPair m;
                    std::memset(&m, 0, sizeof m);
                    m.a_ptr = t->x;
                    tt_status s = encode_planes(m.x, d.x, d.W, d.H, (long long)d.N * d.C, d.box_w, d.in_h, d.tile_c);
                    if (s != TT_OK) return s;
                    if (w->tmaps.size() >= 4096) w->tmaps.clear();
                    w->tmaps.push_back(m);
                    maps = &w->tmaps.back();
                }
            } else d.vec_in = (reinterpret_cast<uintptr_t>(t->x) & 15u) == 0;
            d.status = w->status_word;
            d.wait_ns = w->wait_ns;
            e = launch_dw_staged(p.info, d, maps ? maps->x : nullptr, st);
        } else
        e = launch_dw(p.info, d, st);
    } else {
        RowArgs r = p.row;
        r.x = static_cast<const float*>(t->x); r.y = static_cast<float*>(t->y);
        if (((reinterpret_cast<uintptr_t>(t->y) | reinterpret_cast<uintptr_t>(t->x)) & 15u) != 0) { r.vec = 1; r.cached = r.chunk = r.warps = 0; }
        r.status = w->status_word; r.wait_ns = w->wait_ns;
        e = launch_row(p.info, r, st);
    }
    if (e != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
    return TT_OK;
} TT_NO_THROW

static tt_status read_status(tt_workload* w, cudaStream_t st) {
    if (!w->status_word) return TT_ERR_NOT_APPLIED;
    if (cudaStreamSynchronize(st) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
    unsigned v = 0;
    if (cudaMemcpy(&v, w->status_word, 4, cudaMemcpyDeviceToHost) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
    if (v != 0) {
        cudaMemset(w->status_word, 0, 4);
        // A CTA that gave up never reported at its tile's arrival counter: the counters of a workspace split-K record
        // are no longer all zero, and the next run would finish tiles from incomplete partial sums.  Clear them.
        const Plan& p = w->plan;
        if (w->family == TT_FAMILY_GEMM_TC && w->workspace && !p.repack && p.info.workspace_bytes > p.partial_bytes)
            cudaMemset(static_cast<char*>(w->workspace) + p.partial_bytes, 0, (size_t)(p.info.workspace_bytes - p.partial_bytes));
        return (tt_status)(v & 0xffu);
    }
    return TT_OK;
}

static void default_timing(tt_timing_opts* o) {
    if (o->warmup_batches <= 0) o->warmup_batches = 3;
    if (o->batches <= 0) o->batches = 10;
    if (o->min_batch_us <= 0) o->min_batch_us = 200;
    if (o->max_repeats <= 0) o->max_repeats = 4096;
}

static float median_of(std::vector<float>& v, float* q1, float* q3) {
    std::sort(v.begin(), v.end());
    const size_t n = v.size();
    auto at = [&](double pos) {
        const size_t lo = (size_t)pos;
        const size_t hi = std::min(lo + 1, n - 1);
        const double f = pos - (double)lo;
        return (float)(v[lo] * (1.0 - f) + v[hi] * f);
    };
    if (q1) *q1 = at(0.25 * (n - 1));
    if (q3) *q3 = at(0.75 * (n - 1));
    // even count: mean of the two middle order statistics
    return (n & 1) ? v[n / 2] : 0.5f * (v[n / 2 - 1] + v[n / 2]);
}

static tt_status time_applied(tt_workload* w, const tt_tensors* sets, size_t n_sets, cudaStream_t st,
                              const tt_timing_opts* oin, tt_timing* out) try {
    tt_timing_opts o{};
    if (oin) o = *oin;
    default_timing(&o);
    if (n_sets == 0) return TT_ERR_INVALID_ARG;
    std::vector<float> per;                              // (before anything that would have to be given back)
    per.reserve((size_t)o.batches);
    const void* filters_in = w->workspace;
    const bool captured_read = w->captured_read, captured_fill = w->captured_fill;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaStream_t cap = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t gexec = nullptr;
    tt_status rc = TT_OK;
    size_t next = 0;
    auto fail = [&](tt_status s) { rc = s; };
    auto run_n = [&](int n, cudaStream_t s) -> tt_status {
        for (int i = 0; i < n; ++i) {
            if (o.floor) {
                // the launch floor of the applied record: an empty kernel with the same launch shape
                const Plan& p = w->plan;
                const bool gemm = w->family == TT_FAMILY_GEMM_TC;
                const int cluster = !gemm ? 0 : p.repack ? (p.pm.split > 1 ? p.pm.split : 0) : p.g.cluster;
                for (int l = 0; l < p.info.launches; ++l)
                    if (launch_floor(p.info, p.run_smem ? p.run_smem : p.info.smem_bytes, cluster, s) != cudaSuccess) {
                        cudaGetLastError();
                        return TT_ERR_CUDA;
                    }
                continue;
            }
            tt_status r = launch(w, &sets[next], s);
            next = (next + 1) % n_sets;
            if (r != TT_OK) return r;
        }
        return TT_OK;
    };
    do {
        if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) { fail(TT_ERR_CUDA); break; }
        // first launch alone: surfaces launch errors and a tripped wait before anything is timed
        if ((rc = run_n(1, st)) != TT_OK) break;
        if ((rc = read_status(w, st)) != TT_OK) break;
        // calibrate the number of launches per batch
        float ms = 0.f;
        const int probe = 4;
        cudaEventRecord(e0, st);
        if ((rc = run_n(probe, st)) != TT_OK) break;
        cudaEventRecord(e1, st);
        if (cudaEventSynchronize(e1) != cudaSuccess) { fail(TT_ERR_CUDA); break; }
        cudaEventElapsedTime(&ms, e0, e1);
        const double est_us = std::max(0.2, (double)ms * 1000.0 / probe);
        int reps = (int)std::min<double>((double)o.max_repeats, std::max(1.0, std::ceil(o.min_batch_us / est_us)));
        if (o.use_graph) {
            // one batch = one graph of `reps` launches: no CPU launch gaps between them
            reps = (int)((reps + n_sets - 1) / n_sets * n_sets);      // every replay walks the sets identically
            if (cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking) != cudaSuccess) { fail(TT_ERR_CUDA); break; }
            // tensor maps must exist before capture (encoding is host work, but keep the capture pure launches)
            if (cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal) != cudaSuccess) { fail(TT_ERR_CUDA); break; }
            tt_status r = run_n(reps, cap);
            cudaError_t ce = cudaStreamEndCapture(cap, &graph);
            if (r != TT_OK) { fail(r); break; }
            if (ce != cudaSuccess || !graph) { fail(TT_ERR_CUDA); break; }
            if (cudaGraphInstantiate(&gexec, graph, 0) != cudaSuccess) { fail(TT_ERR_CUDA); break; }
        }
        for (int b = 0; b < o.warmup_batches + o.batches; ++b) {
            cudaEventRecord(e0, st);
            if (gexec) {
                if (cudaGraphLaunch(gexec, st) != cudaSuccess) { fail(TT_ERR_CUDA); break; }
            } else if ((rc = run_n(reps, st)) != TT_OK) break;
            cudaEventRecord(e1, st);
            if (cudaEventSynchronize(e1) != cudaSuccess) { fail(TT_ERR_CUDA); break; }
            cudaEventElapsedTime(&ms, e0, e1);
            if (b >= o.warmup_batches) per.push_back(ms * 1000.f / (float)reps);
        }
        if (rc != TT_OK) break;
        if ((rc = read_status(w, st)) != TT_OK) break;
        tt_timing t{};
        t.repeats = reps; t.batches = (int)per.size();
        t.median_us = median_of(per, &t.q1_us, &t.q3_us);
        t.min_us = per.front(); t.max_us = per.back();
        *out = t;
    } while (false);
    if (gexec) cudaGraphExecDestroy(gexec);
    if (graph) cudaGraphDestroy(graph);
    if (w->plan.repack) {
        // the batch's graph is gone: nobody reads or fills the filters' workspace on its account any more
        const bool same = w->workspace == filters_in;
        w->captured_read = same && captured_read; w->captured_fill = same && captured_fill;
        if (w->repacked_in != 0) w->repacked_for = nullptr;
    }
    if (cap) cudaStreamDestroy(cap);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (rc == TT_ERR_CUDA) cudaGetLastError();
    return rc;
} TT_NO_THROW

static tt_status apply_impl(tt_workload* w, const tt_schedule_record* rec, int mode, int strict_class, tt_apply_info* info) {
    if (!w || !rec) return TT_ERR_INVALID_ARG;
    Plan np;
    tt_status s = legalise(w, rec, mode, strict_class, &np);
    if (info && (s == TT_OK || s == TT_ERR_RESOURCE)) *info = np.info;
    if (s != TT_OK) return s;                     // the previously applied record, if any, stays in force
    Plan old = w->plan;
    w->plan = np;
    s = bind_device(w);
    if (s != TT_OK) { w->plan = old; w->plan.applied = false; return s; }
    w->plan.applied = true;
    w->plan.strict = mode == TT_MODE_STRICT;
    plan_groups(w);
    if (info) *info = w->plan.info;               // (the grid that the device holds)
    return TT_OK;
}

}  // namespace tt

using namespace tt;

extern "C" {

tt_status tt_schedule_apply(tt_workload* w, const tt_schedule_record* rec, tt_apply_info* info_out) {
    return apply_impl(w, rec, TT_MODE_LEGALISE, 0, info_out);
}

tt_status tt_schedule_apply_ex(tt_workload* w, const tt_schedule_record* rec, int32_t mode, int32_t strict_class,
                               tt_apply_info* info_out) {
    if (mode != TT_MODE_LEGALISE && mode != TT_MODE_STRICT) return TT_ERR_INVALID_ARG;
    return apply_impl(w, rec, mode, strict_class, info_out);
}

tt_status tt_run(tt_workload* w, const tt_tensors* t, void* cuda_stream) { return launch(w, t, cuda_stream); }

// ---- chained passes -----------------------------------------------------------------------------------------

// Layers that go to the device together, and where.
struct ChainLaunch {
    size_t first; int count; bool attention;
    int32_t lane;
    bool needed, moved;                                  // somebody on another lane waits for it; a member's plan lane is another one
    Ahead ahead;
};

constexpr size_t kAheadBytes = 10u << 20;                // weights that a launch asks for ahead, at most

struct Range { const char* p; size_t bytes; };
static bool overlap(const Range& a, const Range& b) { return a.p && b.p && a.p < b.p + b.bytes && b.p < a.p + a.bytes; }
// x, w, bias, residual, y of a layer
static Range range_of(const tt_chain_step& s, int which) {
    const tt_tensors& t = *s.tensors;
    const void* p[5] = {t.x, t.w, t.bias, t.residual, t.y};
    return Range{static_cast<const char*>(p[which]), tensor_elems(s.workload, which) * 4};
}
// May layer b run beside layer a (neither writes what the other one touches)?
static bool independent(const tt_chain_step& a, const tt_chain_step& b) {
    const Range ya = range_of(a, 4), yb = range_of(b, 4);
    for (int i = 0; i < 5; ++i)
        if (overlap(ya, range_of(b, i)) || overlap(yb, range_of(a, i))) return false;
    return true;
}
static bool usable(const tt_chain_step& s) {
    return s.workload && s.tensors && s.workload->plan.applied && s.tensors->x && s.tensors->y && (s.workload->op == TT_OP_SOFTMAX || s.tensors->w) &&
           (!s.workload->sh.has_bias || s.tensors->bias) && (!s.workload->sh.has_residual || s.tensors->residual);
}
static bool waits_in_front(const tt_chain_step& s, size_t first) {
    for (int32_t j = 0; j < s.n_waits; ++j) if ((size_t)s.waits[j] >= first) return false;
    return true;
}

// How many layers from `first` on are one plan on the same activations: the projections of an attention block.  One launch of
// three fills the SMs that a launch of one leaves idle (768 -> 768 on 128 rows: 48 CTAs), without streams to fork and join.
static int group_at(const tt_chain_step* steps, size_t n_steps, size_t first) {
    const tt_chain_step& a = steps[first];
    if (!usable(a)) return 1;
    const tt_workload* w = a.workload;
    if (!(w->group[0].applied || w->group[1].applied)) return 1;
    int count = 1;
    while (count < 3 && first + count < n_steps) {
        const tt_chain_step& b = steps[first + count];
        if (b.workload != w || !usable(b) || b.tensors->x != a.tensors->x || !waits_in_front(b, first)) break;
        // (a layer that cannot run is left to fail by itself)
        if (((reinterpret_cast<uintptr_t>(a.tensors->w) | reinterpret_cast<uintptr_t>(b.tensors->w)) & 15u) != 0) break;
        // one launch stores all members the same way
        if (((reinterpret_cast<uintptr_t>(b.tensors->y) ^ reinterpret_cast<uintptr_t>(a.tensors->y)) & 15u) != 0) break;
        bool apart = true;
        for (int i = 0; i < count; ++i) apart = apart && independent(steps[first + i], b);
        if (!apart) break;
        ++count;
    }
    while (count > 1 && !w->group[count - 2].applied) --count;
    return count;
}

// Scores, softmax, context from `first` on, as one launch: 12 heads of 128 rows and 64 columns took three launches of 3.6, 1.6
// and 5.4 us, the 12-layer encoder 511 us with them and 430 with this one.  Only where the heads' blocks of query rows are resident at once (batch 1); from there on the layers fill the chip
// one by one and each has a kernel made for that.
static bool attention_at(const tt_chain_step* steps, size_t n_steps, size_t first, AttnArgs* g) {
    if (first + 3 > n_steps) return false;
    const tt_chain_step *s = steps + first;
    for (int i = 0; i < 3; ++i)
        if (!usable(s[i]) || s[i].workload->plan.strict) return false;
    const tt_workload *qk = s[0].workload, *sm = s[1].workload, *pv = s[2].workload;
    if (qk->op != TT_OP_BATCH_MATMUL || !qk->sh.trans_b || sm->op != TT_OP_SOFTMAX || pv->op != TT_OP_BATCH_MATMUL || pv->sh.trans_b) return false;
    for (const tt_workload* w : {qk, pv})
        if (w->sh.has_bias || w->sh.has_residual || w->sh.act != TT_ACT_NONE || w->plan.g.x3) return false;
    const int heads = qk->sh.batch, m = qk->sh.m, n = qk->sh.nn, d = qk->sh.kk, dv = pv->sh.nn;
    if (sm->sh.batch != heads || sm->sh.m != m || sm->sh.nn != n || pv->sh.batch != heads || pv->sh.m != m || pv->sh.kk != n) return false;
    if (n > 256 || d > 128 || dv > 128 || d % 4 || dv % 4 || (long long)heads * ((m + kAttnRows - 1) / kAttnRows) > kSms) return false;
    const tt_tensors &tq = *s[0].tensors, &ts = *s[1].tensors, &tv = *s[2].tensors;
    if (ts.x != tq.y || tv.x != ts.y || ((reinterpret_cast<uintptr_t>(tq.x) | reinterpret_cast<uintptr_t>(tq.w) | reinterpret_cast<uintptr_t>(tv.w)) & 15u)) return false;
    // the three outputs lie apart from each other and from everything that is read
    const Range in[3] = {range_of(s[0], 0), range_of(s[0], 1), range_of(s[2], 1)}, out[3] = {range_of(s[0], 4), range_of(s[1], 4), range_of(s[2], 4)};
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j)
            if (overlap(out[i], in[j]) || (i != j && overlap(out[i], out[j]))) return false;
    // waits and streams: a layer behind the first may only wait for layers in front of it or inside
    for (int i = 0; i < 3; ++i)
        for (int32_t j = 0; j < s[i].n_waits; ++j) if ((size_t)s[i].waits[j] >= first + i) return false;
    AttnArgs a{};
    a.scores = static_cast<float*>(tq.y); a.probs = static_cast<float*>(ts.y); a.ctx = static_cast<float*>(tv.y);
    a.status = qk->status_word; a.status_more[0] = sm->status_word; a.status_more[1] = pv->status_word;
    a.wait_ns = std::min({qk->wait_ns, sm->wait_ns, pv->wait_ns});
    a.extra_tx = std::max({qk->extra_tx, sm->extra_tx, pv->extra_tx});
    a.m = m; a.n = n; a.dv = dv; a.tiles_m = (m + kAttnRows - 1) / kAttnRows;
    a.n16 = (n + 15) / 16 * 16; a.n8 = (n + 7) / 8 * 8; a.n_blocks = (n + 31) / 32;
    a.d_atoms = (d + 31) / 32; a.d_steps = (d + 7) / 8; a.v_boxes = (dv + 31) / 32;
    const auto vec = [](const void* p, int cols) { return cols % 4 == 0 && (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
    a.scores_vec = vec(a.scores, n); a.probs_vec = vec(a.probs, n); a.ctx_vec = vec(a.ctx, dv);
    // The order in which the layers' records add up.  What the kernel has no order for takes three launches: splits of several
    // accumulators each, the softmax from memory (other alignments, rows of few lanes).
    const auto products = [](const GemmArgs& p, int steps, int* accs, int* per) {
        *per = p.split_k > 1 ? p.k_tiles_per_split * (p.tile_k / 8) : 0;
        *accs = p.split_k > 1 ? p.split_k : std::min(p.n_acc, steps);
        return p.split_k == 1 || p.n_acc == 1;
    };
    if (!products(qk->plan.g, a.d_steps, &a.s_accs, &a.s_per) || !products(pv->plan.g, a.n8 / 8, &a.o_accs, &a.o_per)) return false;
    const RowArgs& rows = sm->plan.row;
    if (rows.cached == 0 && rows.chunk == 0) return false;
    if (((reinterpret_cast<uintptr_t>(ts.x) | reinterpret_cast<uintptr_t>(ts.y)) & 15u) != 0 || rows.lanes_per_row < 4) return false;
    a.lanes4 = rows.lanes_per_row / 4; a.lane_groups = rows.cached > 0;
    a.scale = sm->sh.scale;
    const int block = kAttnRows * 128;                   // 32 columns of a tile of query rows
    a.p_off = (unsigned)(a.d_atoms * block);
    a.k_off = a.p_off + (unsigned)(a.n_blocks * block);
    // (the scores' tile and the partial sums behind it take the keys' place)
    a.x_off = a.k_off + (unsigned)(a.n_blocks * block);
    a.v_off = a.k_off + (unsigned)((std::max(a.d_atoms * a.n16 * 128, a.n_blocks * block + kAttnRows * (int)kAttnSumLine) + 1023) / 1024 * 1024);
    // (the tensor core reads 128 rows of a tile that has 32: all of that lies inside)
    const int over = 128 * 128 - block;
    const int bytes = std::max((int)a.v_off + a.v_boxes * a.n8 * 128, (int)a.k_off + over) + 1024;
    if (bytes > kDynSmemLimit) return false;
    a.smem_bytes = bytes;
    a.o_col = a.s_accs * a.n_blocks * 32;
    const int columns = a.o_col + a.o_accs * a.v_boxes * 32;
    if (columns > 512) return false;
    a.tmem_cols = 32;
    while ((int)a.tmem_cols < columns) a.tmem_cols *= 2;
    const unsigned tf32 = (1u << 4) | (2u << 7) | (2u << 10) | ((unsigned)(kHwTileM >> 4) << 24);
    a.idesc_s = tf32 | ((unsigned)(a.n16 >> 3) << 17);
    a.idesc_o = tf32 | ((unsigned)((dv + 15) / 16 * 2) << 17) | (1u << 16);
    if (g) *g = a;
    return true;
}

// How many layers from `first` on go to the device together.
static int together_at(const tt_chain_step* steps, size_t n_steps, size_t first, bool* attention) {
    *attention = attention_at(steps, n_steps, first, nullptr);
    return *attention ? 3 : group_at(steps, n_steps, first);
}

static tt_status launch_chain_attention(const tt_chain_step* s, const AttnArgs& g, cudaStream_t st) {
    tt_workload *qk = s[0].workload, *pv = s[2].workload;
    const tt_shapes& sh = qk->sh;
    // the maps of the queries and keys are kept with the scores' workload, the values' with the context's
    const auto cached = [](tt_workload* w, const void* a, const void* b) -> const TmapPair* {
        for (const TmapPair& m : w->tmaps) if (m.plan == kAttnMaps && m.a_ptr == a && m.b_ptr == b) return &m;
        return nullptr;
    };
    const auto keep = [](tt_workload* w, TmapPair& m, const void* a, const void* b) {
        m.plan = kAttnMaps; m.a_ptr = a; m.b_ptr = b;
        if (w->tmaps.size() >= 4096) w->tmaps.clear();
        w->tmaps.push_back(m);
        return &w->tmaps.back();
    };
    const void *q = s[0].tensors->x, *k = s[0].tensors->w, *v = s[2].tensors->w;
    const TmapPair* m = cached(qk, q, k);
    if (!m) {
        TmapPair e;
        std::memset(&e, 0, sizeof e);
        tt_status r = encode_operand(e.a, static_cast<const float*>(q), sh.kk, sh.m, sh.batch, sh.kk, (long long)sh.m * sh.kk, true, 32, kAttnRows);
        if (r == TT_OK) r = encode_operand(e.b, static_cast<const float*>(k), sh.kk, sh.nn, sh.batch, sh.kk, (long long)sh.nn * sh.kk, true, 32, g.n16);
        if (r != TT_OK) return r;
        m = keep(qk, e, q, k);
    }
    unsigned char maps[2][128];
    std::memcpy(maps[0], m->a, 128); std::memcpy(maps[1], m->b, 128);
    m = cached(pv, v, v);
    if (!m) {
        TmapPair e;
        std::memset(&e, 0, sizeof e);
        const tt_status r = encode_operand_mn(e.a, static_cast<const float*>(v), g.dv, g.n, sh.batch, g.dv, (long long)g.n * g.dv, true, g.n8);
        if (r != TT_OK) return r;
        m = keep(pv, e, v, v);
    }
    if (launch_attention(g, sh.batch, maps[0], maps[1], m->a, st) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
    return TT_OK;
}

// The launches of a pass, on the lanes of their first layers, and what they bring into the L2.  Whether layers share any: then all
// dense layers take the chain build.
static bool plan_launches(const tt_chain_step* steps, size_t n_steps, std::vector<ChainLaunch>& plan) {
    bool shared = false;
    plan.reserve(n_steps);
    for (size_t i = 0; i < n_steps;) {
        bool attention = false;
        const int count = together_at(steps, n_steps, i, &attention);
        ChainLaunch l{i, count, attention, steps[i].lane, false, false, Ahead{}};
        for (int m = 0; m < l.count; ++m) l.moved = l.moved || steps[i + (size_t)m].lane != l.lane;
        shared = shared || count > 1;
        plan.push_back(l);
        i += (size_t)l.count;
    }
    // In a pass with shared launches, a dense or attention launch whose CTAs are resident at once brings the weights of the launches up to
    // three behind it into the L2 while it runs: whole layers, kAheadBytes in all.  12-layer encoder, 64 tokens 332 -> 320 us, 128 tokens
    // 386 -> 381, 256 tokens 535 -> 527, as much as with 24 MB.  Not more, because weights that the L2 does not keep are read twice (two
    // times 768 -> 768 -> 4096 -> 16384 -> 768 on one row: 202 us with whatever came next, 142 with 24 MB, 136 without), and not in
    // other passes, whose layers it slows by 1 to 6 % at every size (32 times 1024 -> 1024 on 32 rows: 137 us without, 143 with).
    for (size_t l = 0, next = 0; shared && l < plan.size(); ++l) {
        next = std::max(next, l + 1);
        const tt_chain_step& from = steps[plan[l].first];
        if (!plan[l].attention) {
            if (!usable(from) || !chain_form(from.workload, from.workload->plan)) continue;
            const tt_apply_info& I = (plan[l].count > 1 ? from.workload->group[plan[l].count - 2] : from.workload->plan).info;
            if ((long long)I.grid_x * I.grid_y * plan[l].count > kSms) continue;
        }
        int n = 0;
        for (size_t bytes = 0; n < 3 && next < plan.size() && next <= l + 3; ++next) {
            const ChainLaunch& c = plan[next];
            const tt_chain_step& s = steps[c.first];
            if (c.attention || !usable(s) || (s.workload->op != TT_OP_DENSE && s.workload->op != TT_OP_CONV2D) || s.workload->plan.repack) continue;
            if (n + c.count > 3) break;
            for (int m = 0; m < c.count; ++m) {
                const Range w = range_of(steps[c.first + (size_t)m], 1);
                const size_t skip = (16 - reinterpret_cast<uintptr_t>(w.p)) & 15u;
                if (w.bytes < skip + 16 || bytes + w.bytes > kAheadBytes) continue;
                plan[l].ahead.p[n] = w.p + skip; plan[l].ahead.bytes[n++] = (unsigned)(w.bytes - skip) & ~15u;
                bytes += w.bytes;
            }
        }
    }
    return shared;
}

tt_status tt_run_chain(const tt_chain_step* steps, size_t n_steps, void* const* streams, size_t n_streams, size_t* failed_at) try {
    if (!steps || n_steps == 0 || !streams || n_streams == 0) return TT_ERR_INVALID_ARG;
    constexpr size_t kNone = ~(size_t)0;
    std::vector<ChainLaunch> plan;
    std::vector<size_t> launch_of(n_steps), waits, first_wait, tail(n_streams, kNone);
    std::vector<char> used(n_streams, 0);
    waits.reserve(n_steps); first_wait.reserve(n_steps + 1);
    for (size_t i = 0; i < n_steps; ++i) {
        const tt_chain_step& s = steps[i];
        if (failed_at) *failed_at = i;
        if (s.lane < 0 || (size_t)s.lane >= n_streams || s.n_waits < 0 || (s.n_waits && !s.waits)) return TT_ERR_INVALID_ARG;
        for (int32_t j = 0; j < s.n_waits; ++j)
            if (s.waits[j] < 0 || (size_t)s.waits[j] >= i) return TT_ERR_INVALID_ARG;
    }
    const bool chained = plan_launches(steps, n_steps, plan);
    for (size_t l = 0; l < plan.size(); ++l)
        for (int m = 0; m < plan[l].count; ++m) launch_of[plan[l].first + (size_t)m] = l;
    // What a launch waits for: the launches of the layers its layers name, the last launch of each of its layers' lanes where that
    // went to another one, and, where it shares scratch (re-packed filters, partial sums and arrival counters) with an earlier
    // launch of the same workload, that one.
    bool side = false;
    {
        std::unordered_map<const tt_workload*, size_t> last;
        bool lanes = false;
        for (size_t i = 0; i < n_steps; ++i) lanes = lanes || steps[i].lane != 0;
        for (size_t l = 0; l < plan.size(); ++l) {
            first_wait.push_back(waits.size());
            const auto after = [&](size_t dep) {
                if (dep == kNone || dep == l || plan[dep].lane == plan[l].lane) return;
                if (std::find(waits.begin() + (long)first_wait[l], waits.end(), dep) != waits.end()) return;
                waits.push_back(dep);
                plan[dep].needed = true;
            };
            for (int m = 0; m < plan[l].count && lanes; ++m) {
                const tt_chain_step& s = steps[plan[l].first + (size_t)m];
                for (int32_t j = 0; j < s.n_waits; ++j) after(launch_of[(size_t)s.waits[j]]);
                after(tail[(size_t)s.lane]);
                if (s.workload && s.workload->plan.info.workspace_bytes != 0 && !plan[l].attention) {
                    const auto seen = last.find(s.workload);
                    if (seen != last.end()) after(seen->second);
                    last[s.workload] = l;
                }
            }
            for (int m = 0; m < plan[l].count; ++m) tail[(size_t)steps[plan[l].first + (size_t)m].lane] = l;
            side = side || plan[l].lane != 0 || plan[l].moved;
        }
        first_wait.push_back(waits.size());
        for (size_t k = 1; k < n_streams; ++k) if (tail[k] != kNone && plan[tail[k]].lane != (int32_t)k) plan[tail[k]].needed = true;
    }
    EventLoan events(plan.size() + 2 * n_streams + 2);   // (nothing below allocates once the pass is being enqueued)
    std::vector<cudaEvent_t> done(plan.size(), nullptr);
    tt_status rc = TT_OK;
    cudaEvent_t start = nullptr;
    cudaStream_t main_stream = static_cast<cudaStream_t>(streams[0]);
    if (side) {
        start = events.get();
        if (!start || cudaEventRecord(start, main_stream) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
    }
    for (size_t l = 0; l < plan.size() && rc == TT_OK; ++l) {
        const ChainLaunch& c = plan[l];
        const tt_chain_step& s = steps[c.first];
        if (failed_at) *failed_at = c.first;
        cudaStream_t st = static_cast<cudaStream_t>(streams[c.lane]);
        cudaError_t e = cudaSuccess;
        // a side stream forks (a capture, or the caller's ordering) where a layer of its lane is first used
        for (int m = 0; m < c.count && e == cudaSuccess; ++m) {
            const size_t lane = (size_t)steps[c.first + (size_t)m].lane;
            if (lane != 0 && !used[lane]) {
                e = cudaStreamWaitEvent(static_cast<cudaStream_t>(streams[lane]), start, 0);
                if (e == cudaSuccess && lane != (size_t)c.lane) {
                    // (the layer runs on another lane: behind what the caller had put on its own)
                    cudaEvent_t in = events.get();
                    e = in ? cudaEventRecord(in, static_cast<cudaStream_t>(streams[lane])) : cudaErrorUnknown;
                    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, in, 0);
                }
            }
            used[lane] = 1;
        }
        for (size_t j = first_wait[l]; j < first_wait[l + 1] && e == cudaSuccess; ++j) e = cudaStreamWaitEvent(st, done[waits[j]], 0);
        if (e == cudaSuccess) {
            AttnArgs g;
            if (c.attention && attention_at(steps, n_steps, c.first, &g)) {
                g.ahead = c.ahead;
                rc = launch_chain_attention(&s, g, st);
            } else {
                Beside b;
                b.chained = chained;
                b.ahead = c.ahead;
                for (int m = 1; m < c.count; ++m) b.more[b.n_more++] = steps[c.first + (size_t)m].tensors;
                rc = launch_with(s.workload, s.tensors, st, b);
            }
        }
        if (e == cudaSuccess && rc == TT_OK && c.needed) {
            done[l] = events.get();
            e = done[l] ? cudaEventRecord(done[l], st) : cudaErrorUnknown;
        }
        if (e != cudaSuccess) { cudaGetLastError(); rc = TT_ERR_CUDA; }
    }
    for (size_t l = 1; l < n_streams; ++l) {
        if (!used[l]) continue;
        // (a layer of this lane that ran on another one: what the caller puts on the lane's stream comes behind it)
        if (rc == TT_OK && tail[l] != kNone && plan[tail[l]].lane != (int32_t)l && cudaStreamWaitEvent(static_cast<cudaStream_t>(streams[l]), done[tail[l]], 0) != cudaSuccess) {
            cudaGetLastError();
            rc = TT_ERR_CUDA;
        }
        cudaEvent_t end = events.get();
        if (!end || cudaEventRecord(end, static_cast<cudaStream_t>(streams[l])) != cudaSuccess ||
            cudaStreamWaitEvent(main_stream, end, 0) != cudaSuccess) { cudaGetLastError(); if (rc == TT_OK) rc = TT_ERR_CUDA; }
    }
    return rc;
} TT_NO_THROW

// (the arguments of the two functions below)
static tt_status check_chain(const tt_chain_step* steps, size_t n_steps) {
    if (!steps || n_steps == 0) return TT_ERR_INVALID_ARG;
    for (size_t i = 0; i < n_steps; ++i) {
        const tt_chain_step& s = steps[i];
        if (!s.workload || !s.workload->plan.applied) return TT_ERR_NOT_APPLIED;
        for (int32_t j = 0; j < s.n_waits; ++j) if (!s.waits || s.waits[j] < 0 || (size_t)s.waits[j] >= i) return TT_ERR_INVALID_ARG;
    }
    return TT_OK;
}

tt_status tt_chain_launches(const tt_chain_step* steps, size_t n_steps, size_t* launches) {
    const tt_status st = launches ? check_chain(steps, n_steps) : TT_ERR_INVALID_ARG;
    if (st != TT_OK) return st;
    *launches = 0;
    for (size_t i = 0; i < n_steps;) {
        bool attention = false;
        const int count = together_at(steps, n_steps, i, &attention);
        *launches += attention ? 1 : (size_t)steps[i].workload->plan.info.launches;
        i += (size_t)count;
    }
    return TT_OK;
}

tt_status tt_chain_ahead(const tt_chain_step* steps, size_t n_steps, size_t* bytes) try {
    const tt_status st = bytes ? check_chain(steps, n_steps) : TT_ERR_INVALID_ARG;
    if (st != TT_OK) return st;
    std::vector<ChainLaunch> plan;
    plan_launches(steps, n_steps, plan);
    std::fill(bytes, bytes + n_steps, (size_t)0);
    for (const ChainLaunch& l : plan) for (const unsigned b : l.ahead.bytes) bytes[l.first] += b;
    return TT_OK;
} TT_NO_THROW

tt_status tt_workload_set_constant_weights(tt_workload* w, int32_t on) {
    if (!w) return TT_ERR_INVALID_ARG;
    w->constant_weights = on != 0;
    if (!on) w->repacked_for = nullptr;                  // (what is promised from here on is about the weights as they are then)
    return TT_OK;
}

tt_status tt_workload_set_wait_limit(tt_workload* w, uint64_t nanoseconds) {
    if (!w || nanoseconds == 0) return TT_ERR_INVALID_ARG;
    w->wait_ns = nanoseconds;
    return TT_OK;
}

tt_status tt_workload_test_stall(tt_workload* w, uint32_t extra_bytes) {
    if (!w || (extra_bytes & 15u)) return TT_ERR_INVALID_ARG;
    w->extra_tx = extra_bytes;
    return TT_OK;
}

tt_status tt_workload_status(tt_workload* w, void* cuda_stream) {
    if (!w) return TT_ERR_INVALID_ARG;
    return read_status(w, static_cast<cudaStream_t>(cuda_stream));
}

static tt_status run_host_impl(tt_workload* w, const tt_tensors* host, void* cuda_stream, int64_t* bytes_h2d, int64_t* bytes_d2h,
                               bool synchronise) {
    if (!w || !host) return TT_ERR_INVALID_ARG;
    if (!w->plan.applied) return TT_ERR_NOT_APPLIED;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const void* src[4] = {host->x, host->w, host->bias, host->residual};
    int64_t up = 0;
    for (int i = 0; i < 5; ++i) {
        const size_t bytes = tensor_elems(w, i) * 4;
        if (bytes == 0) continue;
        if (i < 4 && !src[i]) return TT_ERR_INVALID_ARG;
        if (bytes > w->hbytes[i]) {
            if (w->hbuf[i]) cudaFree(w->hbuf[i]);
            w->hbuf[i] = nullptr; w->hbytes[i] = 0;
            if (cudaMalloc(&w->hbuf[i], bytes) != cudaSuccess) { cudaGetLastError(); return TT_ERR_OOM; }
            w->hbytes[i] = bytes;
        }
        if (i < 4) {
            if (cudaMemcpyAsync(w->hbuf[i], src[i], bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
            up += (int64_t)bytes;
        }
    }
    if (!host->y) return TT_ERR_INVALID_ARG;
    tt_tensors dev{w->hbuf[0], w->hbuf[1], w->hbuf[2], w->hbuf[3], w->hbuf[4]};
    tt_status s = launch(w, &dev, st);
    if (s != TT_OK) return s;
    const size_t ybytes = tensor_elems(w, 4) * 4;
    if (cudaMemcpyAsync(host->y, w->hbuf[4], ybytes, cudaMemcpyDeviceToHost, st) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
    if (synchronise) s = read_status(w, st);
    if (bytes_h2d) *bytes_h2d = up;
    if (bytes_d2h) *bytes_d2h = (int64_t)ybytes;
    return s;
}

tt_status tt_run_host(tt_workload* w, const tt_tensors* host, void* cuda_stream, int64_t* bytes_h2d, int64_t* bytes_d2h) {
    return run_host_impl(w, host, cuda_stream, bytes_h2d, bytes_d2h, true);
}

tt_status tt_run_host_async(tt_workload* w, const tt_tensors* host, void* cuda_stream, int64_t* bytes_h2d, int64_t* bytes_d2h) {
    return run_host_impl(w, host, cuda_stream, bytes_h2d, bytes_d2h, false);
}

tt_status tt_time(tt_workload* w, const tt_tensors* sets, size_t n_sets, void* cuda_stream, const tt_timing_opts* o,
                  tt_timing* out) {
    if (!w || !sets || !out) return TT_ERR_INVALID_ARG;
    if (!w->plan.applied) return TT_ERR_NOT_APPLIED;
    return time_applied(w, sets, n_sets, static_cast<cudaStream_t>(cuda_stream), o, out);
}

static tt_status transfer_tune_impl(tt_workload* const* wls, const tt_tensors* tensors, const size_t* set_counts, size_t n_wl,
                                    const tt_schedule_record* pool, size_t n_pool, const tt_tune_opts* oin, void* cuda_stream,
                                    tt_tune_result* out);

tt_status tt_transfer_tune(tt_workload* const* wls, const tt_tensors* tensors, size_t n_wl, const tt_schedule_record* pool,
                           size_t n_pool, const tt_tune_opts* oin, void* cuda_stream, tt_tune_result* out) {
    return transfer_tune_impl(wls, tensors, nullptr, n_wl, pool, n_pool, oin, cuda_stream, out);
}

tt_status tt_transfer_tune_sets(tt_workload* const* wls, const tt_tensors* tensors, const size_t* set_counts, size_t n_wl,
                                const tt_schedule_record* pool, size_t n_pool, const tt_tune_opts* oin, void* cuda_stream,
                                tt_tune_result* out) {
    if (!set_counts) return TT_ERR_INVALID_ARG;
    for (size_t i = 0; i < n_wl; ++i) if (set_counts[i] == 0) return TT_ERR_INVALID_ARG;
    return transfer_tune_impl(wls, tensors, set_counts, n_wl, pool, n_pool, oin, cuda_stream, out);
}

static tt_status transfer_tune_impl(tt_workload* const* wls, const tt_tensors* tensors, const size_t* set_counts, size_t n_wl,
                                    const tt_schedule_record* pool, size_t n_pool, const tt_tune_opts* oin, void* cuda_stream,
                                    tt_tune_result* out) try {
    if (!wls || !tensors || !out || (n_pool && !pool) || !out->chosen || !out->best_us || !out->times_us || !out->status)
        return TT_ERR_INVALID_ARG;
    tt_tune_opts o{};
    o.include_default = 1;
    if (oin) o = *oin;
    if (!device_present()) return TT_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const auto t_begin = std::chrono::steady_clock::now();
    const size_t n_cols = n_pool + 1;
    int timed = 0, invalid = 0, skipped = 0;
    std::vector<tt_schedule_record> cols(n_cols);
    size_t first_set = 0;
    // pool sub-sampling: the order in which a workload's columns are evaluated -- default first, then the seeded
    // subset, then (only if the subset gained too little over the default) the rest of the pool
    const bool sub = o.subsample_percent > 0 && o.subsample_percent < 100 && n_pool > 1;
    size_t n_first = n_pool;
    std::vector<int32_t> order(n_pool);
    for (size_t j = 0; j < n_pool; ++j) order[j] = (int32_t)j;
    if (sub) {
        n_first = std::max<size_t>(1, (n_pool * (size_t)o.subsample_percent + 99) / 100);
        std::vector<int32_t> firsts(n_first);
        if (tt_pool_subsample(n_pool, n_first, o.subsample_seed, firsts.data()) != TT_OK) return TT_ERR_INVALID_ARG;
        std::vector<char> taken(n_pool, 0);
        size_t k = 0;
        for (int32_t f : firsts) { order[k++] = f; taken[(size_t)f] = 1; }
        for (size_t j = 0; j < n_pool; ++j) if (!taken[j]) order[k++] = (int32_t)j;
    }
    for (size_t i = 0; i < n_wl; ++i) {
        tt_workload* w = wls[i];
        if (!w) return TT_ERR_INVALID_ARG;
        const size_t n_sets = set_counts ? set_counts[i] : 1;
        const tt_tensors* sets = tensors + first_set;
        first_set += n_sets;
        tt_default_schedule(w, &cols[0]);
        for (size_t j = 0; j < n_pool; ++j) cols[j + 1] = pool[j];
        bool stop_early = false;
        float best_first = -1.f;                         // fastest time among the subset's records
        for (size_t step = 0; step < n_cols; ++step) {
            const size_t j = step == 0 ? 0 : (size_t)order[step - 1] + 1;
            float& cell = out->times_us[i * n_cols + j];
            int32_t& cst = out->status[i * n_cols + j];
            cell = -1.f;
            if (sub && step == n_first + 1) {
                // the subset is done: go on only if it did not beat the default record by the asked-for margin
                const float def = out->times_us[i * n_cols];
                stop_early = best_first >= 0.f && def >= 0.f && best_first <= def * (1.f - 0.01f * (float)o.subsample_gain_percent);
            }
            if (stop_early) { cst = TT_SKIPPED; ++skipped; continue; }
            if (j == 0 && !o.include_default) { cst = TT_ERR_INVALID_SCHEDULE; continue; }
            // the default record is the workload's own: never subject to the class rule
            tt_status s = apply_impl(w, &cols[j], j == 0 ? TT_MODE_LEGALISE : o.mode, j == 0 ? 0 : o.strict_class, nullptr);
            if (s == TT_OK) {
                tt_timing tm{};
                s = time_applied(w, sets, n_sets, st, &o.timing, &tm);
                if (s == TT_OK) {
                    cell = tm.median_us; ++timed;
                    if (step >= 1 && step <= n_first && (best_first < 0.f || cell < best_first)) best_first = cell;
                }
            }
            cst = s;
            if (s != TT_OK) {
                if (s == TT_ERR_CUDA || s == TT_ERR_OOM) return s;   // the device is unwell: stop, do not mislabel
                ++invalid;                                          // an invalid pair is a result, not a failure
            }
        }
        tt_select(&out->times_us[i * n_cols], 1, n_cols, &out->chosen[i]);
        const int c = out->chosen[i];
        out->best_us[i] = c >= 0 ? out->times_us[i * n_cols + c] : -1.f;
        if (c >= 0) {
            tt_status s = apply_impl(w, &cols[c], c == 0 ? TT_MODE_LEGALISE : o.mode, c == 0 ? 0 : o.strict_class, nullptr);
            if (s != TT_OK) return s;
        }
    }
    out->pairs_timed = timed; out->pairs_invalid = invalid; out->pairs_skipped = skipped;
    out->search_seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t_begin).count();
    return TT_OK;
} TT_NO_THROW

tt_status tt_grid_tune(tt_workload* w, const tt_tensors* t, void* cuda_stream, const tt_timing_opts* o, int32_t level,
                       size_t top_k, tt_schedule_record* out_records, float* out_us, size_t* n_out, int32_t* n_tried) try {
    if (!w || !t || !out_records || !out_us || !n_out || top_k == 0) return TT_ERR_INVALID_ARG;
    if (!device_present()) return TT_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    tt_schedule_record base;
    tt_default_schedule(w, &base);
    std::vector<tt_schedule_record> cand;
    auto push = [&](const tt_schedule_record& r) -> bool {
        // keep only records that are legal as written: a record that needs rounding duplicates another candidate
        tt_apply_info info;
        if (tt_schedule_check(w, &r, TT_MODE_LEGALISE, 0, &info) != TT_OK) return false;
        // (a pipeline made shallower to fit short reductions or shared memory is kept: exact duplicates are dropped below)
        // (includes a reformulated reduction order; a tap-major tile and the staged depthwise forms are laid out for the kernel's
        // size, and tried as that)
        int free_here = TT_CHG_TILE_M | TT_CHG_STAGES;
        if (info.legal.k_order) free_here |= TT_CHG_TILE_N | TT_CHG_TILE_K | TT_CHG_CLUSTER;
        if (w->family == TT_FAMILY_DW_SIMT && r.raster == 1 && info.legal.raster == 1) free_here |= TT_CHG_BLOCK | TT_CHG_ITEMS | TT_CHG_VEC | TT_CHG_FORM;
        if (info.changed & ~free_here) return false;
        cand.push_back(info.legal);
        return true;
    };
    const bool full = level > 0;
    if (w->family == TT_FAMILY_GEMM_TC) {
        const std::vector<int> tns = full ? std::vector<int>{16, 32, 48, 64, 96, 128, 192, 256} : std::vector<int>{32, 64, 128, 256};
        const std::vector<int> tks = full ? std::vector<int>{8, 16, 32, 64, 128} : std::vector<int>{32, 64, 128};
        const std::vector<int> sts = full ? std::vector<int>{2, 3, 4, 6, 8} : std::vector<int>{2, 3, 4};
        const std::vector<int> sks = full ? std::vector<int>{1, 2, 3, 4, 5, 6, 7, 8, 12, 16, 24, 32} : std::vector<int>{1, 2, 3, 4, 6, 8};
        const std::vector<int> ras = full ? std::vector<int>{0, 1} : std::vector<int>{0};
        for (int ax : {1, 2}) for (int tn : tns) for (int tk : tks) for (int sg : sts) for (int sk : sks) for (int ra : ras) {
            tt_schedule_record r = base;
            r.mma_m_axis = ax; r.tile_m = kHwTileM; r.tile_n = tn; r.tile_k = tk; r.stages = sg; r.split_k = sk; r.raster = ra;
            push(r);
        }
        // the persistent form (alone and as CTA pairs) and the two-CTAs-per-SM build of the one-tile form; on kernels
        // without them these legalise back and are dropped as duplicates-to-be
        for (int ax : {1, 2}) for (int tn : full ? std::vector<int>{32, 64, 128, 192, 240, 256} : std::vector<int>{64, 128, 256})
            for (int tk : {32, 64}) for (int sg : full ? std::vector<int>{2, 3, 4, 6} : std::vector<int>{2, 4, 6}) for (int cg : {1, 2}) {
                tt_schedule_record r = base;
                r.mma_m_axis = ax; r.tile_m = kHwTileM; r.tile_n = tn; r.tile_k = tk; r.stages = sg; r.split_k = 1; r.raster = 0;
                r.persistent = 1; r.cta_group = cg;
                push(r);
            }
        for (int ax : {1, 2}) for (int tn : {64, 128, 256}) for (int sg : {2, 3}) {
            tt_schedule_record r = base;
            r.mma_m_axis = ax; r.tile_m = kHwTileM; r.tile_n = tn; r.tile_k = 32; r.stages = sg; r.split_k = 1; r.raster = 0;
            r.ctas_per_sm = 2;
            push(r);
        }
        if (w->op == TT_OP_CONV2D) {
            for (int tn : {128, 224, 256}) for (int sg : {2, 4}) {
                tt_schedule_record r = base;
                r.mma_m_axis = 1; r.tile_m = kHwTileM; r.tile_n = tn; r.tile_k = 32; r.stages = sg; r.split_k = 1; r.raster = 0;
                r.k_order = 1; r.persistent = 1;
                push(r);
            }
            // a slab that serves one reduction tile per staging: the smallest shared-memory footprint (two CTAs may
            // then share an SM)
            for (int ax : {1, 2}) for (int tn : full ? std::vector<int>{32, 64, 128, 256} : std::vector<int>{64, 128}) for (int sg : {2, 3}) {
                tt_schedule_record r = base;
                r.mma_m_axis = ax; r.tile_m = kHwTileM; r.tile_n = tn; r.tile_k = 32; r.stages = sg; r.split_k = 1; r.raster = 0;
                r.slab_tiles = 1;
                push(r);
            }
            // the tap-major reduction order (records that ask for it on a kernel that has none are legalised back
            // to the stored order and dropped here as duplicates-to-be)
            for (int tn : full ? std::vector<int>{32, 64, 96, 128, 160, 192, 224, 256} : std::vector<int>{64, 128, 224, 256})
                for (int sg : full ? std::vector<int>{1, 2, 3, 4, 5, 6, 8} : std::vector<int>{2, 3, 5}) {
                    tt_schedule_record r = base;
                    r.mma_m_axis = 1; r.tile_m = kHwTileM; r.tile_n = tn; r.tile_k = 32; r.stages = sg; r.split_k = 1; r.raster = 0;
                    r.k_order = 1;
                    push(r);
                }
        }
    } else if (w->family == TT_FAMILY_DW_SIMT) {
        const std::vector<int> tcs = full ? std::vector<int>{1, 2, 4, 8, 16, 32} : std::vector<int>{1, 4, 16};
        const std::vector<int> bys = full ? std::vector<int>{1, 2, 4, 7, 8, 14, 16, 28} : std::vector<int>{4, 8, 16};
        const std::vector<int> bxs = full ? std::vector<int>{8, 16, 28, 32, 56, 64, 112} : std::vector<int>{16, 32, 64};
        const std::vector<int> its = full ? std::vector<int>{1, 2, 4, 8} : std::vector<int>{1, 4};
        for (int tc : tcs) for (int by : bys) for (int bx : bxs) for (int it : its) for (int vw : {1, 4}) for (int th : {128, 256}) {
            tt_schedule_record r = base;
            r.tile_m = tc; r.block_y = by; r.block_x = bx; r.items_per_thread = it; r.vec_width = vw; r.threads = th;
            r.unroll = 0;                               // staged kernel
            push(r);
        }
        // register-window kernel: rows per thread x CTA tile
        const std::vector<int> wys = full ? std::vector<int>{1, 2, 4, 7, 8, 14, 16, 28, 56} : std::vector<int>{4, 8, 16};
        const std::vector<int> wxs = full ? std::vector<int>{8, 16, 28, 32, 56, 64, 112} : std::vector<int>{16, 32, 64, 112};
        for (int it : {4, 8}) for (int ro : {1, 2, 4}) for (int tc : tcs) for (int by : wys) for (int bx : wxs) for (int th : {64, 128, 256}) {
            if (it == 8 && ro == 4) continue;
            tt_schedule_record r = base;
            r.tile_m = tc; r.block_y = by; r.block_x = bx; r.items_per_thread = it; r.threads = th;
            r.unroll = ro;
            for (int vw : {4, 2, 1}) {                  // the widest store the output rows allow
                r.vec_width = vw;
                if (push(r)) break;
            }
        }
        // TMA-staged persistent kernel (raster = 1): strips of 4 or 8 columns, 1-4 rows; tiles span the image width
        // where they can (a box then needs no columns of a neighbouring tile)
        const std::vector<int> pcs = full ? std::vector<int>{1, 2, 4, 8, 16, 32} : std::vector<int>{2, 4, 8, 16};
        const std::vector<int> pys = full ? std::vector<int>{2, 4, 7, 8, 14, 16, 28, 56} : std::vector<int>{4, 8, 14, 28};
        const std::vector<int> pxs = full ? std::vector<int>{16, 28, 32, 56, 64, 112} : std::vector<int>{32, 56, 112};
        for (int it : full ? std::vector<int>{4, 8} : std::vector<int>{4}) for (int ro : {2, 4}) for (int tc : pcs) for (int by : pys)
            for (int bx : pxs) for (int sg : full ? std::vector<int>{2, 3, 4} : std::vector<int>{2, 3}) {
                if (it == 8 && ro == 4) continue;
                tt_schedule_record r = base;
                r.tile_m = tc; r.block_y = by; r.block_x = bx; r.items_per_thread = it; r.threads = 256;
                r.unroll = ro; r.raster = 1; r.stages = sg;
                for (int vw : {4, 2, 1}) {
                    r.vec_width = vw;
                    if (push(r)) break;
                }
            }
    } else {
        for (int bx : {4, 8, 16, 32}) for (int by : {1, 2, 4, 8, 16}) for (int vw : {1, 2, 4}) {
            tt_schedule_record r = base;
            r.block_x = bx; r.block_y = by; r.vec_width = vw;
            push(r);
        }
    }
    if (cand.empty()) {
        // nothing of the grid fits this shape as written: tune around the legalised default record
        tt_apply_info info;
        if (tt_schedule_check(w, &base, TT_MODE_LEGALISE, 0, &info) == TT_OK) cand.push_back(info.legal);
    }
    // drop exact duplicates (legalisation can map different inputs to one record)
    std::vector<tt_schedule_record> uniq;
    for (const auto& r : cand) {
        bool dup = false;
        for (const auto& u : uniq) if (std::memcmp(&u, &r, sizeof r) == 0) { dup = true; break; }
        if (!dup) uniq.push_back(r);
    }
    std::vector<std::pair<float, size_t>> timed;
    for (size_t i = 0; i < uniq.size(); ++i) {
        tt_status s = apply_impl(w, &uniq[i], TT_MODE_LEGALISE, 0, nullptr);
        if (s == TT_ERR_OOM || s == TT_ERR_CUDA) return s;
        if (s != TT_OK) continue;
        tt_timing tm{};
        s = time_applied(w, t, 1, st, o, &tm);
        if (s == TT_ERR_CUDA || s == TT_ERR_OOM) return s;
        if (s == TT_OK) timed.emplace_back(tm.median_us, i);
    }
    if (n_tried) *n_tried = (int32_t)uniq.size();
    std::stable_sort(timed.begin(), timed.end(), [](const auto& a, const auto& b) { return a.first < b.first; });
    const size_t n = std::min(top_k, timed.size());
    for (size_t i = 0; i < n; ++i) {
        out_records[i] = uniq[timed[i].second];
        out_records[i].origin_op = w->op;
        out_records[i].origin = w->sh;
        out_us[i] = timed[i].first;
    }
    *n_out = n;
    if (n > 0) return apply_impl(w, &out_records[0], TT_MODE_LEGALISE, 0, nullptr);
    return TT_ERR_INVALID_SCHEDULE;
} TT_NO_THROW

namespace {
struct RefineCtx { tt_workload* w; const tt_tensors* t; cudaStream_t st; const tt_timing_opts* o; tt_status fatal; };
float refine_time(void* user, const tt_schedule_record* rec) {
    RefineCtx* c = static_cast<RefineCtx*>(user);
    if (c->fatal != TT_OK) return -1.f;
    tt_status s = tt::apply_impl(c->w, rec, TT_MODE_LEGALISE, 0, nullptr);
    if (s == TT_ERR_OOM || s == TT_ERR_CUDA) { c->fatal = s; return -1.f; }
    if (s != TT_OK) return -1.f;
    tt_timing tm{};
    s = tt::time_applied(c->w, c->t, 1, c->st, c->o, &tm);
    if (s == TT_ERR_OOM || s == TT_ERR_CUDA) { c->fatal = s; return -1.f; }
    return s == TT_OK ? tm.median_us : -1.f;
}
}  // namespace

tt_status tt_refine(tt_workload* w, const tt_tensors* t, void* cuda_stream, const tt_timing_opts* o,
                    const tt_schedule_record* start, int32_t max_rounds, float min_gain, tt_schedule_record* best,
                    float* best_us, float* start_us, int32_t* n_timed) {
    if (!w || !t || !start || !best || !best_us) return TT_ERR_INVALID_ARG;
    if (!device_present()) return TT_ERR_CUDA;
    RefineCtx c{w, t, static_cast<cudaStream_t>(cuda_stream), o, TT_OK};
    const tt_status s = tt_refine_with(w, start, refine_time, &c, max_rounds, min_gain, best, best_us, start_us, n_timed);
    if (c.fatal != TT_OK) return c.fatal;
    if (s != TT_OK) return s;
    return tt::apply_impl(w, best, TT_MODE_LEGALISE, 0, nullptr);
}

}  // extern "C"

// ------------------------------------------------------------------------------------------------------------
// Split-K dense layer for callers that must not allocate device memory.
//
// Some hosts of this library cannot call cudaMalloc at the point where they need a kernel: code running inside
// a memory pool that owns the whole device, a real-time loop that may not take the allocator's lock, a plug-in
// whose host application forbids allocations after start-up.  For them the split-K partial sums, the arrival
// counters and the status word live in one fixed array that is part of the library image: every device that
// loads the library carries it until the process exits.
// ------------------------------------------------------------------------------------------------------------
static __device__ __align__(256) unsigned char g_tt_static_scratch[TT_STATIC_SCRATCH_BYTES];

namespace tt {
namespace {
constexpr int kMaxDevices = 64;
constexpr int64_t kStaticStatusBytes = 512;   // the status area, sized like the one tt_schedule_apply allocates
std::atomic<unsigned char*> g_scratch_addr[kMaxDevices] = {};

// In host code the array's name only stands for the symbol; the device address is asked for once per device,
// with that device current.
tt_status static_scratch(unsigned char** out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { cudaGetLastError(); return TT_ERR_CUDA; }
    if (!g_scratch_addr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_tt_static_scratch) != cudaSuccess || !p) { cudaGetLastError(); return TT_ERR_CUDA; }
        g_scratch_addr[dev] = static_cast<unsigned char*>(p);
    }
    *out = g_scratch_addr[dev];
    return TT_OK;
}
}  // namespace
}  // namespace tt

extern "C" tt_status tt_dense_static_scratch(const void* x, const void* w, const void* bias, void* y, int32_t m,
                                             int32_t nn, int32_t kk, int32_t act, const tt_schedule_record* rec,
                                             void* cuda_stream, int64_t* scratch_bytes_used) {
    if (!x || !w || !y || !rec || m <= 0 || nn <= 0 || kk <= 0 || act < TT_ACT_NONE || act > TT_ACT_GELU_ERF)
        return TT_ERR_INVALID_ARG;
    if (!device_present()) return TT_ERR_CUDA;
    // the kernel description, built in place (no handle is created)
    tt_workload wl;
    wl.op = TT_OP_DENSE;
    std::memset(&wl.sh, 0, sizeof wl.sh);
    wl.sh.batch = 1; wl.sh.m = m; wl.sh.nn = nn; wl.sh.kk = kk; wl.sh.trans_b = 1;
    wl.sh.has_bias = bias != nullptr; wl.sh.act = act;
    wl.family = TT_FAMILY_GEMM_TC;
    wl.P = wl.Q = 0;
    wl.view = tt_gemm_view{1, m, nn, kk, 2.0 * m * (double)nn * kk, 0.0};
    Plan plan;
    tt_schedule_record r1 = *rec;
    r1.persistent = 0; r1.cta_group = 1;        // the one-tile-per-CTA form: the persistent one has no split-K, hence no scratch
    tt_status s = legalise(&wl, &r1, TT_MODE_LEGALISE, 0, &plan);
    if (s != TT_OK) return s;
    // layout of the fixed array: status word | arrival counters | partial sums
    const int64_t counters_bytes = ((int64_t)plan.info.grid_x * plan.info.grid_z * 4 + 255) / 256 * 256;
    const int64_t need = kStaticStatusBytes + counters_bytes + (plan.g.split_k > 1 ? plan.partial_bytes : 0);
    if (scratch_bytes_used) *scratch_bytes_used = need;
    if (need > (int64_t)TT_STATIC_SCRATCH_BYTES) return TT_ERR_RESOURCE;   // this record's partial sums do not fit
    if (plan.g.cluster) {
        // as in tt_schedule_apply: a split-K cluster whose CTAs cannot be resident together is an invalid pair
        int fits = 0;
        if (gemm_cluster_fits(plan.g, plan.run_smem, &fits) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
        if (!fits) return TT_ERR_RESOURCE;
    }
    unsigned char* base = nullptr;
    if ((s = static_scratch(&base)) != TT_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    // the array keeps what the previous call left: the status word and the counters must start at zero
    if (cudaMemsetAsync(base, 0, (size_t)(kStaticStatusBytes + counters_bytes), st) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
    GemmArgs g = plan.g;
    const void* tens[2] = {x, w};
    const void* a_ptr = tens[plan.a_tensor];
    const void* b_ptr = tens[plan.b_tensor];
    g.a = static_cast<const float*>(a_ptr);
    g.b = static_cast<const float*>(b_ptr);
    g.y = static_cast<float*>(y);
    g.bias = static_cast<const float*>(bias);
    g.residual = nullptr;
    g.status = reinterpret_cast<unsigned*>(base);
    g.counters = reinterpret_cast<unsigned*>(base + kStaticStatusBytes);
    g.partial = reinterpret_cast<float*>(base + kStaticStatusBytes + counters_bytes);
    g.wait_ns = 1000000000ull;
    g.extra_tx = 0;
    g.w_operand = 0;
    if ((reinterpret_cast<uintptr_t>(y) & 15u) != 0) g.vec_store = 0;
    if (g.bias && (reinterpret_cast<uintptr_t>(g.bias) & 15u) == 0) g.vec_store |= 2;
    TmapPair maps;
    std::memset(&maps, 0, sizeof maps);
    if (g.a_mode == OPM_TMA)
        s = encode_operand(maps.a, g.a, g.K, g.M, g.batch, g.a_rs, g.a_bs, g.a_tma_batched != 0, g.atom_k, kHwTileM);
    if (s == TT_OK && g.b_mode == OPM_TMA)
        s = encode_operand(maps.b, g.b, g.K, g.N, g.batch, g.b_rs, g.b_bs, g.b_tma_batched != 0, g.atom_k, g.tile_n);
    if (g.a_mode == OPM_RAW && (reinterpret_cast<uintptr_t>(g.a) & 15u) != 0) g.a_mode = OPM_GATHER_K;
    if (g.b_mode == OPM_RAW && (reinterpret_cast<uintptr_t>(g.b) & 15u) != 0) g.b_mode = OPM_GATHER_K;
    if (s == TT_OK && g.a_mode == OPM_RAW) s = encode_operand_raw(maps.a, g.a, g.K, g.a_rows_all, g.tile_k, kHwTileM / 4);
    if (s == TT_OK && g.b_mode == OPM_RAW) s = encode_operand_raw(maps.b, g.b, g.K, g.b_rows_all, g.tile_k, g.tile_n / 4);
    if (s != TT_OK) return s;
    if (launch_gemm(plan.info, plan.run_smem, g, maps.a, maps.b, maps.x, st) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
    if (cudaStreamSynchronize(st) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
    unsigned v = 0;
    if (cudaMemcpy(&v, base, 4, cudaMemcpyDeviceToHost) != cudaSuccess) { cudaGetLastError(); return TT_ERR_CUDA; }
    return v ? (tt_status)(v & 0xffu) : TT_OK;
}
