// Host side of the C ABI declared in include/ptq_linear.h: argument validation, parameter
// preparation (padding, reciprocals, tensor maps) and kernel launches.  No compute happens here.
#include "../../include/ptq_linear.h"

#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>
#include <type_traits>
#include <utility>
#include <vector>

#include "ptq_calibrate.cuh"
#include "ptq_fused.cuh"
#include "ptq_gemm.cuh"
#include "ptq_probe.cuh"
#include "ptq_quantize.cuh"
#include "ptq_quantize_dynamic.cuh"
#include "ptq_short_k.cuh"
#include "ptq_small.cuh"

namespace {

thread_local char g_err[512] = "";
std::atomic<unsigned long long> g_launches{0};

ptq_status_t fail(ptq_status_t st, const char *fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return st;
}

#define PTQ_CUDA(...)                                                                          \
    do {                                                                                       \
        cudaError_t e_ = (__VA_ARGS__);                                                        \
        if (e_ != cudaSuccess)                                                                 \
            return fail(e_ == cudaErrorMemoryAllocation ? PTQ_ERR_NOMEM : PTQ_ERR_CUDA,        \
                        "%s failed: %s", #__VA_ARGS__, cudaGetErrorString(e_));                \
    } while (0)

// The body of an entry point that allocates host memory: no exception may leave a C function.
template <class Fn>
ptq_status_t no_throw(Fn fn)
{
    try {
        return fn();
    } catch (const std::exception &) {      // std::bad_alloc is all that these bodies raise
        return fail(PTQ_ERR_NOMEM, "host allocation failed");
    }
}

// cuTensorMapEncodeTiled is reached through the runtime's driver entry point query, so the
// library has no link-time dependency on libcuda and loads on machines without a driver.
typedef CUresult (*encode_tiled_fn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                    const cuuint64_t *, const cuuint32_t *, const cuuint32_t *,
                                    CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                    CUtensorMapFloatOOBfill);

encode_tiled_fn get_encode_tiled()
{
    static encode_tiled_fn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<encode_tiled_fn>(p);
    });
    return fn;
}

// 2-D row-major tensor [rows, cols] with `pitch_bytes` between rows; box [box_rows, box_cols];
// the swizzle mode follows the box's row bytes (128 or 64, which box_cols * elem_bytes must equal);
// out-of-range elements read as zero and are skipped on stores.
ptq_status_t make_map_2d(CUtensorMap *map, CUtensorMapDataType dt, int elem_bytes, const void *ptr,
                         unsigned long long cols, unsigned long long rows, unsigned long long pitch_bytes,
                         unsigned box_cols, unsigned box_rows)
{
    encode_tiled_fn enc = get_encode_tiled();
    if (!enc) return fail(PTQ_ERR_CUDA, "cuTensorMapEncodeTiled entry point not available");
    const unsigned row_bytes = box_cols * elem_bytes;
    if ((row_bytes != 128 && row_bytes != 64) || box_rows == 0 || box_rows > 256)
        return fail(PTQ_ERR_SHAPE, "internal: bad TMA box %u x %u", box_rows, box_cols);
    cuuint64_t dims[2] = {cols, rows};
    cuuint64_t strides[1] = {pitch_bytes};
    cuuint32_t box[2] = {box_cols, box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = enc(map, dt, 2, const_cast<void *>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS)
        return fail(PTQ_ERR_CUDA, "cuTensorMapEncodeTiled failed with CUresult %d (cols %llu rows %llu pitch %llu)",
                    static_cast<int>(r), cols, rows, pitch_bytes);
    return PTQ_OK;
}

// Up to so many k-blocks (K <= 384) the main loop of a tile is short against its epilogue.
constexpr int kShortMainLoop = 3;
static_assert(kShortMainLoop <= ptq::kResMaxKBlocks, "the resident kernel takes every short main loop");

inline int round_up(int v, int m) { return (v + m - 1) / m * m; }

bool ranges_overlap(const void *a, size_t na, const void *b, size_t nb)
{
    const uintptr_t a0 = reinterpret_cast<uintptr_t>(a), b0 = reinterpret_cast<uintptr_t>(b);
    return a0 < b0 + nb && b0 < a0 + na;
}

}  // namespace

// Tensor maps of the caller's buffers, remembered per handle: encoding one costs the host about as much as a
// kernel launch, and a layer is normally called again and again with the same few buffers and batch sizes.
// Keyed by everything the encoding depends on besides the layer (pointer, rows, box width); four entries
// per kind, replaced in turn.  The lock is per handle and held for a lookup or an insertion only.
struct MapCache {
    struct Entry {
        const void *ptr = nullptr;
        long long rows = -1;
        unsigned box_cols = 0;
        CUtensorMap map;
    };
    Entry e[4];
    unsigned next = 0;
    std::mutex mu;
};

struct ptq_linear {
    int K = 0, N = 0, T = 0;
    int Kpad = 0;              // pitch of the codes workspace: K rounded up to 16
    int w_pitch = 0;           // pitch of the padded weight
    int BN = 0, n_tiles = 0;   // GEMM tiling along N
    int k_blocks = 0, last_mmas = 0;
    bool fast_div = false;     // all scales inside the range where the reciprocal route is exact
    int device = -1;
    int num_sms = 0;
    long long l2_bytes = 0;
    unsigned char *d_all = nullptr;   // the one allocation that holds all of the following
    int8_t *d_w = nullptr;     // [n_tiles*BN, w_pitch], zero padded
    float *d_dw = nullptr, *d_bias = nullptr;            // [n_tiles*BN rounded up to 64, +256], zero padded
    float *d_s = nullptr, *d_rs = nullptr;               // [round_up(K,16)]
    float *d_dx = nullptr;                               // [T]
    float2 *d_dx2 = nullptr;                             // [T] {dx, 1/dx}
    int *d_zp = nullptr;                                 // [T] zero offsets (asymmetric layers only)
    int *d_wsum = nullptr;                               // row sums of Wq, padded like d_dw (asymmetric only)
    bool asym = false;
    bool has_bias = false;     // false: d_bias is all zeros
    int act_bits = 8;          // 8: codes in [-128,127] (or [0,255]); 4: codes in [-8,7], one per byte
    unsigned *d_status = nullptr;
    CUtensorMap tmW;
    CUtensorMap tmWh;          // same weights, box of BN/2 rows: the half tile one CTA of a pair loads
    int max_pairs = 0;         // resident 2-CTA clusters of the pair kernel on this device (0: not available)
    // tiling of the fused (A-stationary) kernel
    bool as_ok = false;
    int as_BN = 0, as_n_tiles = 0, as_w_stages = 0, as_w_stage_bytes = 0, as_staging = 0, as_smem = 0;
    CUtensorMap tmWas;
    CUtensorMap tmWsmall;      // box of 128 rows: the one-kernel path for few rows
    CUtensorMap tmWbn[4];      // boxes of 64, 128, 192 and 256 rows: tile widths chosen per call (choose_bn)
    mutable MapCache codes_maps, y_maps;   // tensor maps of caller buffers seen so far
};

namespace {

ptq_status_t check_device(const ptq_linear *h)
{
    int dev = -1;
    PTQ_CUDA(cudaGetDevice(&dev));
    if (dev != h->device)
        return fail(PTQ_ERR_CUDA, "handle belongs to device %d but device %d is current", h->device, dev);
    return PTQ_OK;
}

// make_map_2d through a handle's cache.
ptq_status_t cached_map_2d(MapCache &cache, CUtensorMap *map, CUtensorMapDataType dt, int elem_bytes, const void *ptr,
                           unsigned long long cols, unsigned long long rows, unsigned long long pitch_bytes,
                           unsigned box_cols, unsigned box_rows)
{
    std::lock_guard<std::mutex> lock(cache.mu);
    for (const MapCache::Entry &e : cache.e)
        if (e.ptr == ptr && e.rows == static_cast<long long>(rows) && e.box_cols == box_cols) {
            *map = e.map;
            return PTQ_OK;
        }
    const ptq_status_t st = make_map_2d(map, dt, elem_bytes, ptr, cols, rows, pitch_bytes, box_cols, box_rows);
    if (st != PTQ_OK) return st;
    MapCache::Entry &slot = cache.e[cache.next];
    cache.next = (cache.next + 1u) % 4u;
    slot.ptr = ptr;
    slot.rows = static_cast<long long>(rows);
    slot.box_cols = box_cols;
    slot.map = *map;
    return PTQ_OK;
}

// Opt a kernel in to `bytes` of dynamic shared memory, once per kernel and device (the attribute belongs
// to the function on the CURRENT device, which the callers have checked to be `device`).  The kernel is
// a template argument so that every kernel has its own flags.
template <auto kKern>
ptq_status_t ensure_smem(int device, int bytes)
{
    constexpr int kMaxDevices = 64;
    static std::atomic<bool> done[kMaxDevices] = {};
    if (device < 0 || device >= kMaxDevices) return fail(PTQ_ERR_CUDA, "device index %d out of range", device);
    // lock-free once the attribute is set; two threads racing on the first call both set the same value
    if (!done[device].load(std::memory_order_acquire)) {
        PTQ_CUDA(cudaFuncSetAttribute(kKern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
        done[device].store(true, std::memory_order_release);
    }
    return PTQ_OK;
}

// How many 2-CTA clusters of the pair kernel can be resident at once (0 if cluster launch is unavailable).
int query_max_pairs(int device)
{
    constexpr int kMaxDevices = 64;
    static int cache[kMaxDevices];
    static bool known[kMaxDevices] = {};
    static std::mutex mu;
    if (device < 0 || device >= kMaxDevices) return 0;
    std::lock_guard<std::mutex> lock(mu);
    if (known[device]) return cache[device];
    known[device] = true;                      // per device: attributes and occupancy belong to the current device
    int &cached = cache[device];
    cached = 0;
    if (cudaFuncSetAttribute(ptq::ptq_gemm_dequant_pair_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             ptq::kPairSmemBytes) != cudaSuccess ||
        cudaFuncSetAttribute(ptq::ptq_gemm_dequant_pair_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             ptq::kPairSmemBytes) != cudaSuccess) {
        (void)cudaGetLastError();
        return cached;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2, 1, 1);
    cfg.blockDim = dim3(ptq::kGemmThreads, 1, 1);
    cfg.dynamicSmemBytes = ptq::kPairSmemBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, ptq::ptq_gemm_dequant_pair_kernel<false>, &cfg) == cudaSuccess && n > 0)
        cached = n;
    else
        (void)cudaGetLastError();
    return cached;
}

// Launch with the programmatic-stream-serialization attribute: the kernel may begin (its set-up, up to
// its griddep_wait()) while the previous kernel in the stream drains.  Every kernel launched this way
// calls griddep_wait() before touching anything another kernel may have written.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kern)(KArgs...), int grid, int block, size_t smem, cudaStream_t stream, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(grid), 1, 1);
    cfg.blockDim = dim3(static_cast<unsigned>(block), 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

// Q1 launch for `images` <= kQuantMaxImages images.
ptq_status_t launch_quantize_images(const ptq_linear *h, const void *x, int images, void *q, int q_pitch, cudaStream_t stream)
{
    ptq::QuantParams p;
    p.x = static_cast<const __half *>(x);
    p.q = static_cast<int8_t *>(q);
    p.s = h->d_s;
    p.rs = h->d_rs;
    p.dx2 = h->d_dx2;
    p.zp = h->d_zp;
    p.M = static_cast<long long>(images) * h->T;
    p.K = h->K;
    p.T = h->T;
    p.q_pitch = q_pitch;
    const bool vec = (h->K % 8 == 0) && (reinterpret_cast<uintptr_t>(x) % 16 == 0) &&
                     (reinterpret_cast<uintptr_t>(q) % 8 == 0) && (q_pitch % 8 == 0);
    const int cpr = (h->K + 7) / 8;
    const long long cpi = static_cast<long long>(h->T) * cpr;
    const long long S = ptq::quant_image_step(images, cpi, h->num_sms);     // threads: S * (chunks per image)
    p.B = images;
    p.imgs_per_iter = static_cast<int>(S);
    p.fd_cpi = ptq::make_fastdiv(static_cast<unsigned>(cpi));
    p.fd_cpr = ptq::make_fastdiv(static_cast<unsigned>(cpr));
    const uintptr_t x_align = reinterpret_cast<uintptr_t>(x) | static_cast<uintptr_t>(2 * h->K);
    p.ld_bytes = x_align % 8 == 0 ? 8 : x_align % 4 == 0 ? 4 : 2;
    p.st_bytes = (reinterpret_cast<uintptr_t>(q) % 8 == 0 && q_pitch % 8 == 0) ? 8 : 1;
    const int grid = static_cast<int>((S * cpi + 255) / 256);
    auto go = [&](auto mode, auto fast) -> cudaError_t {
        constexpr int kMode = decltype(mode)::value;
        constexpr bool kFast = decltype(fast)::value;
        return vec ? launch_pdl(ptq::ptq_quantize_vec8_kernel<kFast, kMode, false>, grid, 256, 0, stream, p)
                   : launch_pdl(ptq::ptq_quantize_vec8_kernel<kFast, kMode, true>, grid, 256, 0, stream, p);
    };
    auto pick = [&](auto mode) { return h->fast_div ? go(mode, std::true_type()) : go(mode, std::false_type()); };
    if (h->act_bits == 4)
        PTQ_CUDA(pick(std::integral_constant<int, ptq::kCodeS4>()));
    else if (h->asym)
        PTQ_CUDA(pick(std::integral_constant<int, ptq::kCodeU8>()));
    else
        PTQ_CUDA(pick(std::integral_constant<int, ptq::kCodeS8>()));
    g_launches.fetch_add(1, std::memory_order_relaxed);
    PTQ_CUDA(cudaGetLastError());
    return PTQ_OK;
}

// Q1: codes of M rows to `q` with `q_pitch` bytes between rows.
ptq_status_t launch_quantize(const ptq_linear *h, const void *x, long long M, void *q, int q_pitch, cudaStream_t stream)
{
    const long long B = M / h->T;
    for (long long b = 0; b < B; b += ptq::kQuantMaxImages) {
        const int images = static_cast<int>(B - b < ptq::kQuantMaxImages ? B - b : ptq::kQuantMaxImages);
        const ptq_status_t st = launch_quantize_images(h, static_cast<const __half *>(x) + b * h->T * h->K, images,
                                                       static_cast<int8_t *>(q) + b * h->T * q_pitch, q_pitch, stream);
        if (st != PTQ_OK) return st;
    }
    return PTQ_OK;
}

// Dynamic comparator: codes to `q` and the per-row steps to `dx_row`.
ptq_status_t launch_quantize_dynamic(const ptq_linear *h, const void *x, long long M, void *q, int q_pitch,
                                     float *dx_row, cudaStream_t stream)
{
    ptq::DynQuantParams p;
    p.x = static_cast<const __half *>(x);
    p.q = static_cast<int8_t *>(q);
    p.dx_row = dx_row;
    p.s = h->d_s;
    p.rs = h->d_rs;
    p.M = M;
    p.K = h->K;
    p.q_pitch = q_pitch;
    const bool vec = (h->K % 8 == 0) && (reinterpret_cast<uintptr_t>(x) % 16 == 0) &&
                     (reinterpret_cast<uintptr_t>(q) % 8 == 0) && (q_pitch % 8 == 0);
    const int chunks = (h->K / 8 + 31) / 32;                   // per lane, one row per warp
    const bool row = vec && h->fast_div && chunks <= 6;
    const int lanes = chunks > 1 || h->K > 128 ? 32 : h->K > 64 ? 16 : 8;
    const long long rows_per_cta = row ? 256 / lanes : vec ? 8 * ptq::kDynRowsPerWarp : 8;
    long long want = (M + rows_per_cta - 1) / rows_per_cta;
    const long long cap = static_cast<long long>(h->num_sms) * (row ? ptq::dyn_row_ctas_per_sm(chunks) : 8);
    if (want > cap) want = cap;
    if (want < 1) want = 1;
    if (row) {
        auto go = [&](auto n, auto l) {
            return launch_pdl(ptq::ptq_quantize_dynamic_row_kernel<decltype(n)::value, decltype(l)::value>, static_cast<int>(want), 256, 0, stream, p);
        };
        const std::integral_constant<int, 32> warp;
        switch (chunks) {
            case 1:
                if (lanes == 8)
                    PTQ_CUDA(go(std::integral_constant<int, 1>(), std::integral_constant<int, 8>()));
                else if (lanes == 16)
                    PTQ_CUDA(go(std::integral_constant<int, 1>(), std::integral_constant<int, 16>()));
                else
                    PTQ_CUDA(go(std::integral_constant<int, 1>(), warp));
                break;
            case 2: PTQ_CUDA(go(std::integral_constant<int, 2>(), warp)); break;
            case 3: PTQ_CUDA(go(std::integral_constant<int, 3>(), warp)); break;
            case 4: PTQ_CUDA(go(std::integral_constant<int, 4>(), warp)); break;
            case 5: PTQ_CUDA(go(std::integral_constant<int, 5>(), warp)); break;
            default: PTQ_CUDA(go(std::integral_constant<int, 6>(), warp)); break;
        }
    } else if (!vec)
        PTQ_CUDA(launch_pdl(ptq::ptq_quantize_dynamic_scalar_kernel, static_cast<int>(want), 256, 0, stream, p));
    else if (h->fast_div)
        PTQ_CUDA(launch_pdl(ptq::ptq_quantize_dynamic_vec8_kernel<true>, static_cast<int>(want), 256, 0, stream, p));
    else
        PTQ_CUDA(launch_pdl(ptq::ptq_quantize_dynamic_vec8_kernel<false>, static_cast<int>(want), 256, 0, stream, p));
    g_launches.fetch_add(1, std::memory_order_relaxed);
    PTQ_CUDA(cudaGetLastError());
    return PTQ_OK;
}

// Per-channel vectors a GEMM kernel keeps in shared memory: weight steps, bias, and (short main loops) row sums.
void set_vectors(const ptq_linear *h, ptq::GemmParams &p)
{
    p.ws_copy = h->asym && h->k_blocks <= kShortMainLoop ? 1 : 0;
    p.vectors = 1 + p.has_bias + p.ws_copy;
}

// Whether this launch takes the panel kernel (the codes of a row panel resident in shared memory for a
// group of N tiles), and with which tiling: fills p.group, p.groups, p.b_stages, p.b_stage_bytes.
// It pays on large compute-bound layers only (measured: 2-3 % of the Vim-B step, nothing or a loss on
// layers with K <= 384 or few tiles), so it is taken when the layer has at least four k-blocks and
// eight tiles per SM, and only with a group size G whose work units divide over the CTAs as evenly as
// single tiles do: rounds(G) * G <= rounds(1).  Among those the largest G wins (fewest panel loads).
bool plan_panel(const ptq_linear *h, ptq::GemmParams &p, bool tma_store)
{
    p.group = p.groups = p.b_stages = p.b_stage_bytes = 0;
    const long long tiles = static_cast<long long>(p.m_tiles) * p.n_tiles;
    if (!tma_store || p.n_tiles < 2 || p.k_blocks < 4 || p.k_blocks > ptq::kPanelMaxKBlocks ||
        tiles < 8ll * h->num_sms)
        return false;
    const int stage_bytes = p.BN * ptq::kBK;
    const int fixed = ptq::panel_smem_bytes(p.k_blocks, 0, 0, p.boxes, p.vectors);
    int stages = (ptq::kPanelSmemLimit - fixed) / stage_bytes;
    if (stages < 3) return false;
    if (stages > ptq::kPanelMaxBStages) stages = ptq::kPanelMaxBStages;
    const long long rounds1 = (tiles + h->num_sms - 1) / h->num_sms;
    int best_g = 1;
    for (int g = 2; g <= p.n_tiles; ++g) {
        const long long units = static_cast<long long>((p.n_tiles + g - 1) / g) * p.m_tiles;
        const long long grid = units < h->num_sms ? units : h->num_sms;
        const long long rounds = (units + grid - 1) / grid;
        if (rounds * g <= rounds1) best_g = g;
    }
    if (best_g < 2) return false;
    p.group = best_g;
    p.groups = (p.n_tiles + best_g - 1) / best_g;
    p.fd_groups = ptq::make_fastdiv(static_cast<unsigned>(p.groups));
    p.b_stages = stages;
    p.b_stage_bytes = stage_bytes;
    return true;
}

// Whether the kernel with resident weights (and its epilogue in two teams) is taken: short main loop (K <= 384) and TMA stores.  Symmetric layers
// from more than one tile for the busiest CTA: against the streaming kernel below three, 116 random layers with 1 to 14 tiles per CTA
// (33 <= K <= 384), each replayed alone, take 0.957 of the time, 18321 x 298 -> 592 17.4 / 15.4 us, 50176 x 384 -> 192 17.4 / 16.8, 12608 x 192 -> 768 9.78 /
// 9.43; none is slower by more than 1 % (10047 x 64 -> 1176 10.0 / 9.9, 17927 x 48 -> 96 6.5 / 6.2).  Among other layers less of it is left, because
// every further kernel in turn has to be fetched into the SMs again: in_proj and out_proj of Vim-Ti at batch 64 take 18.6 us with both
// in one kernel and 19.1 with one in each.  So a layer of one tile per CTA that narrows by half, as the last of a block does, takes it where
// the block's first one, on the same rows and four times as wide as this one, makes more tiles than SMs, with half as many row tiles as SMs or more
// (below that no difference).  Both streaming / both resident / so, us: 128 -> 512 and 256 -> 128 on 92 row tiles, twice, 32.5 / 31.3 / 31.5, 112 -> 448 and
// 224 -> 112 on 148 37.8 / 36.8 / 34.8; where the first one is a tile per CTA too, 64 -> 256 and 128 -> 64 on 130, 26.4 / 26.4 / 26.4, 27.2 with one in
// each.  Up to 48 columns it is taken below two thirds of the SMs, where that costs nothing (48 -> 192 and 96 -> 48 on 76 24.6 / 24.0, with one
// in each 24.8; on 148 26.4 / 27.0 / 27.3).  Others do not take it, they lose, 206 -> 208 and 75 -> 33 on 140 row tiles 19.8 / 21.1, 91 -> 179 among
// 463 -> 199 and two narrow ones on 96 37.2 / 37.9; beside K > 384 narrowing ones lose too, up to 3 % (298 -> 112 before 596 -> 190 on 80
// 23.0 / 23.7), which a layer cannot know.  Asymmetric layers from three tiles: 6304 x 384 -> 1536 alone 12.2 / 11.9, but with 6304 x 768 -> 384
// behind it 24.4 / 24.55.
bool takes_resident(const ptq_linear *h, int m_tiles, int n_tiles)
{
    if (h->k_blocks > kShortMainLoop) return false;
    const long long sms = h->num_sms, rows = m_tiles, tiles = rows * n_tiles;
    if (h->asym) return tiles >= 3 * sms;
    if (tiles > sms) return true;
    const long long first_tiles = rows * ((4ll * h->N + ptq::kMaxBN - 1) / ptq::kMaxBN);
    return 2ll * h->N <= h->K && 2 * rows >= sms && (first_tiles > sms || (h->N <= 48 && 3 * rows < 2 * sms));
}

// N tiles per unit of the kernel with resident weights: all of them where their weights fit in shared memory and the busiest CTA gets no more
// tiles, else one.  A row panel's codes are then loaded once, and its output is written as whole rows at a time.  Both kernels, us, one / all:
// 200704 x 96 -> 384 41.3 / 39.7, 50176 x 128 -> 512 17.7 / 17.3, the same asymmetric 20.9 / 20.9, 50176 x 96 -> 384 14.6 / 14.1; with a tile more for the
// busiest CTA 100352 x 96 -> 384 (11 / 12 tiles) 22.1 / 22.6.  Some of them gain nothing: 50176 x 48 -> 1000 in pairs of four 36.9 / 36.7.
int resident_group(const ptq_linear *h, const ptq::GemmParams &p)
{
    const long long sms = h->num_sms, tiles = static_cast<long long>(p.m_tiles) * p.n_tiles;
    if (p.n_tiles == 1 || ptq::res_smem_bytes(p.k_blocks, p.n_tiles, p.BN, p.vectors) > ptq::kResSmemMax) return 1;
    return (p.m_tiles + sms - 1) / sms * p.n_tiles <= (tiles + sms - 1) / sms ? p.n_tiles : 1;
}

// Cycles of one tile of `cols` columns in the streaming kernel, as fitted to timings of 24 shapes at all widths: an MMA of K = 32
// takes 35 + 0.52 cols; the eight epilogue warps take 360 per tile and 670 per pair of 64-column steps.
double mma_cycles(const ptq_linear *h, int cols) { return (h->K + 31) / 32 * (35.0 + 0.52 * cols); }
double epilogue_cycles(int cols) { return 360.0 + 670.0 * (((cols + 63) / 64 + 1) / 2); }

// Columns per piece of the streaming kernel's last round with tiles of `bn` columns, 0 where it is not cut: at least one full
// round before it, SMs enough for all pieces at once (narrow ones first), and a long main loop: the epilogue gains little by
// a narrower tile.  GEMM kernel alone, us, whole and cut, at the width that is chosen: 6304 x 1536 -> 768 (256 columns) 10.7 -> 8.9,
// 6304 x 768 -> 3072 (256) 15.8 -> 14.8, 1568 x 768 -> 3072 (192) 7.0 -> 6.7, 3136 x 768 -> 3072 (256) 10.2 -> 9.5; with K <= 384 25088 x 384 -> 192
// (192) 5.12 -> 5.14, 12608 x 192 -> 768 (192) 6.3 -> 6.3, 6304 x 384 -> 1536 (192) 6.8 -> 6.8.  (Of whole forward passes with K <= 384 one gained by a
// cut: 25088 x 384 -> 192 16.5 -> 15.9; 12608 x 192 -> 768 10.7 -> 10.7, 6304 x 384 -> 768 9.6 -> 9.4.)
// Every tile of the round counts with all its pieces: those of an N tile that ends early and lie wholly beyond N are issued too, load zero
// weights, multiply and store nothing.
int cut_cols(const ptq_linear *h, const ptq::GemmParams &p, int bn)
{
    const long long tiles = static_cast<long long>(p.m_tiles) * ((h->N + bn - 1) / bn), last = tiles % h->num_sms;
    if (tiles < h->num_sms || last == 0 || h->k_blocks <= kShortMainLoop) return 0;
    for (int cols = 64; cols <= 128 && cols < bn; cols += 64)
        if (last * ((bn + cols - 1) / cols) <= h->num_sms) return cols;
    return 0;
}

// Cycles of the busiest CTA of the streaming kernel with tiles of `bn` columns; the hand-overs take 420 per tile.  Of what a cut
// last round should save nine tenths are believed.
double gemm_cycles(const ptq_linear *h, const ptq::GemmParams &p, int bn)
{
    const long long tiles = static_cast<long long>(p.m_tiles) * ((h->N + bn - 1) / bn);
    const double rounds = static_cast<double>((tiles + h->num_sms - 1) / h->num_sms);
    auto longer = [](double a, double b) { return a > b ? a : b; };
    auto busiest = [&](int last) {                                            // columns of the last round's tiles
        if (rounds < 2.0) return mma_cycles(h, last) + epilogue_cycles(last) + 420.0;
        return mma_cycles(h, bn) + (rounds - 2.0) * longer(mma_cycles(h, bn), epilogue_cycles(bn)) +
               longer(mma_cycles(h, last), epilogue_cycles(bn)) + epilogue_cycles(last) + 420.0 * rounds;
    };
    const int cut = cut_cols(h, p, bn);
    return cut ? 0.9 * busiest(cut) + 0.1 * busiest(bn) : busiest(bn);
}

// Tile width for this many rows, in the streaming kernel and below three rounds in the one with resident weights: the layer's own (as few N
// tiles as possible), unless another leaves the busiest CTA clearly less to do: idle SMs in a single round, or a last round that is nearly empty.  GEMM kernel alone,
// us, own width -> the one chosen: 2793 x 1536 -> 768 (256 -> 128) 7.4 -> 5.3, 1568 x 1536 -> 768 (256 -> 128) 7.3 -> 4.9, 3152 x 768 -> 384 (192 -> 128)
// 4.7 -> 3.8, 12544 x 768 -> 384 (192, cut -> 128) 6.6 -> 6.1, 11229 x 520 -> 600 (256 -> 128) 8.9 -> 8.6, 12608 x 192 -> 768 (256 -> 192) 6.6 -> 6.3.
// The margin keeps what the model cannot tell apart: 25216 x 768 -> 384 (192 -> 128, predicted -1.6 %) 10.7 -> 10.9.  What it gets wrong: 6304 x 768 ->
// 384 keeps 192 columns, 5.0, where 128 with a cut round take 4.5, and 6304 x 384 -> 192 takes 128, 3.4, where 64 take 3.1.  Whole forward passes of 1536
// random layers, every width: the chosen one 0.4 % above the best on average; the furthest off 1078 x 46 -> 3072 with a bias (192 columns, 7.7,
// where 256 take 6.9), 13867 x 298 -> 384 (128, 15.2, where 192 take 14.1) and 5047 x 576 -> 600 dynamic (128, cut, 14.0, where 256 take 13.0).  Wider
// margins, less belief in the cut and a second round forbidden were tried on them: each slows as many layers as it mends.  With a
// short main loop and three rounds or more the widths are not compared: they are within 3 % of one another either way.  With fewer the
// kernel with resident weights takes the width chosen here (116 random layers: 1.3 % above the best of the four widths on average; furthest off
// 14578 x 320 -> 640 asymmetric, 256 columns 14.9 where 128 take 12.6).
constexpr long long kOwnWidthRounds = 3;
int choose_bn(const ptq_linear *h, const ptq::GemmParams &p)
{
    auto many = [&](int bn) {
        return h->k_blocks <= kShortMainLoop && static_cast<long long>(p.m_tiles) * ((h->N + bn - 1) / bn) >= kOwnWidthRounds * h->num_sms;
    };
    int best = h->BN;
    if (many(best)) return best;
    double best_cost = 0.975 * gemm_cycles(h, p, best);
    for (int bn = 64; bn <= ptq::kMaxBN && bn < h->N + 64; bn += 64) {
        if (many(bn)) continue;
        const double cost = gemm_cycles(h, p, bn);
        if (cost < best_cost) {
            best = bn;
            best_cost = cost;
        }
    }
    return best;
}

void set_bn(const ptq_linear *h, ptq::GemmParams &p, int bn)
{
    p.BN = bn;
    p.n_tiles = (h->N + bn - 1) / bn;
    p.fd_n_tiles = ptq::make_fastdiv(static_cast<unsigned>(p.n_tiles));
}

// Which of the streaming and the resident kernel takes a launch, with tiles of how many columns, and of how many each piece of its
// last round (0: whole).  p.BN and the numbers of tiles are set to it.
struct Tiling {
    int bn = 0, cut = 0;
    bool resident = false;
};
Tiling choose_tiling(const ptq_linear *h, ptq::GemmParams &p, bool tma_store)
{
    Tiling t;
    t.bn = choose_bn(h, p);
    if (t.bn != h->BN) set_bn(h, p, t.bn);
    t.resident = tma_store && takes_resident(h, p.m_tiles, p.n_tiles);
    t.cut = t.resident ? 0 : cut_cols(h, p, t.bn);
    return t;
}

// Parameters of the GEMM kernels at the layer's own tile width.
void set_gemm_params(const ptq_linear *h, ptq::GemmParams &p, long long M, void *y, void *acc_out, bool tma_store, const float *dx_rows)
{
    p.M = M;
    p.N = h->N;
    p.K = h->K;
    p.T = dx_rows ? static_cast<int>(M) : h->T;
    p.BN = h->BN;
    p.n_tiles = h->n_tiles;
    p.m_tiles = static_cast<int>((M + ptq::kBM - 1) / ptq::kBM);
    p.k_blocks = h->k_blocks;
    p.last_mmas = h->last_mmas;
    p.dx = dx_rows ? dx_rows : h->d_dx;
    p.dw = h->d_dw;
    p.bias = h->d_bias;
    p.has_bias = h->has_bias ? 1 : 0;
    set_vectors(h, p);
    // Short main loops (up to three k-blocks per tile, K <= 384) leave the epilogue little time: three stages and two
    // staging boxes per warp; longer ones keep four stages.  Layers with a bias hold two more scale copies.
    const bool short_k = h->k_blocks <= kShortMainLoop;
    p.stages = (short_k || h->has_bias) ? ptq::kStages - 1 : ptq::kStages;
    p.boxes = short_k ? 2 : 1;
    p.y = static_cast<__half *>(y);
    p.acc_out = static_cast<int32_t *>(acc_out);
    p.status = h->d_status;
    p.use_tma_store = tma_store ? 1 : 0;
    p.y_vec2 = (h->N % 2 == 0 && reinterpret_cast<uintptr_t>(y) % 4 == 0) ? 1 : 0;
    p.y_vec8 = 0;   // this kernel always has a staging buffer; 16-byte alignment means TMA stores
    // An output of more than half of L2 is gone before its consumer reads it all: marked evict-first it does not push out the
    // codes, which this kernel is still reading (50432 x 768 -> 3072, both kernels: 132.7 -> 129.2 us).
    p.y_evict_first = static_cast<long long>(M) * h->N * 2 > h->l2_bytes / 2;
    const uintptr_t y_align = reinterpret_cast<uintptr_t>(y) | static_cast<uintptr_t>(2 * h->N);
    p.y_copy_bytes = y_align % 8 == 0 ? 8 : y_align % 4 == 0 ? 4 : 2;
    p.zp = h->d_zp;
    p.wsum = h->d_wsum;
    p.fd_T = ptq::make_fastdiv(static_cast<unsigned>(p.T));
    p.fd_n_tiles = ptq::make_fastdiv(static_cast<unsigned>(p.n_tiles));
    p.fd_groups = ptq::make_fastdiv(1u);
}

// G1+E1 launch on codes [M, Kpad] at `codes`.
// dx_rows != nullptr: the steps are per ROW (dynamic comparator), i.e. dx = dx_rows and T = M.
ptq_status_t launch_gemm(const ptq_linear *h, const void *codes, long long M, void *y, void *acc_out,
                         cudaStream_t stream, bool want_pair = false, const float *dx_rows = nullptr)
{
    CUtensorMap tmA, tmY;
    ptq_status_t st = cached_map_2d(h->codes_maps, &tmA, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, codes,
                                    static_cast<unsigned long long>(h->K), static_cast<unsigned long long>(M),
                                    static_cast<unsigned long long>(h->Kpad), ptq::kBK, ptq::kBM);
    if (st != PTQ_OK) return st;
    const bool tma_store = (h->N % 8 == 0) && (reinterpret_cast<uintptr_t>(y) % 16 == 0);
    const int m_tiles_ = static_cast<int>((M + ptq::kBM - 1) / ptq::kBM);
    const bool use_pair = want_pair && h->max_pairs > 0 && !h->has_bias &&
                          static_cast<long long>((m_tiles_ + 1) / 2) * h->n_tiles >= h->max_pairs;
    if (tma_store) {
        st = cached_map_2d(h->y_maps, &tmY, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, y, static_cast<unsigned long long>(h->N),
                           static_cast<unsigned long long>(M), static_cast<unsigned long long>(h->N) * 2,
                           ptq::kStreamBoxCols, 32);
        if (st != PTQ_OK) return st;
    } else {
        tmY = h->tmW;   // never dereferenced by the kernel in this mode
    }

    ptq::GemmParams p;
    set_gemm_params(h, p, M, y, acc_out, tma_store, dx_rows);
    const int gemm_smem = ptq::gemm_smem_bytes(p.stages, p.boxes, p.vectors);

    if (use_pair) {
        // enough 256-row tiles to occupy every CTA pair: cta_group::2 kernel (half the weight bytes per CTA)
        const int npairs = h->max_pairs;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(2 * npairs, 1, 1);
        cfg.blockDim = dim3(ptq::kGemmThreads, 1, 1);
        cfg.dynamicSmemBytes = ptq::kPairSmemBytes;
        cfg.stream = stream;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = 2;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (acc_out)
            PTQ_CUDA(cudaLaunchKernelEx(&cfg, ptq::ptq_gemm_dequant_pair_kernel<true>, tmA, h->tmWh, tmY, p));
        else
            PTQ_CUDA(cudaLaunchKernelEx(&cfg, ptq::ptq_gemm_dequant_pair_kernel<false>, tmA, h->tmWh, tmY, p));
        g_launches.fetch_add(1, std::memory_order_relaxed);
        PTQ_CUDA(cudaGetLastError());
        return PTQ_OK;
    }
    const bool dbg = acc_out != nullptr;
    if (plan_panel(h, p, tma_store)) {
        // several N tiles and 512 <= K <= 768: the codes of a row panel stay in shared memory for `group` tiles
        const int psmem = ptq::panel_smem_bytes(p.k_blocks, p.b_stages, p.b_stage_bytes, p.boxes, p.vectors);
        const long long units = static_cast<long long>(p.m_tiles) * p.groups;
        const int pgrid = static_cast<int>(units < h->num_sms ? units : h->num_sms);
        auto panel = [&](auto debug, auto asym) -> ptq_status_t {
            constexpr auto kKern = ptq::ptq_gemm_dequant_panel_kernel<decltype(debug)::value, decltype(asym)::value>;
            const ptq_status_t es = ensure_smem<kKern>(h->device, ptq::kPanelSmemLimit);
            if (es != PTQ_OK) return es;
            PTQ_CUDA(launch_pdl(kKern, pgrid, ptq::kGemmThreads, psmem, stream, tmA, h->tmW, tmY, p));
            return PTQ_OK;
        };
        const ptq_status_t ps = h->asym ? (dbg ? panel(std::true_type(), std::true_type()) : panel(std::false_type(), std::true_type()))
                                        : (dbg ? panel(std::true_type(), std::false_type()) : panel(std::false_type(), std::false_type()));
        if (ps != PTQ_OK) return ps;
        g_launches.fetch_add(1, std::memory_order_relaxed);
        PTQ_CUDA(cudaGetLastError());
        return PTQ_OK;
    }
    const Tiling tiling = choose_tiling(h, p, tma_store);
    const int bn = tiling.bn, cut = tiling.cut;
    const CUtensorMap &tmW = bn != h->BN ? h->tmWbn[bn / 64 - 1] : h->tmW;
    const long long tiles = static_cast<long long>(p.m_tiles) * p.n_tiles;
    const int grid = static_cast<int>(tiles < h->num_sms ? tiles : h->num_sms);
    auto go = [&](auto debug, auto asym) -> ptq_status_t {
        constexpr bool kDbg = decltype(debug)::value, kAsym = decltype(asym)::value;
        if (tiling.resident) {
            constexpr auto kKern = ptq::ptq_gemm_dequant_resident_kernel<kDbg, kAsym>;
            ptq::UnitParams rp;
            static_cast<ptq::GemmParams &>(rp) = p;
            rp.group = resident_group(h, p);
            rp.stages = ptq::res_stages(h->K, h->N);
            rp.groups = (p.n_tiles + rp.group - 1) / rp.group;
            const long long units = static_cast<long long>(p.m_tiles) * rp.groups;
            const int rgrid = static_cast<int>(units < h->num_sms ? units : h->num_sms);
            ptq::set_units(rp, rgrid);
            const ptq_status_t es = ensure_smem<kKern>(h->device, ptq::kResSmemMax);
            if (es != PTQ_OK) return es;
            const int smem = ptq::res_smem_bytes(p.k_blocks, rp.group, p.BN, p.vectors);
            PTQ_CUDA(launch_pdl(kKern, rgrid, ptq::kGemmThreads, smem, stream, tmA, tmW, tmY, rp));
        } else if (cut) {
            constexpr auto kKern = ptq::ptq_gemm_dequant_kernel<kDbg, kAsym, ptq::GemmCutParams>;
            ptq::GemmCutParams cp;
            static_cast<ptq::GemmParams &>(cp) = p;
            cp.tmWcut = h->tmWbn[cut / 64 - 1];
            cp.full_tiles = static_cast<int>(tiles / h->num_sms) * h->num_sms;
            cp.piece_cols = cut;
            cp.pieces = (bn + cut - 1) / cut;
            cp.fd_pieces = ptq::make_fastdiv(static_cast<unsigned>(cp.pieces));
            const ptq_status_t es = ensure_smem<kKern>(h->device, ptq::kGemmSmemBytes);
            if (es != PTQ_OK) return es;
            PTQ_CUDA(launch_pdl(kKern, grid, ptq::kGemmThreads, gemm_smem, stream, tmA, tmW, tmY, cp));
        } else {
            constexpr auto kKern = ptq::ptq_gemm_dequant_kernel<kDbg, kAsym, ptq::GemmParams>;
            const ptq_status_t es = ensure_smem<kKern>(h->device, ptq::kGemmSmemBytes);
            if (es != PTQ_OK) return es;
            PTQ_CUDA(launch_pdl(kKern, grid, ptq::kGemmThreads, gemm_smem, stream, tmA, tmW, tmY, p));
        }
        return PTQ_OK;
    };
    const ptq_status_t gs = h->asym ? (dbg ? go(std::true_type(), std::true_type()) : go(std::false_type(), std::true_type()))
                                    : (dbg ? go(std::true_type(), std::false_type()) : go(std::false_type(), std::false_type()));
    if (gs != PTQ_OK) return gs;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    PTQ_CUDA(cudaGetLastError());
    return PTQ_OK;
}

// Tiling of the A-stationary kernel for a layer: the code panel (k_blocks x 16 KB) stays resident, the
// rest of shared memory holds weight stages and, if it fits, the epilogue's staging buffers.
void choose_astat(ptq_linear *h)
{
    h->as_ok = false;
    if (h->k_blocks > ptq::kFusedMaxKBlocks) return;
    const int cand_bn[3] = {h->BN, 128, 64};
    for (int staging = 1; staging >= 0 && !h->as_ok; --staging) {
        for (int c = 0; c < 3 && !h->as_ok; ++c) {
            int bn = cand_bn[c];
            if (c > 0 && bn >= h->BN) continue;
            const int n_tiles = (c == 0) ? h->n_tiles : (h->N + bn - 1) / bn;
            const int stage_bytes = bn * ptq::kBK;
            const int fixed = ptq::fused_smem_bytes(h->k_blocks, 0, 0, staging);
            int stages = (ptq::kFusedSmemLimit - fixed) / stage_bytes;
            if (stages < 2) continue;
            if (stages > ptq::kFusedMaxWStages) stages = ptq::kFusedMaxWStages;
            h->as_ok = true;
            h->as_BN = bn;
            h->as_n_tiles = n_tiles;
            h->as_w_stages = stages;
            h->as_w_stage_bytes = stage_bytes;
            h->as_staging = staging;
            h->as_smem = ptq::fused_smem_bytes(h->k_blocks, stages, stage_bytes, staging);
        }
    }
}

template <auto kKern>
ptq_status_t launch_fused_kernel(const ptq_linear *h, const CUtensorMap &tmY, const ptq::FusedParams &fp, int grid,
                                 cudaStream_t stream)
{
    const ptq_status_t attr_status = ensure_smem<kKern>(h->device, ptq::kFusedSmemLimit);
    if (attr_status != PTQ_OK) return attr_status;
    kKern<<<grid, ptq::kFusedThreadsQuant, h->as_smem, stream>>>(h->tmWas, tmY, fp);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    PTQ_CUDA(cudaGetLastError());
    return PTQ_OK;
}

// F1 launch: x fp16 [M,K] -> y (Q1 + G1 + E1 in one kernel, the code panel of a row tile resident in shared memory).
ptq_status_t launch_fused(const ptq_linear *h, const void *x, long long M, void *y, void *acc_out, cudaStream_t stream)
{
    CUtensorMap tmY;
    ptq_status_t st;
    const bool aligned = (h->N % 8 == 0) && (reinterpret_cast<uintptr_t>(y) % 16 == 0);
    const bool tma_store = aligned && h->as_staging;
    if (tma_store) {
        st = cached_map_2d(h->y_maps, &tmY, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, y, static_cast<unsigned long long>(h->N),
                           static_cast<unsigned long long>(M), static_cast<unsigned long long>(h->N) * 2,
                           ptq::kStoreBoxCols, 32);
        if (st != PTQ_OK) return st;
    } else {
        tmY = h->tmWas;   // never dereferenced by the kernel in this mode
    }
    ptq::FusedParams fp;
    ptq::GemmParams &p = fp.g;
    p.M = M;
    p.N = h->N;
    p.K = h->K;
    p.T = h->T;
    p.BN = h->as_BN;
    p.n_tiles = h->as_n_tiles;
    p.m_tiles = static_cast<int>((M + ptq::kBM - 1) / ptq::kBM);
    p.k_blocks = h->k_blocks;
    p.last_mmas = h->last_mmas;
    p.dx = h->d_dx;
    p.dw = h->d_dw;
    p.bias = h->d_bias;
    p.has_bias = h->has_bias ? 1 : 0;
    p.vectors = 1;
    p.ws_copy = 0;
    p.y = static_cast<__half *>(y);
    p.acc_out = static_cast<int32_t *>(acc_out);
    p.status = h->d_status;
    p.use_tma_store = tma_store ? 1 : 0;
    p.y_vec2 = (h->N % 2 == 0 && reinterpret_cast<uintptr_t>(y) % 4 == 0) ? 1 : 0;
    p.y_vec8 = (aligned && !tma_store) ? 1 : 0;
    p.y_copy_bytes = 2;   // not used by this kernel
    p.y_evict_first = 0;
    p.zp = nullptr;
    p.wsum = nullptr;
    fp.x = static_cast<const __half *>(x);
    fp.s = h->d_s;
    fp.rs = h->d_rs;
    fp.dx2 = h->d_dx2;
    fp.w_stages = h->as_w_stages;
    fp.w_stage_bytes = h->as_w_stage_bytes;
    fp.has_staging = h->as_staging;
    const int grid = p.m_tiles < h->num_sms ? p.m_tiles : h->num_sms;
    const bool dbg = acc_out != nullptr;
    if (h->fast_div)
        return dbg ? launch_fused_kernel<ptq::ptq_fused_linear_kernel<true, true>>(h, tmY, fp, grid, stream)
                   : launch_fused_kernel<ptq::ptq_fused_linear_kernel<true, false>>(h, tmY, fp, grid, stream);
    return dbg ? launch_fused_kernel<ptq::ptq_fused_linear_kernel<false, true>>(h, tmY, fp, grid, stream)
               : launch_fused_kernel<ptq::ptq_fused_linear_kernel<false, false>>(h, tmY, fp, grid, stream);
}

// The one-kernel path for few rows: taken where its CTAs (128 output channels x `tn` tokens) are all resident at once.
struct SmallPlan {
    int tn, grid, min_ctas;
};

// 16 tokens per CTA while that makes at most one CTA per SM, then 32 (the weights of a CTA are loaded half as often), then
// the same two with two CTAs per SM where shared memory allows.  Beyond that a CTA waits for another to leave and the
// quantization repeated per 128 output channels shows: the two kernels are faster.  us, one kernel against two:
//   rows x K -> N     197 x 384 -> 1536  (156 CTAs, two per SM)  4.2 / 6.8     788 x 768 -> 384  (75 CTAs)   6.3 / 8.0
//                     788 x 192 -> 768   (150, two per SM)       4.2 / 6.6    3152 x 384 -> 192  (198)       6.1 / 7.7
//   not taken:        788 x 384 -> 1536  (300)                   8.4 / 7.4   12608 x 384 -> 44   (394)      11.4 / 9.4
bool plan_small(const ptq_linear *h, long long M, SmallPlan &pl)
{
    if (h->k_blocks > ptq::kSmallMaxKBlocks) return false;
    const long long n_tiles = (h->N + ptq::kSmallRows - 1) / ptq::kSmallRows;
    for (int per_sm = 1; per_sm <= 2; ++per_sm)
        for (int tn = 16; tn <= 32; tn += 16) {
            const long long grid = (M + tn - 1) / tn * n_tiles;
            const int smem = ptq::small_smem_bytes(tn, h->k_blocks, h->K);
            if (grid > static_cast<long long>(per_sm) * h->num_sms || per_sm * (smem + 1024) > ptq::kSmallSmemPerSm ||
                smem > ptq::kSmallSmemLimit)
                continue;
            pl.tn = tn;
            pl.grid = static_cast<int>(grid);
            pl.min_ctas = per_sm;
            return true;
        }
    return false;
}

template <int kMode, int kTN, int kMinCtas>
ptq_status_t launch_small_kernel(const ptq_linear *h, const ptq::SmallParams &p, int grid, cudaStream_t stream)
{
    const ptq_status_t st = ensure_smem<ptq::ptq_small_kernel<kMode, kTN, kMinCtas>>(h->device, ptq::kSmallSmemLimit);
    if (st != PTQ_OK) return st;
    PTQ_CUDA(launch_pdl(ptq::ptq_small_kernel<kMode, kTN, kMinCtas>, grid, ptq::kSmallThreads,
                        ptq::small_smem_bytes(kTN, h->k_blocks, h->K), stream, h->tmWsmall, p));
    g_launches.fetch_add(1, std::memory_order_relaxed);
    PTQ_CUDA(cudaGetLastError());
    return PTQ_OK;
}

ptq_status_t launch_small(const ptq_linear *h, const SmallPlan &pl, const void *x, long long M, void *y, void *acc_out, cudaStream_t stream)
{
    ptq::SmallParams p;
    p.x = static_cast<const __half *>(x);
    p.s = h->d_s;
    p.rs = h->d_rs;
    p.dx2 = h->d_dx2;
    p.zp = h->d_zp;
    p.wsum = h->d_wsum;
    p.dw = h->d_dw;
    p.bias = h->d_bias;
    p.y = static_cast<__half *>(y);
    p.acc_out = static_cast<int32_t *>(acc_out);
    p.status = h->d_status;
    p.M = static_cast<int>(M);
    p.N = h->N;
    p.K = h->K;
    p.T = h->T;
    p.k_blocks = h->k_blocks;
    p.last_mmas = h->last_mmas;
    p.n_tiles = (h->N + ptq::kSmallRows - 1) / ptq::kSmallRows;
    const uintptr_t x_align = reinterpret_cast<uintptr_t>(x) | static_cast<uintptr_t>(2 * h->K);
    p.ld_bytes = x_align % 16 == 0 ? 16 : x_align % 8 == 0 ? 8 : 2;
    p.fast = h->fast_div ? 1 : 0;
    p.fd_T = ptq::make_fastdiv(static_cast<unsigned>(h->T));
    p.fd_cpr = ptq::make_fastdiv(static_cast<unsigned>((h->K + 7) / 8));
    p.fd_n_tiles = ptq::make_fastdiv(static_cast<unsigned>(p.n_tiles));
    auto go = [&](auto mode) {
        constexpr int kMode = decltype(mode)::value;
        if (pl.min_ctas == 1)
            return pl.tn == 16 ? launch_small_kernel<kMode, 16, 1>(h, p, pl.grid, stream)
                               : launch_small_kernel<kMode, 32, 1>(h, p, pl.grid, stream);
        return pl.tn == 16 ? launch_small_kernel<kMode, 16, 2>(h, p, pl.grid, stream)
                           : launch_small_kernel<kMode, 32, 2>(h, p, pl.grid, stream);
    };
    if (h->act_bits == 4) return go(std::integral_constant<int, ptq::kCodeS4>());
    if (h->asym) return go(std::integral_constant<int, ptq::kCodeU8>());
    return go(std::integral_constant<int, ptq::kCodeS8>());
}

// The one-kernel path for layers of a few channels: up to 32, and eight outputs or more per channel, so that the four quantizer
// warps are not what a CTA waits for.  us, two kernels -> one: 3152 x 12 -> 384 5.6 -> 4.9, 25216 x 12 -> 384 10.4 -> 8.2, 12608 x 17 ->
// 200 7.6 -> 6.5, 50432 x 24 -> 768 17.9 -> 17.6, 200704 x 8 -> 64 13.7 -> 13.8; not taken: 200704 x 16 -> 64 14.5 -> 15.6, 200704 x 32 -> 128
// 19.1 -> 22.5, 12608 x 48 -> 1536 13.6 -> 15.9, 50176 x 64 -> 256 11.7 -> 14.0.
// At the range's other end (with a bias, launches replayed from a graph): 12608 x 1 -> 32 5.8 -> 4.1, 201728 x 1 -> 32 14.4 -> 12.6, 50432 x
// 2 -> 32 8.9 -> 5.9, 50432 x 6 -> 64 9.6 -> 6.0, 201728 x 6 -> 64 14.7 -> 13.2, 201728 x 8 -> 64 13.5 -> 12.0.  The nearest to a loss: 6304 x 32 ->
// 256 5.8 -> 6.3, 100864 x 32 -> 768 33.2 -> 33.1.  A thread takes the slower routes of the quantizer for a whole row, so activations
// far from the calibrated steps (every thirtieth code saturated or near a tie) cost this kernel more: 25216 x 24 -> 768 12.0 -> 13.8.
bool plan_short_k(const ptq_linear *h, const void *y)
{
    return h->K <= ptq::kShortKMaxK && h->N >= 8 * h->K && !h->asym && h->fast_div && h->N % 8 == 0 &&
           reinterpret_cast<uintptr_t>(y) % 16 == 0;
}

ptq_status_t launch_short_k(const ptq_linear *h, const void *x, long long M, void *y, void *acc_out, cudaStream_t stream)
{
    CUtensorMap tmY;
    ptq_status_t st = cached_map_2d(h->y_maps, &tmY, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, y, static_cast<unsigned long long>(h->N),
                                    static_cast<unsigned long long>(M), static_cast<unsigned long long>(h->N) * 2, ptq::kStreamBoxCols, 32);
    if (st != PTQ_OK) return st;
    ptq::ShortKParams sp;
    ptq::UnitParams &p = sp.g;
    set_gemm_params(h, p, M, y, acc_out, true, nullptr);
    p.group = ptq::short_k_group(p.m_tiles, p.n_tiles, h->num_sms);
    p.groups = (p.n_tiles + p.group - 1) / p.group;
    sp.x = static_cast<const __half *>(x);
    sp.s = h->d_s;
    sp.rs = h->d_rs;
    sp.dx2 = h->d_dx2;
    const uintptr_t x_align = reinterpret_cast<uintptr_t>(x) | static_cast<uintptr_t>(2 * h->K);
    sp.ld_bytes = x_align % 16 == 0 ? 16 : x_align % 8 == 0 ? 8 : 2;
    const long long units = static_cast<long long>(p.m_tiles) * p.groups;
    const int grid = static_cast<int>(units < h->num_sms ? units : h->num_sms);
    ptq::set_units(p, grid);
    const int smem = ptq::short_k_smem_bytes(p.group * p.BN * ptq::kBK, p.vectors);
    auto go = [&](auto chunks, auto mode, auto debug) -> ptq_status_t {
        constexpr auto kKern = ptq::ptq_short_k_kernel<decltype(chunks)::value, decltype(mode)::value, decltype(debug)::value>;
        const ptq_status_t es = ensure_smem<kKern>(h->device, ptq::kShortKSmemMax);
        if (es != PTQ_OK) return es;
        PTQ_CUDA(launch_pdl(kKern, grid, ptq::kShortKThreads, smem, stream, h->tmW, tmY, sp));
        return PTQ_OK;
    };
    auto mode = [&](auto chunks) {
        const std::integral_constant<int, ptq::kCodeS4> s4;
        const std::integral_constant<int, ptq::kCodeS8> s8;
        return h->act_bits == 4 ? (acc_out ? go(chunks, s4, std::true_type()) : go(chunks, s4, std::false_type()))
                                : (acc_out ? go(chunks, s8, std::true_type()) : go(chunks, s8, std::false_type()));
    };
    st = h->K <= 16 ? mode(std::integral_constant<int, 2>()) : mode(std::integral_constant<int, 4>());
    if (st != PTQ_OK) return st;
    g_launches.fetch_add(1, std::memory_order_relaxed);
    PTQ_CUDA(cudaGetLastError());
    return PTQ_OK;
}

bool fused_usable(const ptq_linear *h) { return h->as_ok && h->K % 16 == 0; }

// Scratch for ptq_linear_forward_static: lives in the library image on every device that loads it.
// In host code the symbol below is only a stand-in; the kernels must be given the device address
// that cudaGetSymbolAddress returns, looked up once per device with that device current.
static __device__ __align__(256) unsigned char g_static_scratch[PTQ_STATIC_SCRATCH_BYTES];

ptq_status_t static_scratch_address(int device, void **out)
{
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static void *addr[kMaxDevices] = {};
    if (device < 0 || device >= kMaxDevices) return fail(PTQ_ERR_CUDA, "device index %d out of range", device);
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[device]) {
        void *p = nullptr;
        PTQ_CUDA(cudaGetSymbolAddress(&p, g_static_scratch));   // the current device is `device` (checked by the caller)
        if (!p) return fail(PTQ_ERR_CUDA, "cudaGetSymbolAddress returned a null address");
        addr[device] = p;
    }
    *out = addr[device];
    return PTQ_OK;
}

ptq_status_t validate_forward(const ptq_linear *h, const void *x, int B, const void *y)
{
    if (!h || !x || !y) return fail(PTQ_ERR_NULL, "handle, x and y must not be NULL");
    if (B < 1) return fail(PTQ_ERR_SHAPE, "B must be >= 1 (got %d)", B);
    const long long M = static_cast<long long>(B) * h->T;
    if (M > 0x7fffff00ll) return fail(PTQ_ERR_SHAPE, "B*T = %lld is too large", M);
    if (reinterpret_cast<uintptr_t>(x) % 2 || reinterpret_cast<uintptr_t>(y) % 2)
        return fail(PTQ_ERR_ALIGN, "x and y must be 2-byte aligned");
    if (ranges_overlap(x, static_cast<size_t>(M) * h->K * 2, y, static_cast<size_t>(M) * h->N * 2))
        return fail(PTQ_ERR_VALUE, "x and y overlap");
    return check_device(h);
}

}  // namespace

extern "C" {

const char *ptq_status_string(ptq_status_t st)
{
    switch (st) {
        case PTQ_OK: return "PTQ_OK";
        case PTQ_ERR_NULL: return "PTQ_ERR_NULL";
        case PTQ_ERR_SHAPE: return "PTQ_ERR_SHAPE";
        case PTQ_ERR_VALUE: return "PTQ_ERR_VALUE";
        case PTQ_ERR_ALIGN: return "PTQ_ERR_ALIGN";
        case PTQ_ERR_ARCH: return "PTQ_ERR_ARCH";
        case PTQ_ERR_CUDA: return "PTQ_ERR_CUDA";
        case PTQ_ERR_NOMEM: return "PTQ_ERR_NOMEM";
        case PTQ_ERR_TIMEOUT: return "PTQ_ERR_TIMEOUT";
    }
    return "PTQ_ERR_UNKNOWN";
}

const char *ptq_last_error(void) { return g_err; }

unsigned long long ptq_kernel_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

void ptq_linear_destroy(ptq_linear_t *h)
{
    if (!h) return;
    cudaFree(h->d_all);
    delete h;
}

static ptq_status_t create_impl(ptq_linear_t **out, int K, int N, int T, const int8_t *w_q, const float *w_step,
                                const float *smooth, const float *act_step, const int32_t *act_zero,
                                const float *bias, unsigned flags, int act_bits = 8)
{
    if (!out) return fail(PTQ_ERR_NULL, "out must not be NULL");
    *out = nullptr;
    if (!w_q || !w_step || !smooth || !act_step)
        return fail(PTQ_ERR_NULL, "w_q, w_step, smooth and act_step must not be NULL");
    if (K < 1 || K > PTQ_MAX_K || N < 1 || N > PTQ_MAX_N || T < 1 || T > PTQ_MAX_T)
        return fail(PTQ_ERR_SHAPE, "K, N, T out of range (K=%d N=%d T=%d)", K, N, T);
    if (flags != PTQ_FLAG_NONE) return fail(PTQ_ERR_VALUE, "flags must be PTQ_FLAG_NONE at create");

    // Parameter values (host-only checks come first so that they are testable without a device).
    const float lo = std::ldexp(1.0f, -30), hi = std::ldexp(1.0f, 30);
    bool fast = true;
    for (int k = 0; k < K; ++k) {
        if (!(smooth[k] > 0.0f) || !std::isfinite(smooth[k]))
            return fail(PTQ_ERR_VALUE, "smooth[%d] = %g must be finite and > 0", k, smooth[k]);
        if (smooth[k] < lo || smooth[k] > hi) fast = false;
    }
    for (int t = 0; t < T; ++t) {
        if (!(act_step[t] > 0.0f) || !std::isfinite(act_step[t]))
            return fail(PTQ_ERR_VALUE, "act_step[%d] = %g must be finite and > 0", t, act_step[t]);
        if (act_step[t] < lo || act_step[t] > hi) fast = false;
    }
    for (int n = 0; n < N; ++n) {
        if (!(w_step[n] > 0.0f) || !std::isfinite(w_step[n]))
            return fail(PTQ_ERR_VALUE, "w_step[%d] = %g must be finite and > 0", n, w_step[n]);
        if (bias && !std::isfinite(bias[n])) return fail(PTQ_ERR_VALUE, "bias[%d] is not finite", n);
    }
    for (int t = 0; act_zero && t < T; ++t)
        if (act_zero[t] < 0 || act_zero[t] > 255)
            return fail(PTQ_ERR_VALUE, "act_zero[%d] = %d is outside [0,255]", t, act_zero[t]);
    if (const void *bad = std::memchr(w_q, 0x80, static_cast<size_t>(N) * K))
        return fail(PTQ_ERR_VALUE, "w_q[%lld] = -128 is outside the symmetric range [-127,127]",
                    static_cast<long long>(static_cast<const int8_t *>(bad) - w_q));

    int dev = -1, major = 0, minor = 0, sms = 0, l2 = 0;
    PTQ_CUDA(cudaGetDevice(&dev));
    PTQ_CUDA(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev));
    PTQ_CUDA(cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev));
    PTQ_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    PTQ_CUDA(cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev));
    if (major != 10 || minor != 0)
        return fail(PTQ_ERR_ARCH, "device %d is compute capability %d.%d; this library needs 10.0 (sm_100a)", dev, major, minor);

    std::unique_ptr<ptq_linear, decltype(&ptq_linear_destroy)> owner(new ptq_linear(), ptq_linear_destroy);
    ptq_linear *h = owner.get();
    h->K = K;
    h->N = N;
    h->T = T;
    h->Kpad = round_up(K, 16);
    // Whole 128-byte lines per weight row: a TMA box is one 128-byte k-block of up to 256 rows, loaded by every CTA for every
    // tile, and a row that straddles two lines is two requests to L2 (and the 16-byte rows of a narrow layer send all
    // CTAs to a handful of lines).  Layers, both kernels: 200704 x 96 -> 384 51.3 -> 43.8 us, 200704 x 192 -> 96 36.5 -> 32.6,
    // 12608 x 12 -> 384 9.9 -> 8.6, 3940 x 1455 -> 784 18.9 -> 17.2.  The codes keep 16-byte rounding: whole lines there cost
    // more footprint than they save requests (200704 x 192 -> 96 32.6 -> 35.0).
    h->w_pitch = round_up(K, 128);
    h->device = dev;
    h->num_sms = sms;
    h->l2_bytes = l2;
    h->fast_div = fast;
    h->n_tiles = (N + ptq::kMaxBN - 1) / ptq::kMaxBN;
    if (h->n_tiles == 1)
        h->BN = round_up(N, 16);
    else
        h->BN = round_up((N + h->n_tiles - 1) / h->n_tiles, 64);
    h->k_blocks = (K + ptq::kBK - 1) / ptq::kBK;
    h->last_mmas = (K - (h->k_blocks - 1) * ptq::kBK + 31) / 32;

    h->asym = act_zero != nullptr;
    h->has_bias = bias != nullptr;
    h->act_bits = act_bits;
    choose_astat(h);
    if (h->asym || act_bits != 8) h->as_ok = false;   // these layers run the quantize kernel + single-CTA GEMM kernel only
    int Npad = h->n_tiles * h->BN;
    if (h->as_ok && h->as_n_tiles * h->as_BN > Npad) Npad = h->as_n_tiles * h->as_BN;
    const int Nvec = round_up(Npad, 64) + 256;      // the last tile of any width reads at most 255 beyond N, a step 64
    const int Kvec = round_up(K, 16);
    // One host image of all parameters, one allocation and one copy: a device allocation costs more than the copy does.
    size_t total = 0;
    auto place = [&](size_t bytes) {
        const size_t at = total;
        total += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t o_w = place(static_cast<size_t>(Npad) * h->w_pitch), o_dw = place(sizeof(float) * Nvec),
                 o_bias = place(sizeof(float) * Nvec), o_s = place(sizeof(float) * Kvec), o_rs = place(sizeof(float) * Kvec),
                 o_dx = place(sizeof(float) * T), o_dx2 = place(sizeof(float2) * T),
                 o_zp = place(h->asym ? sizeof(int) * T : 0), o_wsum = place(h->asym ? sizeof(int) * Nvec : 0),
                 o_status = place(sizeof(unsigned));
    std::vector<unsigned char> image(total, 0);
    int8_t *wpad = reinterpret_cast<int8_t *>(&image[o_w]);
    for (int n = 0; n < N; ++n) std::memcpy(wpad + static_cast<size_t>(n) * h->w_pitch, w_q + static_cast<size_t>(n) * K, K);
    std::memcpy(&image[o_dw], w_step, sizeof(float) * N);
    if (bias) std::memcpy(&image[o_bias], bias, sizeof(float) * N);
    float *sp = reinterpret_cast<float *>(&image[o_s]), *rs = reinterpret_cast<float *>(&image[o_rs]);
    for (int k = 0; k < Kvec; ++k) {
        sp[k] = k < K ? smooth[k] : 1.0f;
        rs[k] = 1.0f / sp[k];
    }
    std::memcpy(&image[o_dx], act_step, sizeof(float) * T);
    float *dx2 = reinterpret_cast<float *>(&image[o_dx2]);
    for (int t = 0; t < T; ++t) {
        dx2[2 * t] = act_step[t];
        dx2[2 * t + 1] = 1.0f / act_step[t];
    }
    if (h->asym) {
        std::memcpy(&image[o_zp], act_zero, sizeof(int) * T);
        int *wsum = reinterpret_cast<int *>(&image[o_wsum]);
        for (int n = 0; n < N; ++n) {
            int acc = 0;
            for (int k = 0; k < K; ++k) acc += w_q[static_cast<size_t>(n) * K + k];
            wsum[n] = acc;
        }
    }

    ptq_status_t st = PTQ_OK;
    auto move_in = [&]() -> ptq_status_t {
        PTQ_CUDA(cudaMalloc(reinterpret_cast<void **>(&h->d_all), total));
        PTQ_CUDA(cudaMemcpy(h->d_all, image.data(), total, cudaMemcpyHostToDevice));
        // A copy from pageable memory returns once the last part is staged, and streams that do not synchronise with the
        // default stream, on which a forward call may follow at once, are not ordered behind it.
        PTQ_CUDA(cudaStreamSynchronize(cudaStreamLegacy));
        return PTQ_OK;
    };
    do {
        if ((st = move_in()) != PTQ_OK) break;
        h->d_w = reinterpret_cast<int8_t *>(h->d_all + o_w);
        h->d_dw = reinterpret_cast<float *>(h->d_all + o_dw);
        h->d_bias = reinterpret_cast<float *>(h->d_all + o_bias);
        h->d_s = reinterpret_cast<float *>(h->d_all + o_s);
        h->d_rs = reinterpret_cast<float *>(h->d_all + o_rs);
        h->d_dx = reinterpret_cast<float *>(h->d_all + o_dx);
        h->d_dx2 = reinterpret_cast<float2 *>(h->d_all + o_dx2);
        if (h->asym) {
            h->d_zp = reinterpret_cast<int *>(h->d_all + o_zp);
            h->d_wsum = reinterpret_cast<int *>(h->d_all + o_wsum);
        }
        h->d_status = reinterpret_cast<unsigned *>(h->d_all + o_status);
        // The maps' rows are whole sectors of the padded lines, not K bytes: where a box reaches beyond its map's rows, TMA fills about 4 cycles a
        // row slower (8 where rows end inside a sector), and a resident group of N tiles loads up to 768 rows before its first MMA.
        // Both kernels, us, rows of K bytes / lines: 13184 x 40 -> 512 9.8 / 7.8, 14720 x 80 -> 528 11.8 / 8.6, 31744 x 48 -> 736 17.0 / 14.3,
        // 29056 x 80 -> 512 13.5 / 11.9; K = 64 and 96 0 to 2 %, K = 128 the same.
        // One sector is enough for K <= 32: a quarter of the bytes, whole sectors all the same.  Lines / sectors: 37632 x 21 -> 3060 73.5 / 72.3,
        // 97216 x 26 -> 2786 169.7 / 167.2, 1182 x 29 -> 180 4.0 / 3.4; 50 layers with 8 <= K <= 32 the same on average.
        const int w_row = K <= 32 ? 32 : h->w_pitch;
        auto weights_map = [&](CUtensorMap *map, int box_rows) {
            return make_map_2d(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, h->d_w, static_cast<unsigned long long>(w_row),
                               static_cast<unsigned long long>(Npad), static_cast<unsigned long long>(h->w_pitch), ptq::kBK,
                               static_cast<unsigned>(box_rows));
        };
        st = weights_map(&h->tmW, h->BN);
        if (st != PTQ_OK) break;
        st = weights_map(&h->tmWh, h->BN / 2);
        if (st != PTQ_OK) break;
        h->max_pairs = h->asym ? 0 : query_max_pairs(dev);
        if (h->as_ok)
            st = weights_map(&h->tmWas, h->as_BN);
        else
            h->tmWas = h->tmW;
        if (st != PTQ_OK) break;
        st = weights_map(&h->tmWsmall, ptq::kSmallRows);
        for (int i = 0; i < 4 && st == PTQ_OK; ++i) st = weights_map(&h->tmWbn[i], 64 * (i + 1));
    } while (0);
    if (st != PTQ_OK) return st;
    *out = owner.release();
    return PTQ_OK;
}

ptq_status_t ptq_linear_create(ptq_linear_t **out, int K, int N, int T, const int8_t *w_q, const float *w_step,
                               const float *smooth, const float *act_step, const float *bias, unsigned flags)
{
    return no_throw([&] { return create_impl(out, K, N, T, w_q, w_step, smooth, act_step, nullptr, bias, flags); });
}

ptq_status_t ptq_linear_create_asym(ptq_linear_t **out, int K, int N, int T, const int8_t *w_q, const float *w_step,
                                    const float *smooth, const float *act_step, const int32_t *act_zero,
                                    const float *bias, unsigned flags)
{
    if (out) *out = nullptr;
    if (!act_zero) return fail(PTQ_ERR_NULL, "act_zero must not be NULL");
    return no_throw([&] { return create_impl(out, K, N, T, w_q, w_step, smooth, act_step, act_zero, bias, flags); });
}

size_t ptq_linear_workspace_bytes(const ptq_linear_t *h, int B, unsigned flags)
{
    if (!h || B < 1) return 0;
    if ((flags & PTQ_FLAG_FUSED_PROLOGUE) && ptq_linear_fused_supported(h)) return 0;
    return static_cast<size_t>(B) * h->T * h->Kpad;
}

int ptq_linear_fused_supported(const ptq_linear_t *h) { return (h && fused_usable(h)) ? 1 : 0; }

ptq_status_t ptq_quantize(const ptq_linear_t *h, const void *x_fp16, int B, void *q_int8, void *stream)
{
    if (!h || !x_fp16 || !q_int8) return fail(PTQ_ERR_NULL, "handle, x and q must not be NULL");
    if (B < 1) return fail(PTQ_ERR_SHAPE, "B must be >= 1 (got %d)", B);
    if (reinterpret_cast<uintptr_t>(x_fp16) % 2) return fail(PTQ_ERR_ALIGN, "x must be 2-byte aligned");
    ptq_status_t st = check_device(h);
    if (st != PTQ_OK) return st;
    const long long M = static_cast<long long>(B) * h->T;
    if (ranges_overlap(x_fp16, static_cast<size_t>(M) * h->K * 2, q_int8, static_cast<size_t>(M) * h->K))
        return fail(PTQ_ERR_VALUE, "x and q overlap");
    return launch_quantize(h, x_fp16, M, q_int8, h->K, static_cast<cudaStream_t>(stream));
}

int ptq_linear_describe(const ptq_linear_t *h, char *buf, int buf_bytes)
{
    if (!h) return 0;
    char tmp[512];
    const int n = snprintf(tmp, sizeof(tmp),
                           "K=%d N=%d T=%d Kpad=%d%s | quantize: %s | gemm: BN=%d n_tiles=%d k_blocks=%d "
                           "pair_clusters=%d | fused: %s BN=%d n_tiles=%d w_stages=%d staging=%d smem=%d",
                           h->K, h->N, h->T, h->Kpad, h->asym ? " asymmetric" : (h->act_bits == 4 ? " w4a4" : ""),
                           h->fast_div ? "screened reciprocal route" : "IEEE division",
                           h->BN, h->n_tiles, h->k_blocks, h->max_pairs,
                           (h->as_ok && h->K % 16 == 0) ? "yes" : "no", h->as_BN, h->as_n_tiles, h->as_w_stages,
                           h->as_staging, h->as_smem);
    if (buf && buf_bytes > 0) {
        strncpy(buf, tmp, static_cast<size_t>(buf_bytes) - 1);
        buf[buf_bytes - 1] = 0;
    }
    return n;
}

int ptq_linear_code_pitch(const ptq_linear_t *h) { return h ? h->Kpad : 0; }

int ptq_linear_gemm_variant(const ptq_linear_t *h, int B) { return ptq_linear_gemm_tiling(h, B, nullptr, nullptr); }

int ptq_linear_gemm_tiling(const ptq_linear_t *h, int B, int *tile_cols, int *piece_cols)
{
    if (tile_cols) *tile_cols = 0;
    if (piece_cols) *piece_cols = 0;
    if (!h || B < 1) return -1;
    const long long M = static_cast<long long>(B) * h->T;
    const bool tma_store = h->N % 8 == 0;
    ptq::GemmParams p = {};
    set_gemm_params(h, p, M, nullptr, nullptr, tma_store, nullptr);
    if (plan_panel(h, p, tma_store)) {
        if (tile_cols) *tile_cols = h->BN;
        return 2;
    }
    const Tiling t = choose_tiling(h, p, tma_store);
    if (tile_cols) *tile_cols = t.bn;
    if (piece_cols) *piece_cols = t.cut;
    return t.resident ? 1 : 0;
}

ptq_status_t ptq_linear_gemm_dequant(const ptq_linear_t *h, const void *q_int8, int B, void *y_fp16, void *stream)
{
    if (!h || !q_int8 || !y_fp16) return fail(PTQ_ERR_NULL, "handle, q and y must not be NULL");
    if (B < 1) return fail(PTQ_ERR_SHAPE, "B must be >= 1 (got %d)", B);
    if (reinterpret_cast<uintptr_t>(q_int8) % 16) return fail(PTQ_ERR_ALIGN, "q must be 16-byte aligned");
    if (reinterpret_cast<uintptr_t>(y_fp16) % 2) return fail(PTQ_ERR_ALIGN, "y must be 2-byte aligned");
    ptq_status_t st = check_device(h);
    if (st != PTQ_OK) return st;
    const long long M = static_cast<long long>(B) * h->T;
    if (ranges_overlap(q_int8, static_cast<size_t>(M) * h->Kpad, y_fp16, static_cast<size_t>(M) * h->N * 2))
        return fail(PTQ_ERR_VALUE, "q and y overlap");
    return launch_gemm(h, q_int8, M, y_fp16, nullptr, static_cast<cudaStream_t>(stream));
}

ptq_status_t ptq_linear_forward_debug(const ptq_linear_t *h, const void *x_fp16, int B, void *y_fp16,
                                      void *q_int8_out, void *acc_int32_out, void *workspace,
                                      size_t workspace_bytes, unsigned flags, void *stream)
{
    ptq_status_t st = validate_forward(h, x_fp16, B, y_fp16);
    if (st != PTQ_OK) return st;
    if (flags & ~(PTQ_FLAG_FUSED_PROLOGUE | PTQ_FLAG_CTA_PAIR)) return fail(PTQ_ERR_VALUE, "unknown flags 0x%x", flags);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const long long M = static_cast<long long>(B) * h->T;
    if ((flags & PTQ_FLAG_FUSED_PROLOGUE) && fused_usable(h) && reinterpret_cast<uintptr_t>(x_fp16) % 16 == 0) {
        // F1: one kernel, no workspace.  The codes never exist in memory; a requested tap is produced by
        // the quantize kernel on its own.
        if ((st = launch_fused(h, x_fp16, M, y_fp16, acc_int32_out, s)) != PTQ_OK) return st;
        if (q_int8_out) return launch_quantize(h, x_fp16, M, q_int8_out, h->K, s);
        return PTQ_OK;
    }
    const size_t need = static_cast<size_t>(M) * h->Kpad;
    if (!workspace) return fail(PTQ_ERR_NULL, "workspace must not be NULL for this layer, alignment and flags");
    if (workspace_bytes < need)
        return fail(PTQ_ERR_SHAPE, "workspace has %zu bytes, %zu needed", workspace_bytes, need);
    if (reinterpret_cast<uintptr_t>(workspace) % 16) return fail(PTQ_ERR_ALIGN, "workspace must be 16-byte aligned");
    if (ranges_overlap(workspace, need, y_fp16, static_cast<size_t>(M) * h->N * 2) ||
        ranges_overlap(workspace, need, x_fp16, static_cast<size_t>(M) * h->K * 2))
        return fail(PTQ_ERR_VALUE, "workspace overlaps x or y");
    SmallPlan pl;
    if (!(flags & PTQ_FLAG_CTA_PAIR) && plan_small(h, M, pl)) {
        // one kernel; the codes never exist in memory: a requested tap is produced by the quantize kernel on its own
        if ((st = launch_small(h, pl, x_fp16, M, y_fp16, acc_int32_out, s)) != PTQ_OK) return st;
        if (q_int8_out) return launch_quantize(h, x_fp16, M, q_int8_out, h->K, s);
        return PTQ_OK;
    }
    if (!(flags & PTQ_FLAG_CTA_PAIR) && plan_short_k(h, y_fp16)) {
        if ((st = launch_short_k(h, x_fp16, M, y_fp16, acc_int32_out, s)) != PTQ_OK) return st;
        if (q_int8_out) return launch_quantize(h, x_fp16, M, q_int8_out, h->K, s);
        return PTQ_OK;
    }
    if ((st = launch_quantize(h, x_fp16, M, workspace, h->Kpad, s)) != PTQ_OK) return st;
    if ((st = launch_gemm(h, workspace, M, y_fp16, acc_int32_out, s, (flags & PTQ_FLAG_CTA_PAIR) != 0)) != PTQ_OK)
        return st;
    if (q_int8_out)
        PTQ_CUDA(cudaMemcpy2DAsync(q_int8_out, h->K, workspace, h->Kpad, h->K, static_cast<size_t>(M),
                                   cudaMemcpyDeviceToDevice, s));
    return PTQ_OK;
}

ptq_status_t ptq_linear_forward(const ptq_linear_t *h, const void *x_fp16, int B, void *y_fp16, void *workspace,
                                size_t workspace_bytes, unsigned flags, void *stream)
{
    return ptq_linear_forward_debug(h, x_fp16, B, y_fp16, nullptr, nullptr, workspace, workspace_bytes, flags, stream);
}

ptq_status_t ptq_linear_forward_static(const ptq_linear_t *h, const void *x_fp16, int B, void *y_fp16,
                                       void *stream)
{
    ptq_status_t st = validate_forward(h, x_fp16, B, y_fp16);
    if (st != PTQ_OK) return st;
    const long long M = static_cast<long long>(B) * h->T;
    const unsigned long long need = static_cast<unsigned long long>(M) * h->Kpad;
    if (need > PTQ_STATIC_SCRATCH_BYTES)
        return fail(PTQ_ERR_SHAPE,
                    "B*T*pitch = %llu bytes of codes exceed the built-in scratch of %u bytes; "
                    "split the batch or use ptq_linear_forward with a caller workspace",
                    need, PTQ_STATIC_SCRATCH_BYTES);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    SmallPlan pl;
    if (plan_small(h, M, pl)) return launch_small(h, pl, x_fp16, M, y_fp16, nullptr, s);
    if (plan_short_k(h, y_fp16)) return launch_short_k(h, x_fp16, M, y_fp16, nullptr, s);
    void *scratch = nullptr;
    if ((st = static_scratch_address(h->device, &scratch)) != PTQ_OK) return st;
    if ((st = launch_quantize(h, x_fp16, M, scratch, h->Kpad, s)) != PTQ_OK) return st;
    return launch_gemm(h, scratch, M, y_fp16, nullptr, s);
}

// Device workspace of the step search: [K] s, [T] base, then [T] dx, [T] best, then the losses [T, C].
struct SearchLayout {
    size_t in, out, loss, total;
};
static SearchLayout search_layout(int K, int T, int C)
{
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    SearchLayout l;
    l.in = 0;
    l.out = up(sizeof(float) * (static_cast<size_t>(K) + static_cast<size_t>(T)));
    l.loss = l.out + up(2 * sizeof(float) * static_cast<size_t>(T));
    l.total = l.loss + up(sizeof(double) * static_cast<size_t>(T) * C);
    return l;
}

size_t ptq_search_workspace_bytes(int K, int T, int n_grid, int j_lo)
{
    if (K < 1 || K > PTQ_MAX_K || T < 1 || T > PTQ_MAX_T || n_grid < 1 || n_grid > PTQ_MAX_SEARCH_GRID || j_lo < 1 || j_lo > n_grid)
        return 0;
    return search_layout(K, T, n_grid - j_lo + 1).total;
}

static ptq_status_t search_check(int K, int T, const void *xcal_fp16, int Bc, const float *smooth, const float *base_step,
                                 int n_grid, int j_lo, const float *act_step_out)
{
    if (!xcal_fp16 || !smooth || !base_step || !act_step_out)
        return fail(PTQ_ERR_NULL, "search: pointers must not be NULL");
    if (K < 1 || K > PTQ_MAX_K || T < 1 || T > PTQ_MAX_T || Bc < 1 ||
        static_cast<long long>(Bc) * K > 0x7fffffffll)
        return fail(PTQ_ERR_SHAPE, "search: dimensions out of range (K=%d T=%d Bc=%d)", K, T, Bc);
    if (n_grid < 1 || n_grid > PTQ_MAX_SEARCH_GRID || j_lo < 1 || j_lo > n_grid)
        return fail(PTQ_ERR_VALUE, "search: need 1 <= j_lo <= n_grid <= %d (got j_lo=%d n_grid=%d)",
                    PTQ_MAX_SEARCH_GRID, j_lo, n_grid);
    if (reinterpret_cast<uintptr_t>(xcal_fp16) % 2) return fail(PTQ_ERR_ALIGN, "xcal must be 2-byte aligned");
    for (int k = 0; k < K; ++k)
        if (!(smooth[k] > 0.0f) || !std::isfinite(smooth[k]))
            return fail(PTQ_ERR_VALUE, "search: smooth[%d] = %g is not positive and finite", k, smooth[k]);
    for (int t = 0; t < T; ++t)
        if (!(base_step[t] >= 1e-30f) || !std::isfinite(base_step[t]))
            return fail(PTQ_ERR_VALUE, "search: base_step[%d] = %g is not in [1e-30, inf)", t, base_step[t]);
    return PTQ_OK;
}

static ptq_status_t search_impl(int K, int T, const void *xcal_fp16, int Bc, const float *smooth, const float *base_step,
                                int n_grid, int j_lo, float *act_step_out, int32_t *best_out, double *loss_out, void *workspace,
                                size_t workspace_bytes, void *stream)
{
    const ptq_status_t st = search_check(K, T, xcal_fp16, Bc, smooth, base_step, n_grid, j_lo, act_step_out);
    if (st != PTQ_OK) return st;
    const int C = n_grid - j_lo + 1;
    const SearchLayout l = search_layout(K, T, C);
    if (!workspace) return fail(PTQ_ERR_NULL, "search: workspace must not be NULL");
    if (workspace_bytes < l.total)
        return fail(PTQ_ERR_SHAPE, "search: workspace has %zu bytes, %zu needed", workspace_bytes, l.total);
    if (reinterpret_cast<uintptr_t>(workspace) % 256) return fail(PTQ_ERR_ALIGN, "search: workspace must be 256-byte aligned");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned char *base = static_cast<unsigned char *>(workspace);
    float *d_s = reinterpret_cast<float *>(base + l.in), *d_base = d_s + K;
    float *d_dx = reinterpret_cast<float *>(base + l.out);
    int *d_best = reinterpret_cast<int *>(d_dx + T);
    double *d_loss = reinterpret_cast<double *>(base + l.loss);
    std::vector<float> in(static_cast<size_t>(K) + T), out(2 * static_cast<size_t>(T));   // one copy each way
    std::memcpy(in.data(), smooth, sizeof(float) * K);
    std::memcpy(in.data() + K, base_step, sizeof(float) * T);
    int dev = -1, sms = 0;
    PTQ_CUDA(cudaGetDevice(&dev));
    PTQ_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    PTQ_CUDA(cudaMemcpyAsync(d_s, in.data(), sizeof(float) * in.size(), cudaMemcpyHostToDevice, s));
    ptq::SearchParams p;
    p.x = static_cast<const __half *>(xcal_fp16);
    p.s = d_s;
    p.base = d_base;
    p.loss = d_loss;
    p.Bc = Bc;
    p.T = T;
    p.K = K;
    p.n_grid = n_grid;
    p.j_lo = j_lo;
    p.fd_K = ptq::make_fastdiv(static_cast<unsigned>(K));
    const ptq::SearchPlan plan = ptq::search_plan(Bc * K, T, C, sms);
    // Not for positions of fewer elements than two per thread: a few threads would divide eight in turn (11 x 197 x 8, 3 candidates, a call 38.4
    // us one at a time, 40.3 eight at a time; 6 x 196 x 8, 28 candidates 40.2 / 42.3).
    p.vec = K % 8 == 0 && reinterpret_cast<uintptr_t>(xcal_fp16) % 16 == 0 && Bc * K >= 2 * plan.block();
    const dim3 grid(static_cast<unsigned>(T), static_cast<unsigned>((C + plan.candidates - 1) / plan.candidates));
    if (plan.candidates == ptq::kSearchMany)
        ptq::ptq_search_loss_kernel<ptq::kSearchGroups><<<grid, plan.block(), 0, s>>>(p);
    else
        ptq::ptq_search_loss_kernel<1><<<grid, plan.block(), 0, s>>>(p);
    ptq::ptq_search_pick_kernel<<<(T + 3) / 4, 128, 0, s>>>(d_loss, d_base, T, n_grid, j_lo, d_best, d_dx);
    g_launches.fetch_add(2, std::memory_order_relaxed);
    PTQ_CUDA(cudaGetLastError());
    PTQ_CUDA(cudaMemcpyAsync(out.data(), d_dx, sizeof(float) * out.size(), cudaMemcpyDeviceToHost, s));
    if (loss_out)
        PTQ_CUDA(cudaMemcpyAsync(loss_out, d_loss, sizeof(double) * static_cast<size_t>(T) * C, cudaMemcpyDeviceToHost, s));
    PTQ_CUDA(cudaStreamSynchronize(s));
    std::memcpy(act_step_out, out.data(), sizeof(float) * T);
    if (best_out) std::memcpy(best_out, out.data() + T, sizeof(int32_t) * T);
    return PTQ_OK;
}

ptq_status_t ptq_search_act_step_in(int K, int T, const void *xcal_fp16, int Bc, const float *smooth,
                                    const float *base_step, int n_grid, int j_lo, float *act_step_out,
                                    int32_t *best_out, double *loss_out, void *workspace, size_t workspace_bytes,
                                    void *stream)
{
    return no_throw([&] {
        return search_impl(K, T, xcal_fp16, Bc, smooth, base_step, n_grid, j_lo, act_step_out, best_out, loss_out, workspace,
                           workspace_bytes, stream);
    });
}

ptq_status_t ptq_search_act_step(int K, int T, const void *xcal_fp16, int Bc, const float *smooth,
                                 const float *base_step, int n_grid, int j_lo, float *act_step_out,
                                 int32_t *best_out, double *loss_out, void *stream)
{
    ptq_status_t st = search_check(K, T, xcal_fp16, Bc, smooth, base_step, n_grid, j_lo, act_step_out);
    if (st != PTQ_OK) return st;
    const size_t bytes = ptq_search_workspace_bytes(K, T, n_grid, j_lo);
    void *ws = nullptr;
    PTQ_CUDA(cudaMalloc(&ws, bytes));
    st = ptq_search_act_step_in(K, T, xcal_fp16, Bc, smooth, base_step, n_grid, j_lo, act_step_out, best_out, loss_out, ws,
                                bytes, stream);
    cudaFree(ws);
    return st;
}

static size_t dynamic_codes_bytes(const ptq_linear *h, long long M)
{
    return (static_cast<size_t>(M) * h->Kpad + 255) / 256 * 256;
}

size_t ptq_linear_workspace_bytes_dynamic(const ptq_linear_t *h, int B)
{
    if (!h || B < 1) return 0;
    const long long M = static_cast<long long>(B) * h->T;
    return dynamic_codes_bytes(h, M) + static_cast<size_t>(M) * sizeof(float);
}

ptq_status_t ptq_linear_forward_dynamic_debug(const ptq_linear_t *h, const void *x_fp16, int B, void *y_fp16,
                                              void *q_int8_out, void *acc_int32_out, void *step_fp32_out,
                                              void *workspace, size_t workspace_bytes, void *stream)
{
    ptq_status_t st = validate_forward(h, x_fp16, B, y_fp16);
    if (st != PTQ_OK) return st;
    if (h->asym || h->act_bits != 8)
        return fail(PTQ_ERR_VALUE, "the dynamic comparator is defined for symmetric 8-bit layers only");
    const long long M = static_cast<long long>(B) * h->T;
    const size_t codes = dynamic_codes_bytes(h, M);
    const size_t need = codes + static_cast<size_t>(M) * sizeof(float);
    if (!workspace) return fail(PTQ_ERR_NULL, "workspace must not be NULL");
    if (workspace_bytes < need)
        return fail(PTQ_ERR_SHAPE, "workspace has %zu bytes, %zu needed", workspace_bytes, need);
    if (reinterpret_cast<uintptr_t>(workspace) % 16) return fail(PTQ_ERR_ALIGN, "workspace must be 16-byte aligned");
    if (ranges_overlap(workspace, need, y_fp16, static_cast<size_t>(M) * h->N * 2) ||
        ranges_overlap(workspace, need, x_fp16, static_cast<size_t>(M) * h->K * 2))
        return fail(PTQ_ERR_VALUE, "workspace overlaps x or y");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    float *dx_row = reinterpret_cast<float *>(static_cast<unsigned char *>(workspace) + codes);
    if ((st = launch_quantize_dynamic(h, x_fp16, M, workspace, h->Kpad, dx_row, s)) != PTQ_OK) return st;
    if ((st = launch_gemm(h, workspace, M, y_fp16, acc_int32_out, s, false, dx_row)) != PTQ_OK) return st;
    if (q_int8_out)
        PTQ_CUDA(cudaMemcpy2DAsync(q_int8_out, h->K, workspace, h->Kpad, h->K, static_cast<size_t>(M),
                                   cudaMemcpyDeviceToDevice, s));
    if (step_fp32_out)
        PTQ_CUDA(cudaMemcpyAsync(step_fp32_out, dx_row, static_cast<size_t>(M) * sizeof(float),
                                 cudaMemcpyDeviceToDevice, s));
    return PTQ_OK;
}

ptq_status_t ptq_linear_forward_dynamic(const ptq_linear_t *h, const void *x_fp16, int B, void *y_fp16,
                                        void *workspace, size_t workspace_bytes, void *stream)
{
    return ptq_linear_forward_dynamic_debug(h, x_fp16, B, y_fp16, nullptr, nullptr, nullptr, workspace,
                                            workspace_bytes, stream);
}

ptq_status_t ptq_linear_device_status(const ptq_linear_t *h)
{
    if (!h) return fail(PTQ_ERR_NULL, "handle must not be NULL");
    ptq_status_t st = check_device(h);
    if (st != PTQ_OK) return st;
    unsigned word = 0;
    PTQ_CUDA(cudaDeviceSynchronize());
    PTQ_CUDA(cudaMemcpy(&word, h->d_status, sizeof(word), cudaMemcpyDeviceToHost));
    if (word & ptq::PTQ_DEV_SMEM_ALIGN) {
        PTQ_CUDA(cudaMemset(h->d_status, 0, sizeof(word)));
        return fail(PTQ_ERR_CUDA, "a kernel found its shared memory misaligned and did not run (status word 0x%x); its output is undefined", word);
    }
    if (word) {
        PTQ_CUDA(cudaMemset(h->d_status, 0, sizeof(word)));
        return fail(PTQ_ERR_TIMEOUT, "a kernel abandoned a bounded wait (status word 0x%x); its output is undefined", word);
    }
    return PTQ_OK;
}

ptq_status_t ptq_linear_selftest_wait_timeout(const ptq_linear_t *h, unsigned limit_us, unsigned *result3, void *stream)
{
    if (!h || !result3) return fail(PTQ_ERR_NULL, "handle and result must not be NULL");
    if (limit_us < 1 || limit_us > 100000) return fail(PTQ_ERR_VALUE, "limit_us must be in [1, 100000] (got %u)", limit_us);
    ptq_status_t st = check_device(h);
    if (st != PTQ_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    unsigned *d_out = nullptr;
    PTQ_CUDA(cudaMalloc(reinterpret_cast<void **>(&d_out), 3 * sizeof(unsigned)));
    auto body = [&]() -> ptq_status_t {
        PTQ_CUDA(cudaMemsetAsync(d_out, 0xff, 3 * sizeof(unsigned), s));
        ptq::ptq_wait_selftest_kernel<<<1, 64, 0, s>>>(h->d_status, 1000ull * limit_us, d_out);
        g_launches.fetch_add(1, std::memory_order_relaxed);
        PTQ_CUDA(cudaGetLastError());
        PTQ_CUDA(cudaMemcpyAsync(result3, d_out, 3 * sizeof(unsigned), cudaMemcpyDeviceToHost, s));
        PTQ_CUDA(cudaStreamSynchronize(s));
        return PTQ_OK;
    };
    st = body();
    cudaFree(d_out);
    return st;
}

ptq_status_t ptq_probe(int kind, void *buf, size_t bytes, int iters, double *result, void *stream)
{
    if (!result) return fail(PTQ_ERR_NULL, "probe: result must not be NULL");
    *result = 0.0;
    if (kind < ptq::kProbeStore16 || kind > ptq::kProbeLaunchPdl) return fail(PTQ_ERR_VALUE, "probe: unknown kind %d", kind);
    if (iters < 1 || iters > 100000) return fail(PTQ_ERR_VALUE, "probe: iters must be in [1, 100000] (got %d)", iters);
    const bool moves_bytes = kind <= ptq::kProbeOperandPull;
    if (moves_bytes && !buf) return fail(PTQ_ERR_NULL, "probe: buf must not be NULL for this kind");
    if (moves_bytes && reinterpret_cast<uintptr_t>(buf) % 256) return fail(PTQ_ERR_ALIGN, "probe: buf must be 256-byte aligned");
    int dev = -1, sms = 0, major = 0, minor = 0;
    PTQ_CUDA(cudaGetDevice(&dev));
    PTQ_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    PTQ_CUDA(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev));
    PTQ_CUDA(cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev));
    if (major != 10 || minor != 0)
        return fail(PTQ_ERR_ARCH, "device %d is compute capability %d.%d; this library needs 10.0 (sm_100a)", dev, major, minor);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    constexpr size_t kTail = 256;                      // the last 256 bytes of buf hold the kernels' status word
    constexpr int N = 3072, K = 768;                   // the Vim-B in_proj shape: y [M, 3072] fp16, codes [M, 768], weights [3072, 768]
    unsigned char *base = static_cast<unsigned char *>(buf);
    unsigned *status = moves_bytes ? reinterpret_cast<unsigned *>(base + (bytes >= kTail ? bytes - kTail : 0)) : nullptr;
    double moved = 0.0;                                // bytes per launch
    int grid = sms, m_tiles = 0;
    CUtensorMap tm0, tm1;
    if (kind == ptq::kProbeStore16) {
        if (bytes < kTail + (1u << 20)) return fail(PTQ_ERR_SHAPE, "probe: buf too small (%zu bytes)", bytes);
        moved = static_cast<double>((bytes - kTail) / 16 * 16);
        grid = sms * 32;
    } else if (kind == ptq::kProbeTmaStore) {
        m_tiles = static_cast<int>((bytes - (bytes >= kTail ? kTail : bytes)) / (static_cast<size_t>(N) * 2 * ptq::kBM));
        if (m_tiles < 1) return fail(PTQ_ERR_SHAPE, "probe: buf too small (%zu bytes)", bytes);
        if (m_tiles > 4096) m_tiles = 4096;
        ptq_status_t st = make_map_2d(&tm0, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, base, N, static_cast<unsigned long long>(m_tiles) * ptq::kBM,
                                      static_cast<unsigned long long>(N) * 2, 64, 32);
        if (st != PTQ_OK) return st;
        moved = static_cast<double>(m_tiles) * ptq::kBM * N * 2;
        PTQ_CUDA(cudaFuncSetAttribute(ptq::ptq_probe_tma_store_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 8 * ptq::kProbeBoxBytes));
    } else if (kind == ptq::kProbeOperandPull) {
        const size_t w_bytes = static_cast<size_t>(N) * K;
        if (bytes < kTail + w_bytes + static_cast<size_t>(ptq::kBM) * K) return fail(PTQ_ERR_SHAPE, "probe: buf too small (%zu bytes)", bytes);
        m_tiles = static_cast<int>((bytes - kTail - w_bytes) / (static_cast<size_t>(ptq::kBM) * K));
        if (m_tiles > 4096) m_tiles = 4096;
        ptq_status_t st = make_map_2d(&tm0, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, base + w_bytes, K, static_cast<unsigned long long>(m_tiles) * ptq::kBM, K, 128, 128);
        if (st == PTQ_OK) st = make_map_2d(&tm1, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, base, K, N, K, 128, 256);
        if (st != PTQ_OK) return st;
        moved = static_cast<double>(m_tiles) * (N / 256) * (K / 128) * ptq::kProbeStageBytes;
        PTQ_CUDA(cudaFuncSetAttribute(ptq::ptq_probe_operand_pull_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      4 * ptq::kProbeStageBytes + 128));
    }
    if (status) PTQ_CUDA(cudaMemsetAsync(status, 0, sizeof(unsigned), s));
    auto launch = [&]() -> cudaError_t {
        switch (kind) {
            case ptq::kProbeStore16:
                ptq::ptq_probe_store16_kernel<<<grid, 256, 0, s>>>(reinterpret_cast<uint4 *>(base), static_cast<unsigned long long>(moved / 16));
                break;
            case ptq::kProbeTmaStore:
                ptq::ptq_probe_tma_store_kernel<<<sms, 256, 8 * ptq::kProbeBoxBytes, s>>>(tm0, m_tiles, N / 256);
                break;
            case ptq::kProbeOperandPull:
                ptq::ptq_probe_operand_pull_kernel<<<sms, 64, 4 * ptq::kProbeStageBytes + 128, s>>>(tm0, tm1, m_tiles, N / 256, K / 128, status);
                break;
            case ptq::kProbeLaunch:
                ptq::ptq_probe_empty_kernel<<<sms, 256, 0, s>>>(0);
                break;
            default:
                return launch_pdl(ptq::ptq_probe_empty_kernel, sms, 256, 0, s, 1);
        }
        return cudaGetLastError();
    };
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    PTQ_CUDA(cudaEventCreate(&e0));
    cudaError_t err = cudaEventCreate(&e1);
    for (int i = 0; i < 3 && err == cudaSuccess; ++i) err = launch();
    if (err == cudaSuccess) err = cudaEventRecord(e0, s);
    for (int i = 0; i < iters && err == cudaSuccess; ++i) err = launch();
    if (err == cudaSuccess) err = cudaEventRecord(e1, s);
    if (err == cudaSuccess) err = cudaEventSynchronize(e1);
    float ms = 0.0f;
    if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, e0, e1);
    g_launches.fetch_add(static_cast<unsigned long long>(iters) + 3ull, std::memory_order_relaxed);
    cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (err != cudaSuccess) return fail(PTQ_ERR_CUDA, "probe: %s", cudaGetErrorString(err));
    if (status) {
        unsigned word = 0;
        PTQ_CUDA(cudaMemcpy(&word, status, sizeof(word), cudaMemcpyDeviceToHost));
        if (word) return fail(PTQ_ERR_TIMEOUT, "probe: a bounded wait gave up (status word 0x%x)", word);
    }
    const double per_launch_s = static_cast<double>(ms) * 1e-3 / iters;
    *result = moves_bytes ? moved / per_launch_s / 1e9 : per_launch_s * 1e6;   // GB/s, or microseconds per launch
    return PTQ_OK;
}

// Device workspace of a calibration: accumulators (zeroed per call), results, weight steps, weights.
struct CalibLayout {
    size_t bits, out, dw, w, total;     // byte offsets and size
};
static CalibLayout calib_layout(int K, int N, int T)
{
    auto up = [](size_t v) { return (v + 255) / 256 * 256; };
    CalibLayout l;
    l.bits = 0;                                                                  // [K] maxX, [T] mu (or hi), [T] -lo, [K] maxW
    l.out = up(sizeof(unsigned) * (2 * static_cast<size_t>(K) + 2 * static_cast<size_t>(T)));   // [K] s, [T] dx, [T] z
    l.dw = l.out + up(sizeof(float) * (static_cast<size_t>(K) + 2 * static_cast<size_t>(T)));
    l.w = l.dw + up(sizeof(float) * static_cast<size_t>(N));
    l.total = l.w + up(static_cast<size_t>(N) * K);
    return l;
}

size_t ptq_calibrate_workspace_bytes(int K, int N, int T)
{
    if (K < 1 || K > PTQ_MAX_K || N < 1 || N > PTQ_MAX_N || T < 1 || T > PTQ_MAX_T) return 0;
    return calib_layout(K, N, T).total;
}

static ptq_status_t calibrate_impl(int scheme, int K, int N, int T, const void *xcal_fp16, int Bc, const void *w_q,
                                   const float *w_step, float *smooth_out, float *act_step_out, int32_t *act_zero_out,
                                   void *workspace, size_t workspace_bytes, void *stream)
{
    const bool asym = scheme == PTQ_CALIB_ASYM, packed = scheme == PTQ_CALIB_W4A4;
    if (scheme < PTQ_CALIB_PTS || scheme > PTQ_CALIB_W4A4) return fail(PTQ_ERR_VALUE, "calibrate: unknown scheme %d", scheme);
    if (!xcal_fp16 || !w_q || !w_step || !smooth_out || !act_step_out || (asym && !act_zero_out) || !workspace)
        return fail(PTQ_ERR_NULL, "calibrate: pointers must not be NULL");
    if (K < 1 || K > PTQ_MAX_K || N < 1 || N > PTQ_MAX_N || T < 1 || T > PTQ_MAX_T || Bc < 1)
        return fail(PTQ_ERR_SHAPE, "calibrate: dimensions out of range (K=%d N=%d T=%d Bc=%d)", K, N, T, Bc);
    if (reinterpret_cast<uintptr_t>(xcal_fp16) % 2) return fail(PTQ_ERR_ALIGN, "xcal must be 2-byte aligned");
    const CalibLayout l = calib_layout(K, N, T);
    if (workspace_bytes < l.total)
        return fail(PTQ_ERR_SHAPE, "calibrate: workspace has %zu bytes, %zu needed", workspace_bytes, l.total);
    if (reinterpret_cast<uintptr_t>(workspace) % 256) return fail(PTQ_ERR_ALIGN, "calibrate: workspace must be 256-byte aligned");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const long long M = static_cast<long long>(Bc) * T;
    const __half *x = static_cast<const __half *>(xcal_fp16);
    unsigned char *base = static_cast<unsigned char *>(workspace);
    unsigned *d_xbits = reinterpret_cast<unsigned *>(base + l.bits), *d_hi = d_xbits + K, *d_nlo = d_hi + T, *d_wbits = d_nlo + T;
    float *d_s = reinterpret_cast<float *>(base + l.out), *d_dx = d_s + K;
    int *d_z = reinterpret_cast<int *>(d_dx + T);
    float *d_dw = reinterpret_cast<float *>(base + l.dw);
    uint8_t *d_w = base + l.w;
    const int row_bytes = packed ? (K + 1) / 2 : K;
    // one copy back: s, dx and (asymmetric) z are adjacent
    const size_t words = static_cast<size_t>(K) + static_cast<size_t>(T) * (asym ? 2 : 1);
    std::vector<float> got(words);

    int dev = -1, sms = 0;
    PTQ_CUDA(cudaGetDevice(&dev));
    PTQ_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));

    // The activations' column maxima first: they run while the weights are on their way from the host.
    PTQ_CUDA(cudaMemsetAsync(d_xbits, 0, sizeof(unsigned) * (2 * static_cast<size_t>(K) + 2 * static_cast<size_t>(T)), s));
    const bool vec = K % 8 == 0 && reinterpret_cast<uintptr_t>(x) % 16 == 0;
    const int cpr = vec ? K / 8 : K;
    const int cgroups = (cpr + ptq::kCalibGroup - 1) / ptq::kCalibGroup;
    const long long rp = 256 / (cpr < ptq::kCalibGroup ? cpr : ptq::kCalibGroup);
    long long rpb = (M * cgroups + 2 * sms - 1) / (2 * sms);              // about two blocks per SM, four rows per thread at least
    if (rpb < 4 * rp) rpb = 4 * rp;
    const long long shares = (M + rpb - 1) / rpb;
    const dim3 cgrid(static_cast<unsigned>(cgroups), static_cast<unsigned>(shares));
    if (vec)
        ptq::ptq_calib_colmax_kernel<8><<<cgrid, 256, 0, s>>>(x, M, K, static_cast<int>(rpb), d_xbits);
    else
        ptq::ptq_calib_colmax_kernel<1><<<cgrid, 256, 0, s>>>(x, M, K, static_cast<int>(rpb), d_xbits);
    PTQ_CUDA(cudaMemcpyAsync(d_dw, w_step, sizeof(float) * N, cudaMemcpyHostToDevice, s));
    PTQ_CUDA(cudaMemcpyAsync(d_w, w_q, static_cast<size_t>(N) * row_bytes, cudaMemcpyHostToDevice, s));
    const bool w4 = row_bytes % 4 == 0;
    const int groups = w4 ? row_bytes / 4 : row_bytes;
    const int wcols = (groups + 127) / 128;
    int wrows = (N * wcols + 2 * sms - 1) / (2 * sms);                    // about two blocks per SM, 16 rows at least
    if (wrows < 16) wrows = 16;
    const dim3 wgrid(static_cast<unsigned>(wcols), static_cast<unsigned>((N + wrows - 1) / wrows));
    if (packed && w4)
        ptq::ptq_calib_wmax_kernel<4, true><<<wgrid, 128, 0, s>>>(d_w, d_dw, N, K, wrows, d_wbits);
    else if (packed)
        ptq::ptq_calib_wmax_kernel<1, true><<<wgrid, 128, 0, s>>>(d_w, d_dw, N, K, wrows, d_wbits);
    else if (w4)
        ptq::ptq_calib_wmax_kernel<4, false><<<wgrid, 128, 0, s>>>(d_w, d_dw, N, K, wrows, d_wbits);
    else
        ptq::ptq_calib_wmax_kernel<1, false><<<wgrid, 128, 0, s>>>(d_w, d_dw, N, K, wrows, d_wbits);
    const ptq::CalibShares shares_of_position = ptq::calib_shares(Bc, T, sms);
    ptq::CalibRange r;
    r.x = x;
    r.max_x_bits = d_xbits;
    r.max_w_bits = d_wbits;
    r.hi_bits = d_hi;
    r.nlo_bits = d_nlo;
    r.s = d_s;
    r.dx = d_dx;
    r.z = d_z;
    r.Bc = Bc;
    r.imgs_per_block = shares_of_position.images;
    r.K = K;
    r.T = T;
    r.qmax = packed ? 7.0f : 127.0f;
    const dim3 rgrid(static_cast<unsigned>(T), static_cast<unsigned>(shares_of_position.blocks));
    r.final = rgrid.y == 1 && scheme != PTQ_CALIB_PER_TENSOR ? 1 : 0;
    if (asym)
        vec ? ptq::ptq_calib_rowrange_kernel<8, true><<<rgrid, 128, 0, s>>>(r) : ptq::ptq_calib_rowrange_kernel<1, true><<<rgrid, 128, 0, s>>>(r);
    else
        vec ? ptq::ptq_calib_rowrange_kernel<8, false><<<rgrid, 128, 0, s>>>(r) : ptq::ptq_calib_rowrange_kernel<1, false><<<rgrid, 128, 0, s>>>(r);
    if (scheme == PTQ_CALIB_PER_TENSOR)
        ptq::ptq_calib_step_tensor_kernel<<<1, 256, 0, s>>>(d_hi, T, d_dx, 127.0f);
    else if (!r.final && asym)
        ptq::ptq_calib_step_asym_kernel<<<(T + 127) / 128, 128, 0, s>>>(d_hi, d_nlo, T, d_dx, d_z);
    else if (!r.final)
        ptq::ptq_calib_step_kernel<<<(T + 127) / 128, 128, 0, s>>>(d_hi, T, d_dx, r.qmax);
    g_launches.fetch_add(r.final ? 3 : 4, std::memory_order_relaxed);
    PTQ_CUDA(cudaGetLastError());
    PTQ_CUDA(cudaMemcpyAsync(got.data(), d_s, sizeof(float) * words, cudaMemcpyDeviceToHost, s));
    PTQ_CUDA(cudaStreamSynchronize(s));
    std::memcpy(smooth_out, got.data(), sizeof(float) * K);
    std::memcpy(act_step_out, got.data() + K, sizeof(float) * T);
    if (asym) std::memcpy(act_zero_out, got.data() + K + T, sizeof(int32_t) * T);
    return PTQ_OK;
}

ptq_status_t ptq_calibrate_in(int scheme, int K, int N, int T, const void *xcal_fp16, int Bc, const void *w_q,
                              const float *w_step, float *smooth_out, float *act_step_out, int32_t *act_zero_out,
                              void *workspace, size_t workspace_bytes, void *stream)
{
    return no_throw([&] {
        return calibrate_impl(scheme, K, N, T, xcal_fp16, Bc, w_q, w_step, smooth_out, act_step_out, act_zero_out, workspace,
                              workspace_bytes, stream);
    });
}

// The entry points without a caller workspace: one temporary device allocation around ptq_calibrate_in.
static ptq_status_t calibrate_alloc(int scheme, int K, int N, int T, const void *xcal_fp16, int Bc, const void *w_q,
                                    const float *w_step, float *smooth_out, float *act_step_out, int32_t *act_zero_out,
                                    void *stream)
{
    if (!xcal_fp16 || !w_q || !w_step || !smooth_out || !act_step_out || (scheme == PTQ_CALIB_ASYM && !act_zero_out))
        return fail(PTQ_ERR_NULL, "calibrate: pointers must not be NULL");
    const size_t bytes = ptq_calibrate_workspace_bytes(K, N, T);
    if (bytes == 0 || Bc < 1)
        return fail(PTQ_ERR_SHAPE, "calibrate: dimensions out of range (K=%d N=%d T=%d Bc=%d)", K, N, T, Bc);
    void *ws = nullptr;
    PTQ_CUDA(cudaMalloc(&ws, bytes));
    const ptq_status_t st = ptq_calibrate_in(scheme, K, N, T, xcal_fp16, Bc, w_q, w_step, smooth_out, act_step_out,
                                             act_zero_out, ws, bytes, stream);
    cudaFree(ws);
    return st;
}

ptq_status_t ptq_calibrate(int K, int N, int T, const void *xcal_fp16, int Bc, const int8_t *w_q,
                           const float *w_step, float *smooth_out, float *act_step_out, void *stream)
{
    return calibrate_alloc(PTQ_CALIB_PTS, K, N, T, xcal_fp16, Bc, w_q, w_step, smooth_out, act_step_out, nullptr, stream);
}

ptq_status_t ptq_calibrate_per_tensor(int K, int N, int T, const void *xcal_fp16, int Bc, const int8_t *w_q,
                                      const float *w_step, float *smooth_out, float *act_step_out, void *stream)
{
    return calibrate_alloc(PTQ_CALIB_PER_TENSOR, K, N, T, xcal_fp16, Bc, w_q, w_step, smooth_out, act_step_out, nullptr, stream);
}

ptq_status_t ptq_calibrate_asym(int K, int N, int T, const void *xcal_fp16, int Bc, const int8_t *w_q,
                                const float *w_step, float *smooth_out, float *act_step_out,
                                int32_t *act_zero_out, void *stream)
{
    return calibrate_alloc(PTQ_CALIB_ASYM, K, N, T, xcal_fp16, Bc, w_q, w_step, smooth_out, act_step_out, act_zero_out, stream);
}

ptq_status_t ptq_calibrate_w4a4(int K, int N, int T, const void *xcal_fp16, int Bc, const uint8_t *w_q_packed,
                                const float *w_step, float *smooth_out, float *act_step_out, void *stream)
{
    return calibrate_alloc(PTQ_CALIB_W4A4, K, N, T, xcal_fp16, Bc, w_q_packed, w_step, smooth_out, act_step_out, nullptr, stream);
}

// Sign-extending unpack of rows of 4-bit values, two per byte, low nibble = even column.
static void unpack_int4_host(const uint8_t *packed, int rows, int cols, std::vector<int8_t> &out)
{
    const int pb = (cols + 1) / 2;
    out.resize(static_cast<size_t>(rows) * cols);
    for (int r = 0; r < rows; ++r)
        for (int k = 0; k < cols; ++k) {
            const int nib = (packed[static_cast<size_t>(r) * pb + k / 2] >> ((k & 1) * 4)) & 15;
            out[static_cast<size_t>(r) * cols + k] = static_cast<int8_t>(nib >= 8 ? nib - 16 : nib);
        }
}

ptq_status_t ptq_linear_create_w4a4(ptq_linear_t **out, int K, int N, int T, const uint8_t *w_q_packed,
                                    const float *w_step, const float *smooth, const float *act_step,
                                    const float *bias, unsigned flags)
{
    if (!out) return fail(PTQ_ERR_NULL, "out must not be NULL");
    *out = nullptr;
    if (!w_q_packed) return fail(PTQ_ERR_NULL, "w_q_packed must not be NULL");
    if (K < 1 || K > PTQ_MAX_K || N < 1 || N > PTQ_MAX_N)
        return fail(PTQ_ERR_SHAPE, "K, N out of range (K=%d N=%d)", K, N);
    return no_throw([&] {
        std::vector<int8_t> w;
        unpack_int4_host(w_q_packed, N, K, w);
        return create_impl(out, K, N, T, w.data(), w_step, smooth, act_step, nullptr, bias, flags, 4);
    });
}

ptq_status_t ptq_quantize_packed4(const ptq_linear_t *h, const void *x_fp16, int B, void *q_packed, void *workspace,
                                  size_t workspace_bytes, void *stream)
{
    if (!h || !x_fp16 || !q_packed || !workspace) return fail(PTQ_ERR_NULL, "handle, x, q and workspace must not be NULL");
    if (h->act_bits != 4) return fail(PTQ_ERR_VALUE, "packed 4-bit codes need a layer made by ptq_linear_create_w4a4");
    if (B < 1) return fail(PTQ_ERR_SHAPE, "B must be >= 1 (got %d)", B);
    if (reinterpret_cast<uintptr_t>(x_fp16) % 2) return fail(PTQ_ERR_ALIGN, "x must be 2-byte aligned");
    if (reinterpret_cast<uintptr_t>(workspace) % 16) return fail(PTQ_ERR_ALIGN, "workspace must be 16-byte aligned");
    ptq_status_t st = check_device(h);
    if (st != PTQ_OK) return st;
    const long long M = static_cast<long long>(B) * h->T;
    const size_t need = static_cast<size_t>(M) * h->Kpad;
    if (workspace_bytes < need) return fail(PTQ_ERR_SHAPE, "workspace has %zu bytes, %zu needed", workspace_bytes, need);
    const size_t out_bytes = static_cast<size_t>(M) * ((h->K + 1) / 2);
    if (ranges_overlap(workspace, need, q_packed, out_bytes) ||
        ranges_overlap(workspace, need, x_fp16, static_cast<size_t>(M) * h->K * 2) ||
        ranges_overlap(q_packed, out_bytes, x_fp16, static_cast<size_t>(M) * h->K * 2))
        return fail(PTQ_ERR_VALUE, "x, q and workspace overlap");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if ((st = launch_quantize(h, x_fp16, M, workspace, h->Kpad, s)) != PTQ_OK) return st;
    long long want = (static_cast<long long>(out_bytes) + 255) / 256;
    const long long cap = static_cast<long long>(h->num_sms) * 16;
    if (want > cap) want = cap;
    ptq::ptq_pack_int4_kernel<<<static_cast<int>(want), 256, 0, s>>>(static_cast<const int8_t *>(workspace), M, h->K,
                                                                    h->Kpad, static_cast<uint8_t *>(q_packed));
    g_launches.fetch_add(1, std::memory_order_relaxed);
    PTQ_CUDA(cudaGetLastError());
    return PTQ_OK;
}

}  // extern "C"
