// C ABI of the SLoPe 2:4-sparse linear layer for B200 (sm_100a): argument checks,
// TMA descriptor construction and kernel launches.  No device memory is allocated here.
#include "../../include/slope.h"

#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <type_traits>
#include <utility>

#include "adapter_kernels.cuh"
#include "dw_adapter_kernel.cuh"
#include "gemm_kernels.cuh"
#include "nm_kernels.cuh"
#include "prune_kernels.cuh"

namespace slope {

static std::atomic<unsigned long long> g_launches{0};

// ------------------------------------------------------------------ device / driver set-up
struct DeviceInfo {
    bool ok = false;
    int dev = 0;
    int sm_count = 0;
    int cc_major = 0;
};

static DeviceInfo device_info() {
    thread_local DeviceInfo cache[64];                       // (per host thread: no lock on every call)
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return DeviceInfo{};
    if (!cache[dev].ok) {
        cudaDeviceProp prop;
        if (cudaGetDeviceProperties(&prop, dev) != cudaSuccess) return DeviceInfo{};
        cache[dev] = DeviceInfo{true, dev, prop.multiProcessorCount, prop.major};
    }
    return cache[dev];
}

// Results of the estimates below, which are pure functions of sizes and of the device: a layer asks for the same ones
// step after step, and working one out costs the host 0.5 ... 5 us.  A small direct-mapped table per host
// thread and estimate.
template <typename V>
struct SizeMemo {
    struct Slot {
        bool valid;
        int key[6];
        V value;
    };
    Slot slots[64] = {};
    template <typename Make>
    const V& get(const int (&key)[6], Make make) {
        unsigned h = 2166136261u;
        for (int k : key) h = (h ^ static_cast<unsigned>(k)) * 16777619u;
        Slot& s = slots[(h ^ (h >> 15)) % 64];
        if (!s.valid || std::memcmp(s.key, key, sizeof(key)) != 0) {
            s.value = make();
            std::memcpy(s.key, key, sizeof(key));
            s.valid = true;
        }
        return s.value;
    }
};

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* sym = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(sym);
    });
    return fn;
}

// Encoding a tensor map is a pure function of (address, extents, box, kind) and costs the host
// about a microsecond; a layer calls with the same buffers step after step.  Each host thread
// keeps the last encodings in a small direct-mapped table (no locks, nothing shared).
struct TmapKey {
    const void* base;
    long long rows;
    int cols, box_rows, box_cols, kind;
    bool operator==(const TmapKey& o) const {
        return base == o.base && rows == o.rows && cols == o.cols && box_rows == o.box_rows && box_cols == o.box_cols &&
               kind == o.kind;
    }
};
struct TmapSlot {
    TmapKey key;
    CUtensorMap tm;
    bool valid;
};
constexpr int kTmapSlots = 256;

static TmapSlot& tmap_slot(const TmapKey& k) {
    thread_local TmapSlot table[kTmapSlots] = {};
    unsigned long long h = reinterpret_cast<uintptr_t>(k.base) >> 4;
    h = h * 0x9E3779B97F4A7C15ull + static_cast<unsigned long long>(k.rows) * 0xC2B2AE3D27D4EB4Full;
    h ^= (static_cast<unsigned long long>(k.cols) << 20) ^ (static_cast<unsigned long long>(k.box_rows) << 8) ^
         (static_cast<unsigned long long>(k.box_cols) << 2) ^ static_cast<unsigned long long>(k.kind);
    h ^= h >> 29;
    return table[h % kTmapSlots];
}

template <typename Encode>
static bool tmap_memo(CUtensorMap* tm, const TmapKey& key, Encode encode) {
    TmapSlot& slot = tmap_slot(key);
    if (slot.valid && slot.key == key) {
        std::memcpy(tm, &slot.tm, sizeof(CUtensorMap));
        return true;
    }
    if (!encode(tm)) return false;
    slot.key = key;
    std::memcpy(&slot.tm, tm, sizeof(CUtensorMap));
    slot.valid = true;
    return true;
}

// 2-D bf16 tensor map over a row-major [rows x cols] matrix, 128-byte swizzle,
// box = box_cols (<= 64) x box_rows, out-of-bounds elements read as zero.
static bool make_tmap(CUtensorMap* tm, const void* base, int rows, int cols, int box_rows, int box_cols) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t gdim[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
    const cuuint64_t gstride[1] = {static_cast<cuuint64_t>(cols) * 2};
    const cuuint32_t box[2] = {static_cast<cuuint32_t>(box_cols), static_cast<cuuint32_t>(box_rows)};
    const cuuint32_t estr[2] = {1, 1};
    return tmap_memo(tm, TmapKey{base, rows, cols, box_rows, box_cols, 0}, [&](CUtensorMap* out) {
        return fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), gdim, gstride, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    });
}

// Metadata as a 2-D tensor of 8-byte words [blocks x 256]: one 2 KB block is ONE contiguous row,
// so a block costs the TMA unit a single request (a 128 x 16-byte box costs 128).
static bool make_tmap_meta(CUtensorMap* tm, const void* base, size_t total_bytes) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t gdim[2] = {256, static_cast<cuuint64_t>(total_bytes / 2048)};
    const cuuint64_t gstride[1] = {2048};
    const cuuint32_t box[2] = {256, 1};
    const cuuint32_t estr[2] = {1, 1};
    return tmap_memo(tm, TmapKey{base, static_cast<long long>(total_bytes / 2048), 256, 1, 256, 1}, [&](CUtensorMap* out) {
        return fn(out, CU_TENSOR_MAP_DATA_TYPE_UINT64, 2, const_cast<void*>(base), gdim, gstride, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    });
}

// 2-D bf16 tensor map for the TMA stores of the transposing epilogues: boxes 64 bytes wide, with the 64-byte swizzle their
// staging tiles are written in.
static bool make_tmap_out(CUtensorMap* tm, const void* base, int rows, int cols, int box_rows, int box_cols) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t gdim[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
    const cuuint64_t gstride[1] = {static_cast<cuuint64_t>(cols) * 2};
    const cuuint32_t box[2] = {static_cast<cuuint32_t>(box_cols), static_cast<cuuint32_t>(box_rows)};
    const cuuint32_t estr[2] = {1, 1};
    return tmap_memo(tm, TmapKey{base, rows, cols, box_rows, box_cols, 3}, [&](CUtensorMap* out) {
        return fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), gdim, gstride, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                  CU_TENSOR_MAP_L2_PROMOTION_NONE,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    });
}

// Launch with thread-block clusters of `cluster` CTAs along x.
template <typename... KArgs, typename... Args>
static slope_status_t launch_cluster_ex(void (*kern)(KArgs...), int grid, int cluster, int threads, int smem_bytes,
                                        bool overlap_prologue, cudaStream_t stream, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem_bytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    // Programmatic dependent launch: the kernel may be scheduled while its predecessor in the
    // stream drains; it synchronises on the device (griddepcontrol.wait) before touching memory.
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap_prologue ? 2 : 1;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return err == cudaSuccess && cudaGetLastError() == cudaSuccess ? SLOPE_OK : SLOPE_ERR_CUDA;
}

// How many clusters of `cluster` CTAs of this kernel the device holds at once (0: query failed).
template <typename Kernel>
static int max_active_clusters(Kernel kern, int cluster, int threads, int smem_bytes, int sm_count) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster * sm_count * 8, 1, 1);      // (the answer is capped by the grid of the query)
    cfg.blockDim = dim3(threads, 1, 1);
    cfg.dynamicSmemBytes = smem_bytes;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = cluster;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

// Launch on clusters of two CTAs (cta_group::2 kernels).
template <typename... KArgs, typename... Args>
static slope_status_t launch_pairs(void (*kern)(KArgs...), int grid, int threads, int smem_bytes,
                                   cudaStream_t stream, Args&&... args) {
    return launch_cluster_ex(kern, grid, 2, threads, smem_bytes, /*overlap_prologue=*/true, stream,
                             std::forward<Args>(args)...);
}

static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

static slope_status_t check_arch(DeviceInfo& info) {
    info = device_info();
    if (!info.ok) return SLOPE_ERR_CUDA;
    if (info.cc_major != 10) return SLOPE_ERR_UNSUPPORTED_ARCH;
    return SLOPE_OK;
}

static slope_status_t launch_result() {
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return cudaGetLastError() == cudaSuccess ? SLOPE_OK : SLOPE_ERR_CUDA;
}

// Opt in to more than 48 KB of dynamic shared memory.  The attribute belongs to the kernel in
// the current device's context; every host thread remembers which (kernel, device) pairs it has
// already set (a process-wide flag would be wrong for a second device).
template <typename Kernel>
static bool set_smem(Kernel k, int bytes) {
    struct Done {
        const void* fn;
        int dev, bytes;
    };
    constexpr int kMax = 64;
    thread_local Done done[kMax];
    thread_local int n_done = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    const void* fn = reinterpret_cast<const void*>(k);
    for (int i = 0; i < n_done; ++i)
        if (done[i].fn == fn && done[i].dev == dev && done[i].bytes >= bytes) return true;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
    // all of the SM's L1 / shared memory as shared memory: a kernel that asks for under half of it
    // would otherwise get a carve-out that holds only one of its CTAs
    if (cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) !=
        cudaSuccess)
        return false;
    if (n_done < kMax) done[n_done++] = Done{fn, dev, bytes};
    return true;
}

// Streaming kernels are launched with programmatic stream serialisation too: every thread waits for the preceding
// kernel before it touches memory (griddep_stream), but the blocks are set up by then, and on large grids the
// ramp-up and tail of back-to-back passes overlap.
template <typename... KArgs, typename... Args>
static slope_status_t launch_stream(void (*kern)(KArgs...), dim3 grid, cudaStream_t stream, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(256, 1, 1);
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return err == cudaSuccess && cudaGetLastError() == cudaSuccess ? SLOPE_OK : SLOPE_ERR_CUDA;
}

// Grid of the grid-stride streaming kernels: many short blocks per SM keep the tail of the last
// wave short (masked copy of a 90 MB matrix: 78 % of the HBM peak with 8 blocks per SM, 91 % with 32).
constexpr int kStreamBlocksPerSm = 32;
static unsigned stream_grid(size_t threads, const DeviceInfo& info) {
    const size_t blocks = (threads + 255) / 256, most = static_cast<size_t>(info.sm_count) * kStreamBlocksPerSm;
    return static_cast<unsigned>(blocks < most ? blocks : most);
}

// ------------------------------------------------------------------ adapter products
struct AdapterOperands {
    const void* A = nullptr;      // the large operand: [M x K], or [K x M] when A_MN
    const void* B = nullptr;      // [N x K], or [K x N] when B_MN
    void* out = nullptr;
    int M = 0;
    int transposed = 0;
};

// Column tile, reduction split (= cluster size) and ring depth of an adapter launch, by estimate.
struct AdapterPlan {
    int n_tile, splits;
    bool deep;                    // one CTA per SM with all of its shared memory; else two that share it
    double us;                    // estimated time, less the launch
};
struct AdapterShape {
    int row_tiles, box_rows;      // 128-row tiles of both problems; rows of the large operand's box
    double a_bytes;               // of the large operands
    int N, K;
    bool b_mn;                    // the small operand is loaded in chunks of 64 columns, whatever N is
};
// How the CTAs of a launch come to lie on the machine.
struct AdapterGrid {
    int ctas, col_tiles, waves, rank_kb;   // rank_kb: k-blocks of a CTA
    bool deep;
    double stages, busy;                   // ring depth; share of the SMs that are at work at a time
};
// SMs that clusters of `size` fill (33 of 4 and 15 of 8 fit on 148).
static int cluster_sms(int size, int sm_count) {
    return size == 8 ? sm_count * 120 / 148 : size == 4 ? sm_count * 132 / 148 : sm_count;
}
static AdapterGrid adapter_grid(const AdapterShape& q, int n_tile, int splits, int sm_count) {
    const int col_tiles = (q.N + n_tile - 1) / n_tile, ctas = q.row_tiles * col_tiles * splits;
    const int sms = cluster_sms(splits, sm_count);
    const bool deep = n_tile == 256 || ctas <= sms;
    const int slots = (deep ? 1 : 2) * sms, waves = (ctas + slots - 1) / slots, num_kb = (q.K + 63) / 64;
    const double stages = n_tile == 64 ? (deep ? 9 : 4) : n_tile == 128 ? (deep ? 7 : 3) : 4;
    return AdapterGrid{ctas, col_tiles, waves, (num_kb + splits - 1) / splits, deep, stages,
                       static_cast<double>(std::min(ctas, slots)) / sm_count};
}
// A launch that has the machine to itself.  Constants fitted to a sweep of tiles, splits and depths over 1 ... 16384 tokens,
// widths 128 ... 13824 and ranks 16 ... 256 (the choice is on average 0.1 %, at most 12 % slower than the best swept one;
// with a split's cost the same for any number of CTAs and boxes always full, dT of 6158 tokens and width 1408 took 7.8
// instead of 6.4 us, of 5 tokens and width 896 4.0 instead of 3.5):
//   - a round trip through the ring takes 1.2 us, a fifth more when all SMs are at it, so a k-block costs at
//     least that over its depth, and at least the rows of its boxes at 1300 a us;
//   - all CTAs together bring in 6.6 TB/s of the large operand, few of them less, and every further
//     column tile costs half of that again;
//   - draining 64 columns costs 0.75 us; when the tile is split 1.3 us more for the two barriers and, per 64
//     columns, what the cluster has to sum: the share of 128 rows that is there and the share of SMs in it.
static AdapterPlan adapter_candidate(const AdapterShape& q, int n_tile, int splits, int sm_count) {
    const AdapterGrid g = adapter_grid(q, n_tile, splits, sm_count);
    const int rows = q.box_rows + std::min(n_tile, q.b_mn ? (q.N + 63) / 64 * 64 : q.N);
    const double kb_us = std::max(1.2 * (1.0 + 0.2 * g.busy) / g.stages, (g.deep ? 1 : 2) * rows / 1300.0);
    const double hbm = std::min(6.6e6, 3.5e6 + 0.03e6 * g.ctas) / (1.0 + 0.5 * (g.col_tiles - 1));
    const double cols = n_tile / 64.0, tail = splits > 1 ? 1.3 + (0.3 + q.box_rows / 128.0 + g.busy) * cols : 0.75 * cols;
    return AdapterPlan{n_tile, splits, g.deep, std::max(g.waves * g.rank_kb * kb_us, q.a_bytes / hbm) + g.waves * tail};
}
// A T launch beside the tile kernel that consumes it.  Its constants go with those of plan_fwd_adapter, which weighs the
// two against each other; with the ones above, which know T alone, forwards of few rows got the wrong share of the
// machine (3057 tokens 9856 -> 384, r = 64: 32.3 instead of 26.4 us):
//   - a k-block costs 0.8 us over the ring's depth, and at least what the SM takes in (150 KB per us);
//   - a CTA brings in 90 GB/s of the large operand, dozens of them less, all together 6 TB/s, and every
//     further column tile costs 8 % of that (its second read comes from L2);
//   - draining a tile costs 0.3 us per 64 columns, 1 us more and 1 us per 64 columns when it is split.
static AdapterPlan adapter_beside_forward(const AdapterShape& q, int n_tile, int splits, int sm_count) {
    const AdapterGrid g = adapter_grid(q, n_tile, splits, sm_count);
    const double kb_us = std::max(0.8 / g.stages, (g.deep ? 1 : 2) * (16.0 + n_tile / 8.0) / 150.0);
    const double hbm = std::min({6.0e6, 0.09e6 * g.ctas, 2.2e6 + 0.03e6 * g.ctas}) / (1.0 + 0.08 * (g.col_tiles - 1));
    const double tail = (splits > 1 ? 1.0 : 0.3) * n_tile / 64.0 + (splits > 1 ? 1.0 : 0.0);
    return AdapterPlan{n_tile, splits, g.deep, std::max(g.waves * g.rank_kb * kb_us, q.a_bytes / hbm) + g.waves * tail};
}
template <typename Visit>
static void adapter_cuts(const AdapterShape& q, Visit visit) {
    for (int n_tile = 64; n_tile <= 256 && (n_tile == 64 || n_tile < 2 * q.N); n_tile *= 2)
        for (int s = 1; s <= 8 && (s == 1 || 2 * s <= (q.K + 63) / 64); s *= 2) visit(n_tile, s);
}
static AdapterPlan adapter_plan(const AdapterShape& q, int sm_count) {
    AdapterPlan best{64, 1, true, 1e30};
    adapter_cuts(q, [&](int n_tile, int splits) {
        const AdapterPlan c = adapter_candidate(q, n_tile, splits, sm_count);
        if (c.us < best.us - 1e-9) best = c;
    });
    return best;
}
// T = X L: `b` tokens of width `d_in`.
static AdapterShape adapter_T_shape(int b, int d_in, int r) {
    return AdapterShape{(b + kBlockM - 1) / kBlockM, adapter_box_rows(b, kBlockM), 2.0 * b * d_in, r, d_in, true};
}

// SMs that the CTAs of a launch over `rows` rows occupy.
static int adapter_sms(const AdapterPlan& plan, int rows, int N, int sm_count) {
    const int ctas = (rows + kBlockM - 1) / kBlockM * ((N + plan.n_tile - 1) / plan.n_tile) * plan.splits;
    return std::min(plan.deep ? ctas : (ctas + 1) / 2, sm_count);
}

template <bool A_MN, bool B_MN, int N_TILE>
static slope_status_t launch_adapter_tile(const AdapterOperands& q0, const AdapterOperands& q1, int N, int K, int splits,
                                          bool deep, cudaStream_t stream, int pdl_mode, const WeightPrefetch& next) {
    using Cfg = AdapterCfg<N_TILE>;
    CUtensorMap tm[4];
    AdapterProblem p[2];
    int tiles = 0;
    for (int i = 0; i < 2; ++i) {
        const bool live = i == 0 || q1.M > 0;
        const AdapterOperands& q = i == 0 ? q0 : (live ? q1 : q0);           // unused slot mirrors problem 0
        const bool okA = A_MN ? make_tmap(&tm[2 * i], q.A, K, q.M, 64, 64)
                              : make_tmap(&tm[2 * i], q.A, q.M, K, adapter_box_rows(q.M, kBlockM), 64);
        const bool okB = B_MN ? make_tmap(&tm[2 * i + 1], q.B, K, N, 64, 64)
                              : make_tmap(&tm[2 * i + 1], q.B, N, K, adapter_box_rows(N, N_TILE), 64);
        if (!okA || !okB) return SLOPE_ERR_CUDA;
        p[i] = AdapterProblem{live ? q.M : 0, N, K, static_cast<uint16_t*>(q.out), q.transposed};
        if (live) tiles += (q.M + kBlockM - 1) / kBlockM;
    }
    const int stages = deep || Cfg::kShared == 0 ? Cfg::kDeep : Cfg::kShared;
    const int ctas = tiles * ((N + N_TILE - 1) / N_TILE) * splits;
    const auto launch = [&](auto prefetch, int further) {
        auto kern = adapter_gemm_kernel<A_MN, B_MN, N_TILE, decltype(prefetch)>;
        if (!set_smem(kern, Cfg::smem_bytes(Cfg::kDeep))) return SLOPE_ERR_CUDA;
        return launch_cluster_ex(kern, ctas + further, splits, kGemmThreads, Cfg::smem_bytes(stages), /*overlap_prologue=*/true,
                                 stream, tm[0], tm[1], p[0], tm[2], tm[3], p[1], stages, pdl_mode, prefetch);
    };
    if constexpr (!A_MN && B_MN)                             // (T)
        if (next.blocks > 0) return launch(next, next.blocks);
    return launch(NoPrefetch{}, 0);
}

// D[M x N] = A B over one or two problems with the same N (= r) and K.
template <bool A_MN, bool B_MN>
static slope_status_t launch_adapter_planned(const AdapterPlan& plan, const AdapterOperands& q0, const AdapterOperands& q1,
                                             int N, int K, cudaStream_t stream, int pdl_mode,
                                             const WeightPrefetch& next = WeightPrefetch{}) {
    switch (plan.n_tile) {
        case 64: return launch_adapter_tile<A_MN, B_MN, 64>(q0, q1, N, K, plan.splits, plan.deep, stream, pdl_mode, next);
        case 128: return launch_adapter_tile<A_MN, B_MN, 128>(q0, q1, N, K, plan.splits, plan.deep, stream, pdl_mode, next);
        default: return launch_adapter_tile<A_MN, B_MN, 256>(q0, q1, N, K, plan.splits, plan.deep, stream, pdl_mode, next);
    }
}
template <bool A_MN, bool B_MN>
static slope_status_t launch_adapter(const AdapterOperands& q0, const AdapterOperands& q1, int N, int K,
                                     cudaStream_t stream, const DeviceInfo& info, int pdl_mode = 0) {
    thread_local SizeMemo<AdapterPlan> memo;
    const AdapterPlan& plan = memo.get({q0.M, q1.M, N, K, info.sm_count, 0}, [&] {
        const int row_tiles = (q0.M + kBlockM - 1) / kBlockM + (q1.M + kBlockM - 1) / kBlockM;
        const int box_rows = A_MN ? kBlockM : adapter_box_rows(std::max(q0.M, q1.M), kBlockM);
        return adapter_plan(AdapterShape{row_tiles, box_rows, 2.0 * K * (static_cast<double>(q0.M) + q1.M), N, K, B_MN},
                            info.sm_count);
    });
    return launch_adapter_planned<A_MN, B_MN>(plan, q0, q1, N, K, stream, pdl_mode);
}

// dT[b x r] = dY[b x d_out] * R[r x d_out]^T   (both K contiguous)
static slope_status_t launch_adapter_dT(const void* dY, const void* R, int b, int d_out, int r, void* dT,
                                        cudaStream_t stream, const DeviceInfo& info, int pdl_mode = 0) {
    return launch_adapter<false, false>(AdapterOperands{dY, R, dT, b, 0}, AdapterOperands{}, r, d_out, stream, info,
                                        pdl_mode);
}

// dR[r x d_out] = (dY^T T)^T and dL[d_in x r] = X^T dT: operands stored [K x M] / [K x N] with K = tokens.
static AdapterOperands adapter_dR(const void* dY, const void* T, int d_out, void* dR) {
    return AdapterOperands{dY, T, dR, d_out, 1};
}
static AdapterOperands adapter_dL(const void* X, const void* dT, int d_in, void* dL) {
    return AdapterOperands{X, dT, dL, d_in, 0};
}

// ------------------------------------------------------------------ CTA-pair launches (main GEMMs)
// Everything a launch of the two sparse tile kernels has in common.
struct SparseTileArgs {
    CUtensorMap tmA, tmB, tmE, tmA2, tmB2, tmO;
    SparseGemmParams p;
};
static bool sparse_tile_args(SparseTileArgs& a, const void* act, int ntok, const void* vals, const void* meta, int M, int K,
                             const void* act2, const void* fac2, int r, bool a2_mn, void* out, int width, int stages,
                             int pdl_mode) {
    if (!make_tmap(&a.tmA, vals, M, K / 2, kBlockM, 64) || !make_tmap(&a.tmB, act, ntok, K, width / 2, 64) ||
        !make_tmap_meta(&a.tmE, meta, static_cast<size_t>(M) * K / 8) ||
        !make_tmap_out(&a.tmO, out, ntok, M, SparsePairCfg::kStoreRows, SparsePairCfg::kStoreCols))
        return false;
    if (r > 0) {
        const bool ok2 = a2_mn ? make_tmap(&a.tmA2, fac2, r, M, 64, 64) : make_tmap(&a.tmA2, fac2, M, r, kBlockM, 64);
        if (!ok2 || !make_tmap(&a.tmB2, act2, ntok, r, width / 2, 64)) return false;
    } else {
        a.tmA2 = a.tmA;
        a.tmB2 = a.tmB;
    }
    a.p = SparseGemmParams{};
    a.p.M = M; a.p.K = K; a.p.Ntok = ntok; a.p.r = r; a.p.a2_mn_major = a2_mn ? 1 : 0;
    a.p.width = width; a.p.num_n = (ntok + width - 1) / width; a.p.stages = stages; a.p.pdl_mode = pdl_mode;
    a.p.out = static_cast<uint16_t*>(out);
    return true;
}

// Pipeline stages that fit beside the staging buffers at a tile width.
constexpr int kMaxTileSmem = 232448;
template <typename Cfg>
static int tile_stages(int width) {
    int n = kMaxTileStages;
    while (n > 1 && Cfg::smem_bytes(width, n) > kMaxTileSmem) --n;
    return n;
}

static slope_status_t launch_sparse_pair(const void* act, int ntok, const void* vals, const void* meta, int M, int K,
                                         const void* act2, const void* fac2, int r, bool a2_mn, void* out, int width,
                                         int max_pairs, cudaStream_t stream, int pdl_mode) {
    using Cfg = SparsePairCfg;
    SparseTileArgs a;
    const int stages = tile_stages<Cfg>(width);
    if (!sparse_tile_args(a, act, ntok, vals, meta, M, K, act2, fac2, r, a2_mn, out, width, stages, pdl_mode))
        return SLOPE_ERR_CUDA;
    if (!set_smem(sparse_gemm_pair_kernel, kMaxTileSmem)) return SLOPE_ERR_CUDA;
    const int tiles = ((M / kBlockM + 1) / 2) * ((ntok + width - 1) / width);
    const int pairs = std::min(tiles, max_pairs);
    return launch_pairs(sparse_gemm_pair_kernel, 2 * pairs, Cfg::kThreads, Cfg::smem_bytes(width, stages), stream, a.tmA,
                        a.tmB, a.tmE, a.tmA2, a.tmB2, a.tmO, a.p);
}

// Row tiles per raster group of the 512-row-tile kernel (see quad_tile).  All pairs that work on
// one token block share its activations, so with every row tile in one group the activations
// cross HBM once -- but a wave of the machine then touches the whole compressed weight, and
// when that is more than L2 keeps next to the streams (about 30 MB here) it is fetched again
// every wave.  Splitting the row tiles into g groups re-reads the activations g times and keeps
// a group's weights resident.  Pick the g with the least estimated DRAM traffic
// (measured at 16384 tokens: 4096 -> 11008 two groups +7 %, 5120 -> 13824 three groups +11 %,
// square and long-reduction layers one group).
static int quad_group_m(int M, int K, int ntok, int width, int num_pairs) {
    const int num_m = (M / kBlockM + 3) / 4, num_n = (ntok + width - 1) / width;
    const double w_tile = 512.0 * K * 1.125, w_total = static_cast<double>(M) * K * 1.125;
    const double x_total = static_cast<double>(ntok) * K * 2.0;
    constexpr double kL2Keeps = 30e6;
    int best_gm = num_m;
    double best = 1e300;
    for (int g = 1; g <= num_m; ++g) {
        const int gm = (num_m + g - 1) / g, groups = (num_m + gm - 1) / gm;
        const double rounds = static_cast<double>(gm) * num_n / num_pairs;
        const double traffic = groups * x_total + (gm * w_tile <= kL2Keeps ? w_total : w_total * (rounds > 1.0 ? rounds : 1.0));
        if (traffic < best * 0.98) { best = traffic; best_gm = gm; }       // prefer fewer groups on a near tie
    }
    return best_gm;
}

static slope_status_t launch_sparse_quad(const void* act, int ntok, const void* vals, const void* meta, int M, int K,
                                         const void* act2, const void* fac2, int r, bool a2_mn, void* out, int width,
                                         int max_pairs, cudaStream_t stream, int pdl_mode) {
    using Cfg = SparseQuadCfg;
    SparseTileArgs a;
    const int stages = tile_stages<Cfg>(width);
    if (!sparse_tile_args(a, act, ntok, vals, meta, M, K, act2, fac2, r, a2_mn, out, width, stages, pdl_mode))
        return SLOPE_ERR_CUDA;
    a.p.group_m = quad_group_m(M, K, ntok, width, max_pairs);
    if (!set_smem(sparse_gemm_quad_kernel, kMaxTileSmem)) return SLOPE_ERR_CUDA;
    const int tiles = ((M / kBlockM + 3) / 4) * ((ntok + width - 1) / width);
    const int pairs = std::min(tiles, max_pairs);
    return launch_pairs(sparse_gemm_quad_kernel, 2 * pairs, Cfg::kThreads, Cfg::smem_bytes(width, stages), stream, a.tmA,
                        a.tmB, a.tmE, a.tmA2, a.tmB2, a.tmO, a.p);
}

// Few tokens (inference / decode sizes): weight-streaming kernel, K split over a cluster.
// K-splits (= cluster size) of the few-token kernel.  A CTA streams ceil(num_kb / s) k-blocks
// of 18 KB.  Measured on B200: alone an SM takes in one k-block per ~0.23 us (about one TMA row
// request per 2 ns), and once enough CTAs pull at the same time HBM is the limit (18 KB at
// 6.5 TB/s = 0.0028 us per k-block and active CTA).  Every wave of clusters pays a fixed
// start-up (launch, prologue, first-byte latency, epilogue), a split pays the cluster
// reduction.  `capacity(s)` is the number of clusters of s CTAs the device holds at once.
constexpr double kSkinnySmUs = 0.23, kSkinnyHbmUs = 0.0028, kSkinnyWaveUs = 4.0, kSkinnyReduceUs = 0.5,
                 kSkinnyReducePerRankUs = 0.07;

// A k-block costs an SM its weight tile (kSkinnySmUs) plus the activation tile's TMA row
// requests (2 per token, ~2 ns each; charged for a full tile, as the constants were fitted, although a box has a row per token).
constexpr double kSkinnyTokenUs = 0.004;

static int skinny_splits(int slabs, int num_kb, int block_n, const int (&cap)[9], double* est_us = nullptr) {
    int best_s = 1;
    double best_cost = 1e30;
    const double sm_us = kSkinnySmUs + kSkinnyTokenUs * block_n;
    for (int s = 1; s <= 8; ++s) {
        const int per = (num_kb + s - 1) / s;
        if ((num_kb + per - 1) / per != s) continue;                 // a rank would be left without a k-block
        if (s > 1 && per < 2) break;
        if (cap[s] <= 0) continue;
        double cost = s > 1 ? kSkinnyReduceUs + kSkinnyReducePerRankUs * s : 0.0;
        for (int left = slabs; left > 0; left -= cap[s]) {
            const int active = (left < cap[s] ? left : cap[s]) * s;
            const double per_kb = active * kSkinnyHbmUs > sm_us ? active * kSkinnyHbmUs : sm_us;
            cost += kSkinnyWaveUs + per * per_kb;
        }
        if (cost < best_cost - 1e-9) { best_cost = cost; best_s = s; }
    }
    if (est_us) *est_us = best_cost;
    return best_s;
}

// Co-resident clusters of the few-token kernel per cluster size, asked of the driver once per
// device and kernel variant.
template <int BLOCK_N, int A_STAGES, int B_STAGES>
static bool skinny_capacity(const DeviceInfo& info, int (&cap)[9]) {
    using Cfg = SparseSkinnyCfg<BLOCK_N, A_STAGES, B_STAGES>;
    static std::mutex mu;
    static int capacity[64][9];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    auto kern = sparse_gemm_skinny_kernel<BLOCK_N, A_STAGES, B_STAGES>;
    std::lock_guard<std::mutex> lock(mu);
    if (capacity[dev][1] == 0) {
        if (!set_smem(kern, Cfg::kSmemBytes)) return false;
        for (int s = 1; s <= 8; ++s)
            capacity[dev][s] = max_active_clusters(kern, s, kGemmThreads, Cfg::kSmemBytes, info.sm_count);
    }
    // The occupancy query answers one CTA per SM for every kernel that allocates tensor memory,
    // whatever its shared memory (it cannot know how many columns a CTA will ask for).  The CTA
    // scheduler itself goes by registers, warps and shared memory: two CTAs of a variant that
    // needs under half of the shared memory do run side by side (measured: a launch of 172 CTAs
    // takes one wave, not two), and their 32- or 128-column allocations fit together.
    const int per_sm = 2 * (Cfg::kSmemBytes + 1024) <= 232448 ? 2 : 1;
    cap[0] = 0;
    for (int s = 1; s <= 8; ++s) cap[s] = capacity[dev][s] * per_sm;
    return cap[1] > 0;
}

// K-splits of a launch of the few-token kernel (0: the device has no room for it).
template <int BLOCK_N, int A_STAGES, int B_STAGES>
static int skinny_split_count(int ntok, int M, int K, int r, const DeviceInfo& info, int pdl_mode) {
    int cap[9];
    if (!skinny_capacity<BLOCK_N, A_STAGES, B_STAGES>(info, cap)) return 0;
    thread_local SizeMemo<int> memo;
    return memo.get({M, K, pdl_mode == 2 ? ntok : 0, pdl_mode == 2 ? r : 0, pdl_mode, info.dev}, [&] {
        if (pdl_mode == 2) {
            // The consumer of a fused pair has to be resident next to its producer, or its last clusters
            // would wait for the producer to finish and the overlap would be lost: count only the
            // clusters that fit beside it.
            const AdapterPlan producer = adapter_plan(adapter_T_shape(ntok, K, r), info.sm_count);
            const int reserved = adapter_sms(producer, ntok, r, info.sm_count);
            for (int sz = 1; sz <= 8; ++sz) {
                cap[sz] -= (reserved + sz - 1) / sz + (sz > 1 ? 1 : 0);
                if (cap[sz] < 0) cap[sz] = 0;
            }
            if (cap[1] <= 0) return 0;
        }
        return skinny_splits(M / kBlockM, K / 128, BLOCK_N, cap);
    });
}

template <int BLOCK_N, int A_STAGES, int B_STAGES>
static slope_status_t launch_sparse_skinny(const void* act, int ntok, const void* vals, const void* meta, int M, int K,
                                           const void* act2, const void* fac2, int r, bool a2_mn, void* out,
                                           cudaStream_t stream, const DeviceInfo& info, int pdl_mode) {
    using Cfg = SparseSkinnyCfg<BLOCK_N, A_STAGES, B_STAGES>;
    // An activation box has a row per token and no more: an SM takes about one 128-byte row of any box per 2 clocks, inside
    // the matrix or not, and what the MMAs read beyond them only reaches accumulator columns that are never stored.  us at one
    // token, boxes of 16 rows / of 1: 4096 -> 22016 23.2 / 20.0, 4096 -> 12288 13.3 / 12.3, 4096 -> 4096 7.1 / 6.9.
    const int rows = std::min(ntok, BLOCK_N);
    CUtensorMap tmA, tmB, tmE, tmA2, tmB2;
    if (r > 0) {
        const bool ok2 = a2_mn ? make_tmap(&tmA2, fac2, r, M, 64, 64) : make_tmap(&tmA2, fac2, M, r, kBlockM, 64);
        if (!ok2 || !make_tmap(&tmB2, act2, ntok, r, rows, 64)) return SLOPE_ERR_CUDA;
    }
    if (!make_tmap(&tmA, vals, M, K / 2, kBlockM, 64)) return SLOPE_ERR_CUDA;
    if (!make_tmap(&tmB, act, ntok, K, rows, 64)) return SLOPE_ERR_CUDA;
    if (!make_tmap_meta(&tmE, meta, static_cast<size_t>(M) * K / 8)) return SLOPE_ERR_CUDA;
    if (r <= 0) {
        tmA2 = tmA;
        tmB2 = tmB;
    }
    SparseGemmParams p = {};
    p.M = M; p.K = K; p.Ntok = ntok; p.r = r; p.a2_mn_major = a2_mn ? 1 : 0;
    p.pdl_mode = pdl_mode; p.width = rows;
    p.out = static_cast<uint16_t*>(out);
    auto kern = sparse_gemm_skinny_kernel<BLOCK_N, A_STAGES, B_STAGES>;
    if (!set_smem(kern, Cfg::kSmemBytes)) return SLOPE_ERR_CUDA;

    const int slabs = M / kBlockM, splits = skinny_split_count<BLOCK_N, A_STAGES, B_STAGES>(ntok, M, K, r, info, pdl_mode);
    if (splits == 0) return SLOPE_ERR_CUDA;
    return launch_cluster_ex(kern, slabs * splits, splits, kGemmThreads, Cfg::kSmemBytes, true, stream, tmA, tmB,
                             tmE, tmA2, tmB2, p);
}

// Few-token GEMM  out[ntok x M] = act * A_2:4^T (+ act2 * fac2^T)  on the weight-streaming kernel,
// token tile chosen by the token count (at most 128).
// A variant of the few-token kernel with a half as deep weight ring fits two CTAs on an SM (the
// same bytes in flight per SM).  It pays when the slabs times K-slices of a launch exceed what the
// machine holds at one CTA per SM (stacked projections, d_out beyond ~19000 rows): one wave
// instead of two.  Decided by the same cost model over both variants' capacities.
template <int BLOCK_N, int A_DEEP, int B_DEEP, int A_FLAT, int B_FLAT>
static bool prefer_two_ctas_per_sm(int M, int K, const DeviceInfo& info) {
    int cap_deep[9], cap_flat[9];
    if (!skinny_capacity<BLOCK_N, A_DEEP, B_DEEP>(info, cap_deep)) return false;
    if (!skinny_capacity<BLOCK_N, A_FLAT, B_FLAT>(info, cap_flat)) return false;
    double est_deep = 0.0, est_flat = 0.0;
    const int slabs = (M + kBlockM - 1) / kBlockM;
    skinny_splits(slabs, K / 128, BLOCK_N, cap_deep, &est_deep);
    skinny_splits(slabs, K / 128, BLOCK_N, cap_flat, &est_flat);
    return est_flat < 0.93 * est_deep;
}

// Calls visit(token tile, weight stages, activation stages), as integral constants, with the variant for a launch.
template <typename Visit>
static auto with_skinny_variant(int ntok, int M, int K, const DeviceInfo& info, Visit visit) {
    using std::integral_constant;
    if (ntok <= 16) {
        thread_local SizeMemo<bool> memo;
        if (memo.get({M, K, info.dev, 0, 0, 0}, [&] { return prefer_two_ctas_per_sm<16, 10, 4, 5, 2>(M, K, info); }))
            return visit(integral_constant<int, 16>{}, integral_constant<int, 5>{}, integral_constant<int, 2>{});
        return visit(integral_constant<int, 16>{}, integral_constant<int, 10>{}, integral_constant<int, 4>{});
    }
    if (ntok <= 64)      // (a two-per-SM variant of this tile, <64, 4, 2>, measured slower: its activation ring is too shallow)
        return visit(integral_constant<int, 64>{}, integral_constant<int, 8>{}, integral_constant<int, 4>{});
    return visit(integral_constant<int, 128>{}, integral_constant<int, 7>{}, integral_constant<int, 3>{});
}
static slope_status_t launch_skinny(const void* act, int ntok, const void* vals, const void* meta, int M, int K,
                                    const void* act2, const void* fac2, int r, bool a2_mn, void* out,
                                    cudaStream_t stream, const DeviceInfo& info, int pdl_mode = 0) {
    return with_skinny_variant(ntok, M, K, info, [&](auto n, auto a, auto b) {
        return launch_sparse_skinny<n(), a(), b()>(act, ntok, vals, meta, M, K, act2, fac2, r, a2_mn, out, stream, info, pdl_mode);
    });
}

// Tile of a sparse GEMM, by estimate:
//   512 rows   two MMA sub-tiles share an activation tile (fewer bytes per FLOP), but tensor memory then holds one
//              accumulator set and a tile's drain is exposed;
//   256 rows   double-buffered accumulators;
//   width      the token tiles of a launch are made equal (500 tokens: three of 192 and less rather than two of
//              224 and one of 64) and as wide as fills the waves of CTA pairs best.
// In SM clocks: a k-block takes the round trip of a pipeline stage (2130, 2515 with all pairs at work) over the stages
// that fit, and at least its bytes (70 per clock and SM) and its MMAs; a 512-row tile exposes 3.3 per token
// of width, the last drain of a launch takes 290 + 8.7 per token (2.4 times that for 512 rows), a launch
// 47 per pair.  Fitted to a sweep of all tiles over 18 layer shapes (768 ... 22016 wide) and 160 ... 8192
// tokens, where the choice is on average 0.7 %, at most 12 % slower than the best tile of the sweep.
struct SparseTile {
    int rows, width;
};
template <typename Cfg>
static double sparse_tile_cost(int M, double num_kb, int ntok, int width, int num_pairs) {
    const bool quad = std::is_same<Cfg, SparseQuadCfg>::value;
    const int rows = quad ? 512 : 256;
    const int tiles = ((M + rows - 1) / rows) * ((ntok + width - 1) / width), active = std::min(tiles, num_pairs);
    const double load = Cfg::stage_bytes(width) / 70.0, mma = rows * std::max(width, 64) / 128.0;
    const double round_trip = 2130.0 + 385.0 * active / num_pairs;
    const double k_block = std::max({round_trip / tile_stages<Cfg>(width), load, mma});
    const double tile = num_kb * k_block + (quad ? 3.3 * width : 0.0);
    const double last_drain = (quad ? 2.4 : 1.0) * (290.0 + 8.7 * width);
    return (tiles + num_pairs - 1) / num_pairs * tile + last_drain + 47.0 * active;
}
static SparseTile choose_sparse_tile(int M, int K, int ntok, int r, int num_pairs, double* cost = nullptr) {
    const double num_kb = K / 128 + 0.6 * ((r + 63) / 64);            // an adapter step is half a k-block of activations
    SparseTile best{256, 32};
    double best_cost = 1e300;
    for (int w = kMaxTokenTile; w >= 32; w -= 32) {
        const int n = (ntok + w - 1) / w, width = ((ntok + n - 1) / n + 31) & ~31;
        const double pair = sparse_tile_cost<SparsePairCfg>(M, num_kb, ntok, width, num_pairs);
        const double quad = sparse_tile_cost<SparseQuadCfg>(M, num_kb, ntok, width, num_pairs);
        if (pair < best_cost) { best_cost = pair; best = SparseTile{256, width}; }
        if (quad < best_cost) { best_cost = quad; best = SparseTile{512, width}; }
    }
    if (cost) *cost = best_cost;
    return best;
}

// Few-token kernel or tile kernel?  Decode sizes (<= 16 tokens) stream the weights through the few-token kernel.  From 17 to
// 128 tokens its K-split has to make up for boxes of every token in every CTA and for a drain that grows with the tokens,
// which takes a reduction that is the longer the more tokens and the more rows there are; a short one, or a tall weight, has
// the tile kernels' narrow tiles.  Up to 44 row slabs, which run in three slices side by side, the line is a fit to 760
// sizes on both kernels (0.2 % slower on average than the better one of the two; by the rule below, which compared the
// two extents only, 5 %); beyond them waves of slabs decide, and no simple line does.  us, few-token / tile kernel: 32 tokens 4096 -> 4096
// 7.8 / 9.2, 1024 -> 1024 4.4 / 4.1, 3072 -> 768 4.7 / 6.4; 64 tokens 512 -> 256 5.0 / 3.4, 2048 -> 1024 5.3 / 5.4, 2048 -> 2048
// 5.8 / 5.4, 4096 -> 4096 8.6 / 9.3; 128 tokens 256 -> 128 7.3 / 3.1, 3072 -> 768 7.0 / 6.5, 4096 -> 512 7.3 / 7.6, 8192 -> 4096
// 14.2 / 15.1; beyond: 17 tokens 4096 -> 11264 16.8 / 11.2, 64 tokens 8192 -> 6656 15.9 / 16.8, 7808 -> 10752 24.7 / 16.5.
static bool use_few_token_kernel(int M, int K, int ntok) {
    if (ntok <= 16) return true;
    if (ntok > 128) return false;
    if (M <= 44 * kBlockM) return K >= (850.0 + 4.0 * ntok + 0.11 * ntok * ntok) * (1.0 + M / 4000.0);
    return K >= 2 * M || (ntok <= 64 && K >= M);
}

static slope_status_t launch_sparse_tile(const SparseTile& t, const void* act, int ntok, const void* vals, const void* meta,
                                         int M, int K, const void* act2, const void* fac2, int r, bool a2_mn, void* out,
                                         int pairs, cudaStream_t stream, int pdl_mode) {
    return t.rows == 512 ? launch_sparse_quad(act, ntok, vals, meta, M, K, act2, fac2, r, a2_mn, out, t.width, pairs, stream,
                                              pdl_mode)
                         : launch_sparse_pair(act, ntok, vals, meta, M, K, act2, fac2, r, a2_mn, out, t.width, pairs, stream,
                                              pdl_mode);
}

// T = X L and the forward that adds T R.  How the adapter launch is cut decides how long it takes and how many SMs
// it keeps from the forward, so the two are planned together, whether they are launched as a fused pair
// or by separate calls (T is the same bits in both).  Behind the producer a forward takes
//   - at least T + 5.9 us (two launches, the adapter steps and the drain);
//   - or its own time + 2 us + the producer's share of the machine; and where pairs on the producer's SMs have as
//     many tiles as the others (the last CTAs of a launch start there, so a ragged last wave leaves
//     them out), most of T on top, unless the tiles are chosen for the SMs beside it.
// us, 4096 -> 4096, r = 64 at 500 / 1000 / 2048 tokens: T split in 2 / 2 / 1: 15.1 / 23.3 / 37.2, in 8: 17.4 / 27.0 /
// 39.7, although T alone is fastest in 8.
struct FwdAdapterPlan {
    AdapterPlan T;
    SparseTile tile;
    int pairs;                    // CTA pairs of the forward
};
static FwdAdapterPlan plan_fwd_adapter(int b, int d_out, int d_in, int r, const DeviceInfo& info) {
    const AdapterShape shape = adapter_T_shape(b, d_in, r);
    constexpr double kClkPerUs = 1850.0;
    FwdAdapterPlan best{};                                  // (no tile rows: the few-token kernel)
    best.pairs = info.sm_count / 2;
    double best_us = 1e300, cost = 0.0;
    if (use_few_token_kernel(d_out, d_in, b)) {                // its K-split is chosen around the producer
        best.T = adapter_plan(shape, info.sm_count);
    } else {
        const int pairs = info.sm_count / 2;
        const SparseTile full = choose_sparse_tile(d_out, d_in, b, r, pairs, &cost);
        const double full_us = cost / kClkPerUs;
        const int last_wave = ((d_out + full.rows - 1) / full.rows) * ((b + full.width - 1) / full.width) % pairs;
        adapter_cuts(shape, [&](int n_tile, int splits) {
            const AdapterPlan c = adapter_beside_forward(shape, n_tile, splits, info.sm_count);
            const int sms = adapter_sms(c, b, r, info.sm_count), beside = (info.sm_count - sms) / 2;
            const double share = static_cast<double>(sms) / info.sm_count;
            const bool blocked = last_wave == 0 || last_wave > beside;
            const double late = std::max(share * c.us, blocked ? (0.6 + 0.4 * share) * c.us : 0.0);
            const double us = std::max(c.us + 5.9, full_us + 2.0 + late);
            if (us < best_us) {
                best_us = us;
                best = FwdAdapterPlan{c, full, pairs};
            }
            if (!blocked || beside < pairs / 2) return;
            const SparseTile t = choose_sparse_tile(d_out, d_in, b, r, beside, &cost);
            const double us_beside = std::max(c.us + 5.9, cost / kClkPerUs + 2.0 + share * c.us);
            if (us_beside < best_us) {
                best_us = us_beside;
                best = FwdAdapterPlan{c, t, beside};
            }
        });
    }
    return best;
}
static FwdAdapterPlan fwd_adapter_plan(int b, int d_out, int d_in, int r, const DeviceInfo& info) {
    thread_local SizeMemo<FwdAdapterPlan> memo;
    return memo.get({b, d_out, d_in, r, info.dev, 0}, [&] { return plan_fwd_adapter(b, d_out, d_in, r, info); });
}

// What the T launch in front of a few-token forward asks L2 for: the first k-blocks of weights of at least 40 MB that are tall enough
// to occupy the SMs without a split, at up to 16 tokens.  Launching the further CTAs costs the pair up to 0.5 us, which a
// shorter or a split stream does not give back.  us without / with it, r = 64, 8 tokens: 4096 -> 22016 21.1 / 19.7, 5120 -> 35840
// 34.45 / 33.6, 4096 -> 16384 16.1 / 15.55, 2304 -> 16384 11.52 / 11.52; on the other side of the line 4096 -> 12288 13.93 / 14.04,
// 11008 -> 4096 13.53 / 13.55, and the four linears of a block of width 2048 / 6400 32.3 / 33.1, 1280 / 4096 27.4 / 29.5.
// The bytes it asks for hold up T itself.  A T of few SMs is in nobody's way; a T of wide ranks (32 SMs at r = 256) is when the forward has
// more CTAs than find room beside it: at r = 256 with 1.5 CTAs per SM and fewer 1 token 3584 -> 19200 19.0 / 17.7, 4096 -> 24576
// 23.7 / 22.5, 8 tokens 5120 -> 27648 29.6 / 29.1, with more of them 16 tokens 5120 -> 32768 35.1 / 35.2, 1 token 5120 -> 40960
// 47.6 / 48.6 (r = 64: 47.0 / 44.75), the four linears of a block of width 5120 / 17920 101.9 / 102.2 (r = 64: 82.7 / 81.5).
constexpr double kPairPrefetchFrom = 40e6;
constexpr int kPairPrefetchRows = 16384;
static WeightPrefetch pair_prefetch(const FwdAdapterPlan& plan, int ntok, const void* vals, const void* meta, int M, int K, int r,
                                    const DeviceInfo& info) {
    if (plan.tile.rows != 0 || ntok > 16 || M < kPairPrefetchRows || 1.125 * M * K < kPairPrefetchFrom) return WeightPrefetch{};
    const int splits = with_skinny_variant(ntok, M, K, info, [&](auto n, auto a, auto b) {
        return skinny_split_count<n(), a(), b()>(ntok, M, K, r, info, 2);
    });
    if (splits == 0) return WeightPrefetch{};
    const int slices = M / kBlockM * splits, T_sms = adapter_sms(plan.T, ntok, r, info.sm_count);
    if (8 * T_sms > info.sm_count && 2 * slices > 3 * info.sm_count) return WeightPrefetch{};
    const int free_sms = cluster_sms(plan.T.splits, info.sm_count) - T_sms;
    const int blocks = std::max(std::min(slices, free_sms), 0) / plan.T.splits * plan.T.splits;
    return WeightPrefetch{static_cast<const uint8_t*>(vals), static_cast<const uint8_t*>(meta), K, splits, slices, blocks};
}

// T[b x r] = X[b x d_in] * L[d_in x r]   (A = X, K contiguous; B = L^T stored [K x N])
static slope_status_t launch_adapter_T(const FwdAdapterPlan& plan, const void* X, const void* L, int b, int d_in, int r,
                                       void* T, cudaStream_t stream, int pdl_mode, const WeightPrefetch& next = WeightPrefetch{}) {
    return launch_adapter_planned<false, true>(plan.T, AdapterOperands{X, L, T, b, 0}, AdapterOperands{}, r, d_in, stream,
                                               pdl_mode, next);
}

static slope_status_t launch_sparse_gemm(const void* act, int ntok, const void* vals, const void* meta, int M, int K,
                                         const void* act2, const void* fac2, int r, bool a2_mn, void* out,
                                         cudaStream_t stream, const DeviceInfo& info) {
    const int pairs = info.sm_count / 2;
    thread_local SizeMemo<SparseTile> memo;                  // (no rows: the few-token kernel)
    const SparseTile& t = memo.get({M, K, ntok, r, info.dev, 0}, [&] {
        return use_few_token_kernel(M, K, ntok) ? SparseTile{0, 0} : choose_sparse_tile(M, K, ntok, r, pairs);
    });
    if (t.rows == 0) return launch_skinny(act, ntok, vals, meta, M, K, act2, fac2, r, a2_mn, out, stream, info);
    return launch_sparse_tile(t, act, ntok, vals, meta, M, K, act2, fac2, r, a2_mn, out, pairs, stream, 0);
}

static int dense_stages(bool b_mn, int epi, int width) {
    int n = DensePairCfg::kMaxStages;
    while (n > 1 && DensePairCfg::smem_bytes(b_mn, epi, width, n) > 232448) --n;
    return n;
}
// Columns per tile of the dense CTA-pair kernel, by estimate.  Narrow tiles give a small matrix enough of them for the
// pairs; wide ones move fewer bytes per FLOP.  In SM clocks: a k-block of 64 takes its bytes at 70 per clock and its
// MMAs (2.36 per column, no fewer than 80 columns' worth), a tile no less than its drain, a launch one more drain
// and 47 per pair.  (192 columns of a [K x N] operand cost the bytes of 256 and are not taken.)  Fitted to a sweep over
// 12 layer shapes (512 ... 9728) and 64 ... 8192 tokens: 0.2 % slower on average than the best width, where 256 x 256
// throughout is 24 %.  us, 256 x 256 / chosen width: forward / input gradient of a dense layer 500 tokens 1024 x 1024
// 9.5 / 9.6 -> 4.9 / 5.6, 740 tokens 8320 -> 6400 forward 84 -> 68, 700 tokens 2048 -> 6144 input gradient 32.6 -> 21.1.
// The plain store's drain term is that of tiles that leave as TMA stores; with the direct stores' (24 per column) weight
// gradients took, before -> now, 256 tokens 4096 x 4096 12.8 -> 10.9, 700 tokens 2048 x 6144 18.2 -> 16.4.
static int choose_dense_width(int M, int N, int K, bool b_mn, bool masked, int num_pairs) {
    const int num_m = (M + 255) / 256, num_kb = (K + 63) / 64;
    int best = 256;
    double best_cost = 1e300;
    for (int width = 256; width >= 64; width -= 64) {
        if (b_mn && width == 192) continue;
        const int tiles = num_m * ((N + width - 1) / width), rem = tiles % num_pairs;
        const bool halves = b_mn && width == 256 && tiles > num_pairs && 2 * rem <= num_pairs;      // see pair_work
        const double waves = tiles / num_pairs + (rem == 0 ? 0.0 : halves ? 0.5 : 1.0);
        const double k_block = std::max(DensePairCfg::stage_bytes(b_mn, width) / 70.0, 2.36 * std::max(width, 80));
        const double drain = masked ? 850.0 + 11.8 * width : 780.0 + 12.0 * width;
        const double cost = waves * std::max(num_kb * k_block, drain) + drain + 47.0 * std::min(tiles, num_pairs);
        if (cost < best_cost) { best_cost = cost; best = width; }
    }
    return best;
}

// Whether a launch takes two tiles in turn, the weight gradient from alternating ends (see raster_tile; 256 x 256 tiles only: the fused
// weight and adapter gradients, which have no others, then add up the same sums in the same order).
static bool long_reduction(int M, int K, int width) {
    return K >= kLongFrom && width == 256 && M > 2 * kBlockM * (kLongTileRows - 1);
}

// D[M x N] on 128 x 128 tiles of single CTAs while they all run at once and the reduction is at most
// 2048 long (measured on both sides of either line: dense_gemm_kernel), else on the CTA-pair kernel; a dense layer with
// fewer than 64 such tiles has more CTAs of the pair kernel's 64-column tiles (256 tokens 512 x 512: 3.7 against 4.3 us).
template <bool A_MN, bool B_MN, int EPI>
static slope_status_t launch_dense(const void* A, const void* B, int M, int N, int K, void* out,
                                   const void* mask, cudaStream_t stream, const DeviceInfo& info) {
    const int max_pairs = info.sm_count / 2, small_tiles = ((M + kBlockM - 1) / kBlockM) * (N / 128);
    const bool small = small_tiles <= info.sm_count && K <= 2048 && (EPI == kEpiMasked || small_tiles >= 64);
    thread_local SizeMemo<int> memo;
    const int width = small ? 128 : memo.get({M, N, K, info.sm_count, 0, 0}, [&] {
        return choose_dense_width(M, N, K, B_MN, EPI == kEpiMasked, max_pairs);
    });
    CUtensorMap tmA, tmB;
    const bool okA = A_MN ? make_tmap(&tmA, A, K, M, 64, 64) : make_tmap(&tmA, A, M, K, dense_a_box(M), 64);
    const bool okB = B_MN ? make_tmap(&tmB, B, K, N, 64, 64) : make_tmap(&tmB, B, N, K, small ? 128 : width / 2, 64);
    if (!okA || !okB) return SLOPE_ERR_CUDA;
    if (small) {
        constexpr int kStages = 6;
        using Cfg = DenseCfg<kStages>;
        const DenseGemmParams p{M, N, K, width, kStages, out, static_cast<const uint8_t*>(mask)};
        auto kern = dense_gemm_kernel<A_MN, B_MN, EPI, kStages>;
        if (!set_smem(kern, Cfg::kSmemBytes)) return SLOPE_ERR_CUDA;
        return launch_cluster_ex(kern, small_tiles, 1, kDenseThreads, Cfg::kSmemBytes, /*overlap_prologue=*/true, stream, tmA,
                                 tmB, p);
    }
    using Cfg = DensePairCfg;
    CUtensorMap tmO = tmA;
    if (EPI == kEpiStore && !make_tmap_out(&tmO, out, M, N, 32, 32)) return SLOPE_ERR_CUDA;
    const int stages = dense_stages(B_MN, EPI, width);
    const DenseGemmParams p{M, N, K, width, stages, out, static_cast<const uint8_t*>(mask)};
    auto kern = long_reduction(M, K, width) ? dense_gemm_pair_kernel<A_MN, B_MN, EPI, true> : dense_gemm_pair_kernel<A_MN, B_MN, EPI, false>;
    if (!set_smem(kern, 232448)) return SLOPE_ERR_CUDA;
    const int tiles = ((M + 2 * kBlockM - 1) / (2 * kBlockM)) * ((N + width - 1) / width);
    const int pairs = std::min(tiles, max_pairs);
    return launch_pairs(kern, 2 * pairs, kDenseThreads, Cfg::smem_bytes(B_MN, EPI, width, stages), stream, tmA, tmB,
                        tmO, p);
}

static int adapter_splits(int b, int rows) {
    // K-splits of the token reduction for the skinny adapter gradients (rows x r outputs).
    // rounds(s) = ceil(tiles * s / SMs) passes over the machine, each 1/s of a tile long; take
    // the s that minimises rounds(s) / s (with a small charge per split for the fp32 partials),
    // keeping at least 4 k-blocks (256 tokens) per split and no split without a k-block.
    // The split count sizes the caller's workspace (slope_adapter_workspace_bytes, which is asked
    // with no device at hand), so it is a function of the shape alone: the SM count is the B200's.
    constexpr int kSms = 148;
    const int tiles = (rows + kBlockM - 1) / kBlockM;
    const int num_kb = (b + 63) / 64;
    int best_s = 1;
    double best_cost = 1e30;
    for (int s = 1; s <= 16 && s * 4 <= num_kb; ++s) {
        const int rounds = (tiles * s + kSms - 1) / kSms;
        const double cost = static_cast<double>(rounds) / s + 0.004 * s;
        if (cost < best_cost - 1e-12) { best_cost = cost; best_s = s; }
    }
    const int per = (num_kb + best_s - 1) / best_s;
    return (num_kb + per - 1) / per;
}

static bool dims_ok(int d_out, int d_in) {
    return d_out > 0 && d_in > 0 && d_out % 128 == 0 && d_in % 128 == 0;
}
static bool rank_ok(int r) { return r >= 0 && r <= 256 && r % 16 == 0; }

}  // namespace slope

using namespace slope;

extern "C" {

size_t slope_values_bytes(int rows, int cols) { return static_cast<size_t>(rows) * cols; }
size_t slope_meta_bytes(int rows, int cols) { return static_cast<size_t>(rows) * cols / 8; }
size_t slope_mask_bytes(int rows, int cols) { return static_cast<size_t>(rows) * cols / 8; }

unsigned long long slope_launch_count(void) { return g_launches.load(); }

const char* slope_status_string(slope_status_t s) {
    switch (s) {
        case SLOPE_OK: return "ok";
        case SLOPE_ERR_INVALID_ARG: return "invalid argument";
        case SLOPE_ERR_SHAPE: return "unsupported shape";
        case SLOPE_ERR_ALIGNMENT: return "pointer not 16-byte aligned";
        case SLOPE_ERR_UNSUPPORTED_ARCH: return "device is not sm_100";
        case SLOPE_ERR_CUDA: return "CUDA call failed";
        case SLOPE_ERR_TIMEOUT: return "device-side wait timed out";
    }
    return "unknown status";
}

slope_status_t slope_kernel_clock_mhz(int kind, void* stream, double* mhz_host) {
    if ((kind != 0 && kind != 1) || !mhz_host) return SLOPE_ERR_INVALID_ARG;
    if (cudaStreamSynchronize(static_cast<cudaStream_t>(stream)) != cudaSuccess) return SLOPE_ERR_CUDA;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SLOPE_ERR_CUDA;
    unsigned long long v[2][2];
    if (cudaMemcpyFromSymbol(v, g_kernel_clock, sizeof(v)) != cudaSuccess) return SLOPE_ERR_CUDA;
    // totals at the previous call, per device and kind
    static std::mutex mu;
    static unsigned long long seen[64][2][2] = {};
    std::lock_guard<std::mutex> lock(mu);
    const unsigned long long cycles = v[kind][0] - seen[dev][kind][0], ns = v[kind][1] - seen[dev][kind][1];
    seen[dev][kind][0] = v[kind][0];
    seen[dev][kind][1] = v[kind][1];
    *mhz_host = ns ? static_cast<double>(cycles) / static_cast<double>(ns) * 1e3 : 0.0;
    return SLOPE_OK;
}

slope_status_t slope_poll_status(void* stream) {
    if (cudaStreamSynchronize(static_cast<cudaStream_t>(stream)) != cudaSuccess) return SLOPE_ERR_CUDA;
    int st = 0;
    if (cudaMemcpyFromSymbol(&st, g_device_status, sizeof(int)) != cudaSuccess) return SLOPE_ERR_CUDA;
    if (st != 0) {
        const int zero = 0;
        if (cudaMemcpyToSymbol(g_device_status, &zero, sizeof(int)) != cudaSuccess) return SLOPE_ERR_CUDA;
    }
    return static_cast<slope_status_t>(st);
}

slope_status_t slope_prune_24(const void* W, int d_out, int d_in, void* Wc_vals, void* Wc_meta, void* mask1_bits,
                              void* stream) {
    if (!W || !Wc_vals || !Wc_meta) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(d_out, d_in)) return SLOPE_ERR_SHAPE;
    if (!aligned16(W) || !aligned16(Wc_vals) || !aligned16(Wc_meta) || !aligned16(mask1_bits)) return SLOPE_ERR_ALIGNMENT;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    dim3 grid(d_in / 128, d_out / 128);
    return launch_stream(prune24_kernel, grid, static_cast<cudaStream_t>(stream),
        static_cast<const uint4*>(W), d_out, d_in, static_cast<uint4*>(Wc_vals), static_cast<uint4*>(Wc_meta),
        static_cast<uint4*>(mask1_bits));
}

slope_status_t slope_double_prune(const void* W, const void* mask1_bits, int d_out, int d_in, void* WTc_vals,
                                  void* WTc_meta, void* mask2_bits, void* stream) {
    if (!W || !mask1_bits || !WTc_vals || !WTc_meta) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(d_out, d_in)) return SLOPE_ERR_SHAPE;
    if (!aligned16(W) || !aligned16(mask1_bits) || !aligned16(WTc_vals) || !aligned16(WTc_meta) ||
        !aligned16(mask2_bits))
        return SLOPE_ERR_ALIGNMENT;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    dim3 grid(d_in / 128, d_out / 128);
    return launch_stream(double_prune_kernel, grid, static_cast<cudaStream_t>(stream),
        static_cast<const uint4*>(W), static_cast<const uint8_t*>(mask1_bits), d_out, d_in,
        static_cast<uint4*>(WTc_vals), static_cast<uint4*>(WTc_meta), static_cast<uint8_t*>(mask2_bits));
}

slope_status_t slope_prune_24_double(const void* W, int d_out, int d_in, void* Wc_vals, void* Wc_meta,
                                     void* mask1_bits, void* WTc_vals, void* WTc_meta, void* mask2_bits, void* stream) {
    if (!W || !Wc_vals || !Wc_meta || !WTc_vals || !WTc_meta) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(d_out, d_in)) return SLOPE_ERR_SHAPE;
    if (!aligned16(W) || !aligned16(Wc_vals) || !aligned16(Wc_meta) || !aligned16(mask1_bits) || !aligned16(WTc_vals) ||
        !aligned16(WTc_meta) || !aligned16(mask2_bits))
        return SLOPE_ERR_ALIGNMENT;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    dim3 grid(d_in / 128, d_out / 128);
    return launch_stream(prune24_double_kernel, grid, static_cast<cudaStream_t>(stream),
        static_cast<const uint4*>(W), d_out, d_in, static_cast<uint2*>(Wc_vals), static_cast<uint4*>(Wc_meta),
        static_cast<uint4*>(mask1_bits), static_cast<uint4*>(WTc_vals), static_cast<uint4*>(WTc_meta),
        static_cast<uint8_t*>(mask2_bits));
}

slope_status_t slope_linear_fwd(const void* X, int b, const void* Wc_vals, const void* Wc_meta, int d_out, int d_in,
                                const void* T, const void* R, int r, void* Y, void* stream) {
    if (!X || !Wc_vals || !Wc_meta || !Y) return SLOPE_ERR_INVALID_ARG;
    if (r != 0 && (!T || !R)) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(d_out, d_in) || b < 1 || !rank_ok(r)) return SLOPE_ERR_SHAPE;
    if (!aligned16(X) || !aligned16(Wc_vals) || !aligned16(Wc_meta) || !aligned16(Y) ||
        (r != 0 && (!aligned16(T) || !aligned16(R))))
        return SLOPE_ERR_ALIGNMENT;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    return launch_sparse_gemm(X, b, Wc_vals, Wc_meta, d_out, d_in, T, R, r, /*a2_mn=*/true, Y,
                              static_cast<cudaStream_t>(stream), info);
}

slope_status_t slope_linear_fwd_adapter(const void* X, int b, const void* Wc_vals, const void* Wc_meta, int d_out,
                                        int d_in, const void* L, const void* R, int r, void* T, void* Y,
                                        void* stream_) {
    if (!X || !Wc_vals || !Wc_meta || !L || !R || !T || !Y) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(d_out, d_in) || b < 1 || !rank_ok(r) || r == 0) return SLOPE_ERR_SHAPE;
    if (!aligned16(X) || !aligned16(Wc_vals) || !aligned16(Wc_meta) || !aligned16(L) || !aligned16(R) ||
        !aligned16(T) || !aligned16(Y))
        return SLOPE_ERR_ALIGNMENT;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const FwdAdapterPlan plan = fwd_adapter_plan(b, d_out, d_in, r, info);
    const WeightPrefetch next = pair_prefetch(plan, b, Wc_vals, Wc_meta, d_out, d_in, r, info);
    if (slope_status_t st = launch_adapter_T(plan, X, L, b, d_in, r, T, stream, 1, next)) return st;
    if (plan.tile.rows == 0) {
        // Two launches of the few-token kernel as a fused pair: T = X L releases its dependent only
        // once everything before it in the stream is complete, so the forward streams its weights
        // and runs its sparse reduction while T is still being computed, and waits only for T.
        return launch_skinny(X, b, Wc_vals, Wc_meta, d_out, d_in, T, R, r, true, Y, stream, info, 2);
    }
    // More tokens: the tile kernels are the consumer of such a pair in the same way.
    return launch_sparse_tile(plan.tile, X, b, Wc_vals, Wc_meta, d_out, d_in, T, R, r, /*a2_mn=*/true, Y, plan.pairs, stream, 2);
}

slope_status_t slope_linear_bwd_dx(const void* dY, int b, const void* WTc_vals, const void* WTc_meta, int d_out,
                                   int d_in, const void* dT, const void* L, int r, void* dX, void* stream) {
    if (!dY || !WTc_vals || !WTc_meta || !dX) return SLOPE_ERR_INVALID_ARG;
    if (r != 0 && (!dT || !L)) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(d_out, d_in) || b < 1 || !rank_ok(r)) return SLOPE_ERR_SHAPE;
    if (!aligned16(dY) || !aligned16(WTc_vals) || !aligned16(WTc_meta) || !aligned16(dX) ||
        (r != 0 && (!aligned16(dT) || !aligned16(L))))
        return SLOPE_ERR_ALIGNMENT;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    return launch_sparse_gemm(dY, b, WTc_vals, WTc_meta, d_in, d_out, dT, L, r, /*a2_mn=*/false, dX,
                              static_cast<cudaStream_t>(stream), info);
}

slope_status_t slope_linear_bwd_dw_masked(const void* dY, const void* X, int b, int d_out, int d_in,
                                          const void* mask1_bits, void* dWc_vals, void* stream) {
    if (!dY || !X || !mask1_bits || !dWc_vals) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(d_out, d_in) || b < 1) return SLOPE_ERR_SHAPE;
    if (!aligned16(dY) || !aligned16(X) || !aligned16(mask1_bits) || !aligned16(dWc_vals)) return SLOPE_ERR_ALIGNMENT;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    return launch_dense<true, true, kEpiMasked>(dY, X, d_out, d_in, b, dWc_vals, mask1_bits,
                                                     static_cast<cudaStream_t>(stream), info);
}

// ------------------------------------------------------------------ dense layer on the same pipeline
static slope_status_t dense_args(const void* a, const void* b_, const void* c, int b, int d_out, int d_in) {
    if (!a || !b_ || !c) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(d_out, d_in) || b < 1) return SLOPE_ERR_SHAPE;
    if (!aligned16(a) || !aligned16(b_) || !aligned16(c)) return SLOPE_ERR_ALIGNMENT;
    return SLOPE_OK;
}

slope_status_t slope_dense_linear_fwd(const void* X, int b, const void* W, int d_out, int d_in, void* Y, void* stream) {
    if (slope_status_t st = dense_args(X, W, Y, b, d_out, d_in)) return st;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    // Y[b x d_out] = X[b x d_in] * W[d_out x d_in]^T: both operands K-contiguous
    return launch_dense<false, false, kEpiStore>(X, W, b, d_out, d_in, Y, nullptr,
                                                              static_cast<cudaStream_t>(stream), info);
}

slope_status_t slope_dense_linear_bwd_dx(const void* dY, int b, const void* W, int d_out, int d_in, void* dX,
                                         void* stream) {
    if (slope_status_t st = dense_args(dY, W, dX, b, d_out, d_in)) return st;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    // dX[b x d_in] = dY[b x d_out] * W[d_out x d_in]: W is the [K x N] operand
    return launch_dense<false, true, kEpiStore>(dY, W, b, d_in, d_out, dX, nullptr,
                                                             static_cast<cudaStream_t>(stream), info);
}

slope_status_t slope_dense_linear_bwd_dw(const void* dY, const void* X, int b, int d_out, int d_in, void* dW,
                                         void* stream) {
    if (slope_status_t st = dense_args(dY, X, dW, b, d_out, d_in)) return st;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    // dW[d_out x d_in] = dY[b x d_out]^T * X[b x d_in]: both operands stored [K x .]
    return launch_dense<true, true, kEpiStore>(dY, X, d_out, d_in, b, dW, nullptr,
                                                            static_cast<cudaStream_t>(stream), info);
}

static size_t adapter_partial_bytes(int b, int rows, int r) {
    return ((static_cast<size_t>(adapter_splits(b, rows)) * rows * r * sizeof(float)) + 255) & ~size_t(255);
}

size_t slope_adapter_workspace_bytes(int b, int d_out, int d_in, int r) {
    if (b <= 0 || d_out <= 0 || d_in <= 0 || r <= 0) return 0;
    return adapter_partial_bytes(b, d_in, r) + adapter_partial_bytes(b, d_out, r);     // dL and dR partial sums
}

static bool overlap(const void* a, size_t a_bytes, const void* b, size_t b_bytes) {
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return b != nullptr && x < y + b_bytes && y < x + a_bytes;
}

// dR = T^T dY and dL = X^T dT: in one launch behind the dT launch, which reads R (`behind_dT`), or in two that are cut each by
// itself.  CTAs store their shares of the gradients while others still read, so gradients that overlap what is being read
// are formed in the workspace and copied into place.
static slope_status_t launch_adapter_grads(const void* X, const void* dY, const void* R, const void* T, const void* dT, int b,
                                           int d_out, int d_in, int r, void* dL, void* dR, void* workspace,
                                           cudaStream_t stream, const DeviceInfo& info, bool behind_dT) {
    const size_t unit = sizeof(uint16_t), rows = b, l_bytes = unit * d_in * r, r_bytes = unit * d_out * r;
    const auto among_operands = [&](const void* g, size_t bytes) {
        return overlap(g, bytes, X, unit * rows * d_in) || overlap(g, bytes, dY, unit * rows * d_out) ||
               overlap(g, bytes, T, unit * rows * r) || overlap(g, bytes, dT, unit * rows * r) || overlap(g, bytes, R, r_bytes);
    };
    const bool staged = among_operands(dL, l_bytes) || among_operands(dR, r_bytes);
    void* to_l = staged ? workspace : dL;
    void* to_r = staged ? static_cast<uint8_t*>(workspace) + adapter_partial_bytes(b, d_in, r) : dR;
    const AdapterOperands qr = adapter_dR(dY, T, d_out, to_r), ql = adapter_dL(X, dT, d_in, to_l);
    if (slope_status_t st = behind_dT ? launch_adapter<true, true>(qr, ql, r, b, stream, info, 2)
                                      : launch_adapter<true, true>(qr, AdapterOperands{}, r, b, stream, info))
        return st;
    if (!behind_dT)
        if (slope_status_t st = launch_adapter<true, true>(ql, AdapterOperands{}, r, b, stream, info)) return st;
    if (staged && (cudaMemcpyAsync(dL, to_l, l_bytes, cudaMemcpyDeviceToDevice, stream) != cudaSuccess ||
                   cudaMemcpyAsync(dR, to_r, r_bytes, cudaMemcpyDeviceToDevice, stream) != cudaSuccess))
        return SLOPE_ERR_CUDA;
    return SLOPE_OK;
}

slope_status_t slope_adapter_fwd_bwd(int phase, const void* X, const void* dY, const void* L, const void* R, int b,
                                     int d_out, int d_in, int r, void* T, void* dT, void* dL, void* dR,
                                     void* workspace, size_t workspace_bytes, void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (phase < 0 || phase > 2) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(d_out, d_in) || b < 1 || !rank_ok(r) || r == 0) return SLOPE_ERR_SHAPE;
    DeviceInfo info;
    if (phase == 0) {
        if (!X || !L || !T) return SLOPE_ERR_INVALID_ARG;
        if (!aligned16(X) || !aligned16(L) || !aligned16(T)) return SLOPE_ERR_ALIGNMENT;
        if (slope_status_t st = check_arch(info)) return st;
        return launch_adapter_T(fwd_adapter_plan(b, d_out, d_in, r, info), X, L, b, d_in, r, T, stream, 0);
    }
    if (phase == 2) {
        if (!dY || !R || !dT) return SLOPE_ERR_INVALID_ARG;
        if (!aligned16(dY) || !aligned16(R) || !aligned16(dT)) return SLOPE_ERR_ALIGNMENT;
        if (slope_status_t st = check_arch(info)) return st;
        return launch_adapter_dT(dY, R, b, d_out, r, dT, stream, info);
    }
    if (!X || !dY || !R || !T || !dT || !dL || !dR || !workspace) return SLOPE_ERR_INVALID_ARG;
    if (!aligned16(X) || !aligned16(dY) || !aligned16(R) || !aligned16(T) || !aligned16(dT) || !aligned16(dL) ||
        !aligned16(dR) || !aligned16(workspace))
        return SLOPE_ERR_ALIGNMENT;
    if (workspace_bytes < slope_adapter_workspace_bytes(b, d_out, d_in, r)) return SLOPE_ERR_INVALID_ARG;
    if (slope_status_t st = check_arch(info)) return st;
    // dR does not read dT: its CTAs run beside the dT launch, those of dL wait for it
    if (slope_status_t st = launch_adapter_dT(dY, R, b, d_out, r, dT, stream, info, 1)) return st;
    return launch_adapter_grads(X, dY, R, T, dT, b, d_out, d_in, r, dL, dR, workspace, stream, info, true);
}

// ------------------------------------------------------------------ masked dW with dL, dR riding along
namespace slope {
constexpr int kCarrySplits = 8;            // partial sums per row block of dR^T / dL in the fused launch

struct DwAdapterPlan {
    bool fused, alternate_k;      // alternate_k: tiles in the order of the weight gradient alone
    int splits_r, splits_l;
};

// The fused launch serves the shapes of the CTA-pair 256 x 256 weight-gradient kernel with r <= 128,
// provided no tile that carries adapter work lies among the halved items of the last wave (those run
// at half width, too narrow to serve as the A operand of the dL product).  Everything else takes the
// separate launches.
static DwAdapterPlan plan_dw_adapter(int b, int d_out, int d_in, int r, int sm_count) {
    DwAdapterPlan plan{false, false, 1, 1};
    const int num_m = (d_out + 255) / 256, num_n = (d_in + 255) / 256, num_kb = (b + 63) / 64;
    if (r > 128 || num_m * num_n * 2 <= sm_count) return plan;
    plan.splits_r = num_n < kCarrySplits ? num_n : kCarrySplits;
    plan.splits_l = num_m < kCarrySplits ? num_m : kCarrySplits;
    if (plan.splits_r > num_kb) plan.splits_r = num_kb;
    if (plan.splits_l > num_kb) plan.splits_l = num_kb;
    const int num_pairs = sm_count / 2, num_tiles = num_m * num_n;
    plan.alternate_k = long_reduction(d_out, b, choose_dense_width(d_out, d_in, b, true, true, num_pairs));
    const int full = (num_tiles / num_pairs) * num_pairs, rem = num_tiles - full;
    if (rem > 0 && 2 * rem <= num_pairs) {
        for (int tile = full; tile < num_tiles; ++tile) {
            int m, n, pos;
            raster_tile(tile, num_m, num_n, plan.alternate_k, m, n, pos);
            if (m < plan.splits_l || pos < plan.splits_r) return plan;
        }
    }
    plan.fused = true;
    return plan;
}
static DwAdapterPlan dw_adapter_plan(int b, int d_out, int d_in, int r, int sm_count) {
    thread_local SizeMemo<DwAdapterPlan> memo;
    return memo.get({b, d_out, d_in, r, sm_count, 0}, [&] { return plan_dw_adapter(b, d_out, d_in, r, sm_count); });
}

static size_t align256(size_t x) { return (x + 255) & ~size_t(255); }
}  // namespace slope

size_t slope_bwd_dw_adapter_workspace_bytes(int b, int d_out, int d_in, int r) {
    if (b <= 0 || d_out <= 0 || d_in <= 0 || r <= 0) return 0;
    const DwAdapterPlan plan = dw_adapter_plan(b, d_out, d_in, r, 148);
    const size_t fused = align256(static_cast<size_t>(plan.splits_r) * d_out * r * sizeof(float)) +
                         align256(static_cast<size_t>(plan.splits_l) * d_in * r * sizeof(float));
    const size_t separate = slope_adapter_workspace_bytes(b, d_out, d_in, r);
    return fused > separate ? fused : separate;
}

slope_status_t slope_linear_bwd_dw_adapter(const void* dY, const void* X, const void* T, const void* dT, int b,
                                           int d_out, int d_in, int r, const void* mask1_bits, void* dWc_vals,
                                           void* dL, void* dR, void* workspace, size_t workspace_bytes,
                                           void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!dY || !X || !T || !dT || !mask1_bits || !dWc_vals || !dL || !dR || !workspace) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(d_out, d_in) || b < 1 || !rank_ok(r) || r == 0) return SLOPE_ERR_SHAPE;
    if (!aligned16(dY) || !aligned16(X) || !aligned16(T) || !aligned16(dT) || !aligned16(mask1_bits) ||
        !aligned16(dWc_vals) || !aligned16(dL) || !aligned16(dR) || !aligned16(workspace))
        return SLOPE_ERR_ALIGNMENT;
    if (workspace_bytes < slope_bwd_dw_adapter_workspace_bytes(b, d_out, d_in, r)) return SLOPE_ERR_INVALID_ARG;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    const DwAdapterPlan plan = dw_adapter_plan(b, d_out, d_in, r, info.sm_count);
    if (!plan.fused || info.sm_count != 148) {
        // the separate launches: masked dW, dR, dL
        if (slope_status_t st = slope_linear_bwd_dw_masked(dY, X, b, d_out, d_in, mask1_bits, dWc_vals, stream_)) return st;
        return launch_adapter_grads(X, dY, nullptr, T, dT, b, d_out, d_in, r, dL, dR, workspace, stream, info, false);
    }
    using Cfg = DwAdapterCfg<6>;
    CUtensorMap tmA, tmB, tmT, tmDT;
    if (!make_tmap(&tmA, dY, b, d_out, 64, 64) || !make_tmap(&tmB, X, b, d_in, 64, 64) ||
        !make_tmap(&tmT, T, b, r, 64, 64) || !make_tmap(&tmDT, dT, b, r, 64, 64))
        return SLOPE_ERR_CUDA;
    DwAdapterParams p = {};
    p.M = d_out; p.N = d_in; p.K = b; p.r = r;
    p.splits_r = plan.splits_r; p.splits_l = plan.splits_l;
    p.alternate_k = plan.alternate_k;
    p.dWc = static_cast<uint16_t*>(dWc_vals);
    p.mask = static_cast<const uint8_t*>(mask1_bits);
    p.ws_r = static_cast<float*>(workspace);
    p.ws_l = reinterpret_cast<float*>(static_cast<uint8_t*>(workspace) +
                                      align256(static_cast<size_t>(plan.splits_r) * d_out * r * sizeof(float)));
    auto kern = dw_adapter_pair_kernel<6>;
    if (!set_smem(kern, Cfg::kSmemBytes)) return SLOPE_ERR_CUDA;
    const int tiles = ((d_out + 255) / 256) * ((d_in + 255) / 256);
    const int max_pairs = info.sm_count / 2;
    const int pairs = tiles < max_pairs ? tiles : max_pairs;
    if (slope_status_t st = launch_pairs(kern, 2 * pairs, Cfg::kThreads, Cfg::kSmemBytes, stream, tmA, tmB, tmT, tmDT, p))
        return st;
    const SplitKReduce rl{p.ws_l, static_cast<uint16_t*>(dL), d_in, r, plan.splits_l, 0};
    const SplitKReduce rr{p.ws_r, static_cast<uint16_t*>(dR), d_out, r, plan.splits_r, 1};
    splitk_reduce_kernel<<<info.sm_count * 4, 256, 0, stream>>>(rl, rr);
    return launch_result();
}

slope_status_t slope_sparse_add(const void* A_vals, const void* B_vals, float beta, float gamma, int rows, int cols,
                                void* out_vals, void* stream) {
    if (!A_vals || !B_vals || !out_vals) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(rows, cols)) return SLOPE_ERR_SHAPE;
    if (!aligned16(A_vals) || !aligned16(B_vals) || !aligned16(out_vals)) return SLOPE_ERR_ALIGNMENT;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    const size_t n_vec = static_cast<size_t>(rows) * cols / 2 / 8;
    return launch_stream(n_vec >= kKeepAddend ? sparse_add_kernel<true> : sparse_add_kernel<false>, dim3(stream_grid(n_vec, info)), static_cast<cudaStream_t>(stream),
                         static_cast<const uint4*>(A_vals), static_cast<const uint4*>(B_vals), beta, gamma, n_vec,
                         static_cast<uint4*>(out_vals));
}

slope_status_t slope_update_sparse_matrix(const void* Wc_vals, const void* mask1_bits, const void* WTc_meta,
                                          int d_out, int d_in, void* WTc_vals, void* stream) {
    if (!Wc_vals || !mask1_bits || !WTc_meta || !WTc_vals) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(d_out, d_in)) return SLOPE_ERR_SHAPE;
    // the kernel indexes its 8-byte and 16-byte units with 32 bits
    if (static_cast<unsigned long long>(d_out) * static_cast<unsigned long long>(d_in) >= (1ull << 35)) return SLOPE_ERR_SHAPE;
    if (!aligned16(Wc_vals) || !aligned16(mask1_bits) || !aligned16(WTc_meta) || !aligned16(WTc_vals))
        return SLOPE_ERR_ALIGNMENT;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    const int tiles = (d_in / 128) * (d_out / 128), slots = info.sm_count * kUpdateBlocksPerSm;
    return launch_stream(update_transposed_kernel, dim3(tiles < slots ? tiles : slots), static_cast<cudaStream_t>(stream),
                         static_cast<const uint2*>(Wc_vals), static_cast<const uint8_t*>(mask1_bits),
                         static_cast<const uint4*>(WTc_meta), d_out, d_in, static_cast<uint4*>(WTc_vals));
}

// ------------------------------------------------------------------ general N:M (masked dense)
static bool nm_ok(int n, int m) { return (m == 2 || m == 4 || m == 8 || m == 16) && n > 0 && n < m; }

slope_status_t slope_prune_nm(const void* W, int d_out, int d_in, int n, int m, void* W_R, void* mask1_bits,
                              void* stream_) {
    if (!W || !W_R) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(d_out, d_in) || !nm_ok(n, m)) return SLOPE_ERR_SHAPE;
    if (!aligned16(W) || !aligned16(W_R) || !aligned16(mask1_bits)) return SLOPE_ERR_ALIGNMENT;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const size_t chunks = static_cast<size_t>(d_out) * d_in / 16;
    const uint4* in = static_cast<const uint4*>(W);
    uint4* out = static_cast<uint4*>(W_R);
    uint16_t* mask = static_cast<uint16_t*>(mask1_bits);
    const dim3 grid(stream_grid(m == 16 ? chunks / 2 : chunks, info));
    auto kern = m == 2 ? prune_nm_kernel<2> : m == 4 ? prune_nm_kernel<4> : m == 8 ? prune_nm_kernel<8> : prune_nm_kernel<16>;
    return launch_stream(kern, grid, stream, in, chunks, n, out, mask);
}

slope_status_t slope_double_prune_nm(const void* W, const void* mask1_bits, int d_out, int d_in, int n, int m,
                                     void* W_RC, void* mask2_bits, void* stream_) {
    if (!W || !mask1_bits || !W_RC) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(d_out, d_in) || !nm_ok(n, m)) return SLOPE_ERR_SHAPE;
    if (!aligned16(W) || !aligned16(W_RC) || !aligned16(mask1_bits) || !aligned16(mask2_bits))
        return SLOPE_ERR_ALIGNMENT;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const uint4* in = static_cast<const uint4*>(W);
    const uint8_t* m1 = static_cast<const uint8_t*>(mask1_bits);
    uint4* out = static_cast<uint4*>(W_RC);
    uint8_t* m2 = static_cast<uint8_t*>(mask2_bits);
    const dim3 grid(stream_grid(static_cast<size_t>(d_out / m) * (d_in / (m == 16 ? 4 : 8)), info));
    auto kern = m == 2 ? double_prune_nm_kernel<2> : m == 4 ? double_prune_nm_kernel<4>
                                                   : m == 8 ? double_prune_nm_kernel<8> : double_prune_nm_kernel<16>;
    return launch_stream(kern, grid, stream, in, m1, d_out, d_in, n, out, m2);
}

slope_status_t slope_apply_mask(const void* G, const void* mask_bits, int d_out, int d_in, void* out, void* stream) {
    if (!G || !mask_bits || !out) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(d_out, d_in)) return SLOPE_ERR_SHAPE;
    if (!aligned16(G) || !aligned16(mask_bits) || !aligned16(out)) return SLOPE_ERR_ALIGNMENT;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    const size_t chunks = static_cast<size_t>(d_out) * d_in / 16;
    return launch_stream(apply_mask_kernel, dim3(stream_grid(chunks, info)), static_cast<cudaStream_t>(stream),
                         static_cast<const uint4*>(G), static_cast<const uint16_t*>(mask_bits), chunks, static_cast<uint4*>(out));
}

slope_status_t slope_mask_difference(const void* mask_a, const void* mask_b, int rows, int cols, void* count_out,
                                     void* stream_) {
    if (!mask_a || !mask_b || !count_out) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(rows, cols)) return SLOPE_ERR_SHAPE;
    if (!aligned16(mask_a) || !aligned16(mask_b) || (reinterpret_cast<uintptr_t>(count_out) & 7u) != 0)
        return SLOPE_ERR_ALIGNMENT;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (cudaMemsetAsync(count_out, 0, sizeof(unsigned long long), stream) != cudaSuccess) return SLOPE_ERR_CUDA;
    const size_t n_vec = static_cast<size_t>(rows) * cols / 8 / 16;
    mask_difference_kernel<<<stream_grid(n_vec, info), 256, 0, stream>>>(
        static_cast<const uint4*>(mask_a), static_cast<const uint4*>(mask_b), n_vec,
        static_cast<unsigned long long*>(count_out));
    return launch_result();
}

slope_status_t slope_selftest_wait_timeout(unsigned int limit_us, void* gave_up_flag, void* stream) {
    if (!gave_up_flag || limit_us == 0 || limit_us > 100000) return SLOPE_ERR_INVALID_ARG;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    wait_timeout_probe_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(
        static_cast<unsigned long long>(limit_us) * 1000ull, static_cast<int*>(gave_up_flag));
    return launch_result();
}

slope_status_t slope_meta_to_canonical(const void* meta_hw, int rows, int cols, void* meta_canon, void* stream) {
    if (!meta_hw || !meta_canon) return SLOPE_ERR_INVALID_ARG;
    if (!dims_ok(rows, cols)) return SLOPE_ERR_SHAPE;
    if (!aligned16(meta_hw) || !aligned16(meta_canon)) return SLOPE_ERR_ALIGNMENT;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    meta_to_canonical_kernel<<<info.sm_count * 4, 256, 0, static_cast<cudaStream_t>(stream)>>>(
        static_cast<const uint16_t*>(meta_hw), rows, cols, static_cast<uint16_t*>(meta_canon));
    return launch_result();
}

}  // extern "C"

// ------------------------------------------------------------------ allocation-free adapter-gradient entry
// The adapter kernels reduce inside a cluster, so dL needs neither an allocation nor a workspace -- unless it is to take
// the place of X or dT: CTAs store their shares while others still read, so it is then formed in a fixed
// array of the library image and copied.  The sizes this call takes are those whose split-K partial sums
// would fit 16 MiB, as its contract says; a bf16 dL is at most half of that.
namespace slope {
constexpr size_t kDlLimitBytes = size_t(16) << 20;
static __device__ __align__(256) uint8_t g_dl_scratch[kDlLimitBytes / 2];
}  // namespace slope

extern "C" {

size_t slope_adapter_dl_noalloc_max_scratch_bytes(void) { return kDlLimitBytes; }

slope_status_t slope_adapter_dl_noalloc(const void* X, const void* dT, int b, int d_in, int r, void* dL,
                                        void* stream_) {
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    if (!X || !dT || !dL) return SLOPE_ERR_INVALID_ARG;
    if (d_in <= 0 || d_in % 128 != 0 || b < 1 || !rank_ok(r) || r == 0) return SLOPE_ERR_SHAPE;
    if (!aligned16(X) || !aligned16(dT) || !aligned16(dL)) return SLOPE_ERR_ALIGNMENT;
    const size_t need = static_cast<size_t>(adapter_splits(b, d_in)) * d_in * r * sizeof(float);
    if (need > kDlLimitBytes) return SLOPE_ERR_SHAPE;
    DeviceInfo info;
    if (slope_status_t st = check_arch(info)) return st;
    const size_t bytes = sizeof(uint16_t) * d_in * r, rows = b;
    const bool staged = overlap(dL, bytes, X, sizeof(uint16_t) * rows * d_in) || overlap(dL, bytes, dT, sizeof(uint16_t) * rows * r);
    void* out = dL;
    if (staged && cudaGetSymbolAddress(&out, g_dl_scratch) != cudaSuccess) return SLOPE_ERR_CUDA;
    if (slope_status_t st = launch_adapter<true, true>(adapter_dL(X, dT, d_in, out), AdapterOperands{}, r, b, stream, info)) return st;
    if (staged && cudaMemcpyAsync(dL, out, bytes, cudaMemcpyDeviceToDevice, stream) != cudaSuccess) return SLOPE_ERR_CUDA;
    return SLOPE_OK;
}

}  // extern "C"
