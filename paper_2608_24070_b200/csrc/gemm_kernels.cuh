// tcgen05 GEMM kernels for sm_100a.
//
// The big-tile kernels are persistent, all are warp-specialised: warp 0 feeds shared memory with TMA,
// warp 1 owns tensor memory and issues the MMAs (one elected thread), the remaining warps
// drain the fp32 accumulators from tensor memory, convert to bf16 and store.  Every mbarrier
// wait is bounded (ptx.cuh); a role that gives up sets a CTA-wide flag, all roles leave their
// loops, tensor memory is released and the kernel returns.
//
//   dense_gemm_kernel          1 CTA per 128 x 128 tile; the same products while they are small
//   dense_gemm_pair_kernel     CTA pair per tile of 256 rows x 64 ... 256 columns (cta_group::2), a
//                              half-empty last wave's tiles halved; dW (masked epilogue) and the dense
//                              layer (store epilogue)
//   sparse_gemm_pair_kernel    CTA pair per tile of 256 rows x 32 ... 224 tokens, tcgen05.mma.sp;
//                              forward / dX with short reductions or few tiles
//   sparse_gemm_quad_kernel    CTA pair per tile of 512 rows x 32 ... 224 tokens (two MMA sub-tiles per
//                              activation tile); forward / dX with long reductions
//   sparse_gemm_skinny_kernel  one CTA per 128-row weight slab and K-slice, cluster reduction
//                              through distributed shared memory; forward / dX with few
//                              tokens (inference, decode), not persistent
// The adapter's low-rank products have a kernel of their own (adapter_kernels.cuh).
#pragma once
#include "ptx.cuh"

namespace slope {

constexpr int kGemmThreads = 192;
constexpr int kBlockM = 128;

struct PipeState {
    int stage = 0;
    uint32_t phase = 0;
    __device__ __forceinline__ void advance(int nstages) {
        if (++stage == nstages) { stage = 0; phase ^= 1u; }
    }
};

// The same with the byte offset of the stage kept along (stage size and count are launch parameters).
struct RingState {
    int stage = 0;
    uint32_t phase = 0, off = 0;
    __device__ __forceinline__ void advance(int nstages, uint32_t stage_bytes) {
        off += stage_bytes;
        if (++stage == nstages) { stage = 0; off = 0; phase ^= 1u; }
    }
};

// Give in-flight bulk copies time to land before the CTA's shared memory goes away.
__device__ __forceinline__ void drain_after_abort() {
    const unsigned long long t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
}

// =====================================================================================
// Sparse GEMM:  O[Ntok x M] (bf16) = ( A_2:4[M x K] * B[Ntok x K]^T  (+ A2[M x r] * B2[Ntok x r]^T) )^T
//   A   compressed values [M x K/2] + tensor-core-order metadata   (sparse operand)
//   B   activations, K contiguous
//   A2  dense adapter factor on the weight side: either [M x r] (K contiguous) or [r x M]
//   B2  dense adapter activations [Ntok x r]
// Used for Eq. (sparse_forward) (M = d_out, K = d_in) and Eq. (sparse_backward_input)
// (M = d_in, K = d_out, A = double-pruned transposed copy); the adapter product of
// Eq. (concat) is accumulated into the same tensor-memory tile by extra dense MMAs.
// Only the A operand of tcgen05.mma.sp can be sparse, hence the accumulator holds the
// transposed output tile (lane = feature, column = token) and the epilogue transposes.
// =====================================================================================
struct SparseGemmParams {
    int M, K, Ntok, r;
    int a2_mn_major;              // 1: A2 is stored [r x M] (M contiguous)
    int width;                    // tile kernels: tokens per tile, a multiple of 32, at most kMaxTokenTile
    int num_n;                    // tile kernels: token tiles
    int stages;                   // tile kernels: pipeline stages that fit at that width
    int group_m;                  // 512-row-tile kernel: row tiles per raster group (0: all in one group)
    int pdl_mode;                 // 2: consumer of a fused pair of launches (see the few-token kernel)
    uint16_t* out;                // [Ntok x M]
};

// =====================================================================================
// Dense GEMM:  D[M x N] = A[M x K] * B[N x K]^T, bf16 in, fp32 accumulate.
//   A_MN / B_MN: the operand is stored with its M (resp. N) index contiguous, i.e. as
//   [K x M] (resp. [K x N]) row-major; otherwise K is contiguous.
// Epilogues:
//   kEpiStore    bf16 D, row-major, leading dimension N
//   kEpiMasked   Eq. (sparse_backward_weight) + Algorithm 1 "pruneAndCompress": keep, per
//                group of 4 columns, the two columns the first-pass mask selects; bf16
//                [M x N/2]
// =====================================================================================
constexpr int kEpiStore = 0, kEpiMasked = 1;

struct DenseGemmParams {
    int M, N, K;
    int width;                    // columns per tile: 64, 128, 192 or 256
    int stages;                   // pipeline stages that fit at that width
    void* out;
    const uint8_t* mask;          // kEpiMasked: [M x N/8]
};

// Rows of a K-contiguous A's box: no more than the matrix has (rows inside the matrix or not, an SM takes about one per two
// clocks; what the MMAs read behind the last one only reaches accumulator rows that are never stored).  us, 128 rows / as many as
// tokens: forward of 2 tokens 11392 -> 3840 57.8 / 28.8, of 8 tokens 640 -> 3456 6.1 / 4.4, input gradient of 10 tokens 6656 <- 2560 18.1 / 10.8.
__host__ __device__ constexpr int dense_a_box(int M) { return M < kBlockM ? M : kBlockM; }
__host__ __device__ constexpr int dense_a_bytes(bool a_mn, int M) { return 128 * (a_mn ? kBlockM : dense_a_box(M)); }

// 16 accumulator columns of a row -> the 8 that the mask keeps, in ascending order per group of 4.
__device__ __forceinline__ uint4 compress_16(const uint32_t (&v)[16], uint32_t mbits) {
    uint32_t w[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        // two of the four bits are set: the lower one is bit 0, 1 or 2, the higher one bit 3, 2 or 1
        const uint32_t e0 = v[4 * g], e1 = v[4 * g + 1], e2 = v[4 * g + 2], e3 = v[4 * g + 3];
        const uint32_t lo = mbits & (1u << (4 * g)) ? e0 : (mbits & (2u << (4 * g)) ? e1 : e2);
        const uint32_t hi = mbits & (8u << (4 * g)) ? e3 : (mbits & (4u << (4 * g)) ? e2 : e1);
        w[g] = pack_bf16x2(__uint_as_float(lo), __uint_as_float(hi));
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// Epilogue warps of the dense kernels: two per tensor-memory lane quadrant, each takes half of a tile's columns.
constexpr int kDenseEpiWarps = 8;
constexpr int kDenseThreads = 64 + 32 * kDenseEpiWarps;

// A row's mask bits of `cols` (32, 64 or 128) columns, fetched before the accumulator is ready: loaded where they are
// used, 16 columns at a time, every load put an L2 round trip into the drain.
__device__ __forceinline__ void load_mask_bits(const uint8_t* row, int cols, uint32_t (&mw)[4]) {
    if (cols == 128) {
        const uint4 v = ld_v4(row);
        mw[0] = v.x; mw[1] = v.y; mw[2] = v.z; mw[3] = v.w;
    } else if (cols == 64) {
        const uint2 v = ld_v2(row);
        mw[0] = v.x; mw[1] = v.y;
    } else {
        mw[0] = ld_u32(row);
    }
}

// Drains `cols` (32, 64 or 128) accumulator columns of this thread's row, up to 64 at a time, so that the tensor-memory loads share one
// wait.  With few tokens the drain, not the main loop, paces the kernel (double-buffered accumulators): four
// warps that took 16 columns at a time, a mask load and a wait each, needed ~9 us for a 256 x 256 tile; as
// it is, 4096 x 4096 with 300 tokens went from 43 to 13 us, 8320 -> 6400 with 740 from 141 to 58, 512 x 512
// with 256 from 7.8 to 3.0 (16384 tokens: unchanged).
template <int COLS, typename Store>
__device__ __forceinline__ void drain_block(uint32_t t_row, int first, Store store) {
    uint32_t v[COLS / 16][16];
#pragma unroll
    for (int k = 0; k < COLS / 16; ++k) tmem_ld_16(t_row + 16 * (first + k), v[k]);
    tmem_ld_wait();
#pragma unroll
    for (int k = 0; k < COLS / 16; ++k) store(first + k, v[k]);
}
template <typename Store>
__device__ __forceinline__ void drain_columns(uint32_t t_row, int cols, Store store) {
    if (cols >= 64) drain_block<64>(t_row, 0, store);
    if (cols == 128) drain_block<64>(t_row, 4, store);
    else if (cols == 32) drain_block<32>(t_row, 0, store);
}

// Writes `cols` drained accumulator columns of output row m from column n0 on, as bf16 (kEpiStore; rows past M take part
// in the warp-wide tensor-memory loads, but store nothing) or the half that the mask bits select (kEpiMasked).
template <int EPI>
__device__ __forceinline__ void drain_row(uint32_t t_row, int cols, const DenseGemmParams& p, int m, int n0, const uint32_t (&mw)[4]) {
    if (EPI == kEpiMasked) {
        uint4* dst = reinterpret_cast<uint4*>(static_cast<uint16_t*>(p.out) + static_cast<size_t>(m) * (p.N >> 1) + (n0 >> 1));
        drain_columns(t_row, cols, [&](int c, const uint32_t (&v)[16]) { dst[c] = compress_16(v, mw[c >> 1] >> (16 * (c & 1))); });
    } else {
        uint4* dst = reinterpret_cast<uint4*>(static_cast<uint16_t*>(p.out) + static_cast<size_t>(m) * p.N + n0);
        drain_columns(t_row, cols, [&](int c, const uint32_t (&v)[16]) {
            if (m >= p.M) return;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const uint32_t* e = v + 8 * k;
                dst[2 * c + k] = make_uint4(pack_bf16x2(__uint_as_float(e[0]), __uint_as_float(e[1])),
                                            pack_bf16x2(__uint_as_float(e[2]), __uint_as_float(e[3])),
                                            pack_bf16x2(__uint_as_float(e[4]), __uint_as_float(e[5])),
                                            pack_bf16x2(__uint_as_float(e[6]), __uint_as_float(e[7])));
            }
        });
    }
}

// Dense GEMM with one 128 x 128 tile per CTA, for products whose tiles all run at once and whose reduction is short: no
// cluster to launch and to synchronise.  us, against the best width of the CTA-pair kernel: masked weight
// gradient 512 x 512 with 256 tokens 3.1 / 3.5, 768 -> 2304 with 1000 tokens 6.0 / 6.9, 1024 -> 2048 with 2048 tokens
// 8.5 / 9.2; with 4096 tokens 16.0 / 15.3, as a CTA then pulls twice the pair's bytes per FLOP.
template <int STAGES>
struct DenseCfg {
    static constexpr int kBlockN = 128;
    static constexpr int kABytes = kBlockM * 128;                // 128 x 64 bf16
    static constexpr int kBBytes = kBlockN * 128;
    static constexpr int kStageBytes = kABytes + kBBytes;
    static constexpr int kSmemBytes = STAGES * kStageBytes + 256 + 1024;
};

template <bool A_MN, bool B_MN, int EPI, int STAGES>
__global__ void __launch_bounds__(kDenseThreads, 1)
dense_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                  const DenseGemmParams p) {
    // N is a multiple of 128; one tile per CTA
    using Cfg = DenseCfg<STAGES>;
    constexpr int kBlockN = Cfg::kBlockN;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + STAGES * Cfg::kStageBytes);
    uint64_t* empty_bar = full_bar + STAGES;
    uint64_t* tfull_bar = empty_bar + STAGES;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tfull_bar + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int num_m = (p.M + kBlockM - 1) / kBlockM, num_kb = (p.K + 63) / 64;
    const int m_blk = blockIdx.x % num_m, n_blk = blockIdx.x / num_m;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        mbar_init(tfull_bar, 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 2 && elect_one()) {
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, kBlockN);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    // Programmatic dependent launch: the set-up above may overlap the tail of the previous kernel in
    // the stream; no thread touches global memory before that kernel has completed.
    griddep_launch_dependents();
    griddep_wait();

    if (warp == 0) {
        if (elect_one()) {
            PipeState ps;
            for (int kb = 0; kb < num_kb; ++kb) {
                if (!mbar_wait(&empty_bar[ps.stage], ps.phase ^ 1u, abort_flag)) break;
                uint8_t* sA = smem + ps.stage * Cfg::kStageBytes;
                uint8_t* sB = sA + Cfg::kABytes;
                uint64_t* bar = &full_bar[ps.stage];
                mbar_expect_tx(bar, dense_a_bytes(A_MN, p.M) + Cfg::kBBytes);
                if (A_MN) {
                    tma_load_2d(sA, &tmA, bar, m_blk * kBlockM, kb * 64);
                    tma_load_2d(sA + 8192, &tmA, bar, m_blk * kBlockM + 64, kb * 64);
                } else {
                    tma_load_2d(sA, &tmA, bar, kb * 64, m_blk * kBlockM);
                }
                if (B_MN) {
                    tma_load_2d(sB, &tmB, bar, n_blk * kBlockN, kb * 64);
                    tma_load_2d(sB + 8192, &tmB, bar, n_blk * kBlockN + 64, kb * 64);
                } else {
                    tma_load_2d(sB, &tmB, bar, kb * 64, n_blk * kBlockN);
                }
                ps.advance(STAGES);
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            constexpr uint32_t idesc = make_idesc_bf16(kBlockM, kBlockN, A_MN, B_MN, false);
            PipeState ps;
            bool ok = true;
            ClockProbe probe;
            if (blockIdx.x == 0) probe.begin();
            for (int kb = 0; kb < num_kb; ++kb) {
                if (!mbar_wait(&full_bar[ps.stage], ps.phase, abort_flag)) { ok = false; break; }
                tc_fence_after_sync();
                const uint32_t sA = smem_u32(smem + ps.stage * Cfg::kStageBytes);
                const uint32_t sB = sA + Cfg::kABytes;
                const uint64_t a0 = A_MN ? make_smem_desc(sA, 8192, 1024, kSwizzle128B) : make_smem_desc(sA, 16, 1024, kSwizzle128B);
                const uint64_t b0 = B_MN ? make_smem_desc(sB, 8192, 1024, kSwizzle128B) : make_smem_desc(sB, 16, 1024, kSwizzle128B);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    umma_bf16(tmem_base, a0 + j * (A_MN ? 128 : 2), b0 + j * (B_MN ? 128 : 2), idesc, (kb | j) != 0 ? 1u : 0u);
                umma_commit(&empty_bar[ps.stage]);
                ps.advance(STAGES);
            }
            if (ok) umma_commit(tfull_bar);
            if (blockIdx.x == 0) probe.end(kClockDense);
        }
    } else {
        const int q = warp & 3, c0 = ((warp - 2) >> 2) * (kBlockN / 2);
        const int m = m_blk * kBlockM + q * 32 + lane, n0 = n_blk * kBlockN + c0;
        uint32_t mw[4];
        if (EPI == kEpiMasked) load_mask_bits(p.mask + static_cast<size_t>(m) * (p.N >> 3) + (n0 >> 3), kBlockN / 2, mw);
        if (mbar_wait(tfull_bar, 0u, abort_flag)) {
            tc_fence_after_sync();
            drain_row<EPI>(tmem_base + c0 + (static_cast<uint32_t>(q * 32) << 16), kBlockN / 2, p, m, n0, mw);
        }
    }

    __syncwarp();
    if (*abort_flag) drain_after_abort();
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, kBlockN);
    }
}

// Fixed-order reduction of K-split partial sums: out = bf16( sum_s ws[s][m][n] ), written
// row-major [M x N] or transposed [N x M].  Up to two reductions per launch (second.M == 0: one).
struct SplitKReduce {
    const float* ws;
    uint16_t* out;
    int M, N, splits, transpose;
};

// A block takes 32 consecutive rows at a time: 16-byte loads of the partial sums, summed in split
// order; the transposed output goes through a padded shared-memory tile so that both the reads
// and the 2-byte writes are contiguous.  N (the adapter rank) is a multiple of 16, at most 256.
__global__ void __launch_bounds__(256) splitk_reduce_kernel(const SplitKReduce r0, const SplitKReduce r1) {
    __shared__ float tile[32][257];
    const int units0 = (r0.M + 31) / 32, units1 = (r1.M + 31) / 32;
    for (int u = blockIdx.x; u < units0 + units1; u += gridDim.x) {
        const bool second = u >= units0;
        const SplitKReduce& r = second ? r1 : r0;
        const int m0 = 32 * (second ? u - units0 : u);
        const int rows = min(32, r.M - m0);
        const size_t total = static_cast<size_t>(r.M) * r.N;
        const float4* ws4 = reinterpret_cast<const float4*>(r.ws + static_cast<size_t>(m0) * r.N);
        const size_t split_stride4 = total / 4;
        const int chunks = rows * r.N / 4;
        for (int c = threadIdx.x; c < chunks; c += blockDim.x) {
            float4 acc = ws4[c];
            for (int s = 1; s < r.splits; ++s) {
                const float4 t = ws4[static_cast<size_t>(s) * split_stride4 + c];
                acc.x += t.x; acc.y += t.y; acc.z += t.z; acc.w += t.w;
            }
            if (r.transpose) {
                const int mm = (4 * c) / r.N, n = (4 * c) % r.N;
                tile[mm][n] = acc.x; tile[mm][n + 1] = acc.y; tile[mm][n + 2] = acc.z; tile[mm][n + 3] = acc.w;
            } else {
                uint2 o;
                o.x = pack_bf16x2(acc.x, acc.y);
                o.y = pack_bf16x2(acc.z, acc.w);
                *reinterpret_cast<uint2*>(r.out + static_cast<size_t>(m0) * r.N + 4 * static_cast<size_t>(c)) = o;
            }
        }
        if (r.transpose) {
            __syncthreads();
            for (int e = threadIdx.x; e < 32 * r.N; e += blockDim.x) {
                const int n = e >> 5, mm = e & 31;
                if (mm < rows) r.out[static_cast<size_t>(n) * r.M + m0 + mm] = to_bf16(tile[mm][n]);
            }
            __syncthreads();
        }
    }
}

// =====================================================================================
// CTA-pair versions (cluster of 2, tcgen05 cta_group::2).  One MMA spans both SMs: the pair
// owns a 256-row tile of the A operand (128 rows per CTA) and each CTA stages only HALF of
// the B tile, which halves the activation bytes every SM pulls from L2 per MMA and leaves
// room for twice as many pipeline stages.  The leader CTA (rank 0) issues all MMAs; both
// CTAs run their own TMA producer (completion bytes are counted on the leader's barrier)
// and their own epilogue (each drains its 128 accumulator rows).  tcgen05.commit arrives on
// the barriers of both CTAs; the epilogues release an accumulator stage by arriving on the
// leader's barrier through the cluster shared-memory window.
// =====================================================================================
// Tokens per tile of the sparse tile kernels.  The width is chosen per launch (any multiple of 32, the epilogue's
// block and the step of N for an MMA of 256 rows), so that the tiles of a token count come out equal
// and fill the waves of the machine; narrower tiles leave room for more pipeline stages.  224 is what
// tensor memory (two accumulators and the metadata columns) and shared memory (four, or three
// 512-row, stages) hold.  The last tile is only as wide as the tokens that are left, rounded up to 32:
// the MMAs run with that N, the second CTA's half starts at its middle, and the epilogue stops there.
constexpr int kMaxTokenTile = 224;
__device__ __forceinline__ int token_tile_width(int ntok, int n0, int tile_width) {
    const int left = ntok - n0;
    return left >= tile_width ? tile_width : ((left + 31) & ~31);
}

// An epilogue block of 32 features x 32 tokens: read from tensor memory as accumulator fragments and packed to bf16 pairs
// of adjacent tokens ...
__device__ __forceinline__ void load_packed_block(uint32_t t_addr, uint32_t (&block)[16]) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {                                // features 0..15 and 16..31
        uint32_t v[16];
        tmem_ld_16x256b_x4(t_addr + (static_cast<uint32_t>(16 * h) << 16), v);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 4; ++j) {                            // tokens 8j .. 8j + 7
            block[4 * j + 2 * h] = pack_bf16x2(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]));
            block[4 * j + 2 * h + 1] = pack_bf16x2(__uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3]));
        }
    }
}
// ... and written transposed, [token][32 features], by four stmatrix: 16-byte pieces XOR-swizzled as the store's tensor map
// expects (64-byte rows, piece index XOR bits 7..8 of the address).  lane -> (matrix = feature group of 8, row =
// token within a group of 8).
__device__ __forceinline__ void stage_packed_block(uint32_t buf, int lane, const uint32_t (&block)[16]) {
    const uint32_t row_addr = buf + (lane & 7) * 64 + (((lane >> 3) ^ ((lane >> 1) & 3)) << 4);
#pragma unroll
    for (int j = 0; j < 4; ++j)
        stmatrix_x4_trans(row_addr + j * 512, block[4 * j], block[4 * j + 1], block[4 * j + 2], block[4 * j + 3]);
}

constexpr int kMaxTileStages = 8;
struct SparsePairCfg {
    static constexpr int kABytes = kBlockM * 128;
    static constexpr int kEBytes = 2048;
    static constexpr int kStoreRows = 32;                         // tokens per TMA store
    static constexpr int kStoreCols = 32;                         // features per TMA store (one warp's lanes)
    static constexpr int kStoreBytes = kStoreRows * kStoreCols * 2;
    static constexpr int kEpiWarps = 8;                           // two warps per tensor-memory lane quadrant
    static constexpr int kThreads = 64 + 32 * kEpiWarps;
    static constexpr int kStagingBytes = kEpiWarps * 2 * kStoreBytes;
    static constexpr int kECol = 2 * kMaxTokenTile;
    __host__ __device__ static constexpr int b_bytes(int width) { return width * 128; }          // per CTA: width / 2 tokens x 128
    __host__ __device__ static constexpr int stage_bytes(int width) { return kABytes + b_bytes(width) + kEBytes; }
    __host__ __device__ static constexpr int smem_bytes(int width, int stages) {
        return stages * stage_bytes(width) + kStagingBytes + 256 + 1024;
    }
    static_assert(kMaxTokenTile % 32 == 0 && 2 * kMaxTokenTile + 8 <= 512, "tile does not fit tensor memory");
};

__global__ void __launch_bounds__(SparsePairCfg::kThreads, 1)
sparse_gemm_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                        const __grid_constant__ CUtensorMap tmE, const __grid_constant__ CUtensorMap tmA2,
                        const __grid_constant__ CUtensorMap tmB2, const __grid_constant__ CUtensorMap tmO,
                        const SparseGemmParams p) {
    using Cfg = SparsePairCfg;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int stages = p.stages, stage_bytes = Cfg::stage_bytes(p.width);
    const uint32_t b_half = p.width * 64;                    // bytes of one 64-column half of the activation tile
    uint8_t* staging = smem + stages * stage_bytes;
    uint64_t* full_bar = reinterpret_cast<uint64_t*>(staging + Cfg::kStagingBytes);
    uint64_t* empty_bar = full_bar + kMaxTileStages;
    uint64_t* tfull_bar = empty_bar + kMaxTileStages;
    uint64_t* tempty_bar = tfull_bar + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty_bar + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t cta = cluster_ctarank();                  // 0 = leader
    const int pair_id = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;
    const int num_mb = p.M / kBlockM;                        // 128-row blocks of A
    const int num_m = (num_mb + 1) / 2;                      // 256-row pair tiles
    const int num_n = p.num_n;
    const int num_tiles = num_m * num_n;
    const int num_kb = p.K / 128;
    const int num_ab = (p.r + 63) / 64;
    const int total_kb = num_kb + num_ab;

    if (threadIdx.x == 0) {
#pragma unroll
        for (int s = 0; s < kMaxTileStages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(&tfull_bar[a], 1); mbar_init(&tempty_bar[a], 2 * Cfg::kEpiWarps); }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 2 && elect_one()) {
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
        tma_prefetch_desc(&tmE);
    }
    if (warp == 1) {
        tmem_alloc_pair(tmem_slot, 512);
        tmem_relinquish_pair();
    }
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync_all();                                      // peer barriers are initialised
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    // Programmatic dependent launch: the set-up above may overlap the tail of the previous kernel in
    // the stream; no thread touches global memory before that kernel has completed.
    // (As the consumer of a fused pair of launches -- pdl_mode 2, see the few-token kernel -- only the
    // producer thread waits, right before its first load of the adapter operand T.)
    griddep_launch_dependents();
    if (p.pdl_mode != 2) griddep_wait();

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer (both CTAs)
        if (elect_one()) {
            const uint64_t keep = l2_policy_evict_last();
            RingState ps;
            bool ok = true;
            bool waited = false;
            for (int tile = pair_id; ok && tile < num_tiles; tile += num_pairs) {
                const int m_pair = tile % num_m, n_blk = tile / num_m;
                const int mb = m_pair * 2 + static_cast<int>(cta);           // this CTA's 128-row block
                const int mb_e = mb < num_mb ? mb : num_mb - 1;              // rows past M: any valid metadata block
                const int width = token_tile_width(p.Ntok, n_blk * p.width, p.width);
                const int n_row0 = n_blk * p.width + static_cast<int>(cta) * (width / 2);
                for (int kb = 0; kb < total_kb; ++kb) {
                    if (!mbar_wait(&empty_bar[ps.stage], ps.phase ^ 1u, abort_flag)) { ok = false; break; }
                    uint8_t* sA = smem + ps.off;
                    uint8_t* sB = sA + Cfg::kABytes;
                    uint8_t* sE = sB + 2 * b_half;
                    const uint32_t bar = mapa_shared(smem_u32(&full_bar[ps.stage]), 0);
                    if (kb < num_kb) {
                        if (cta == 0) mbar_expect_tx(&full_bar[ps.stage], 2 * stage_bytes);
                        tma_load_2d_pair_hint(sA, &tmA, bar, kb * 64, mb * kBlockM, keep);
                        tma_load_2d_pair(sB, &tmB, bar, kb * 128, n_row0);
                        tma_load_2d_pair(sB + b_half, &tmB, bar, kb * 128 + 64, n_row0);
                        tma_load_2d_pair_hint(sE, &tmE, bar, 0, mb_e * num_kb + kb, keep);
                    } else {
                        const int ab = kb - num_kb;
                        if (p.pdl_mode == 2 && !waited) {
                            griddep_wait();
                            waited = true;
                        }
                        if (cta == 0) mbar_expect_tx(&full_bar[ps.stage], 2 * (Cfg::kABytes + b_half));
                        if (p.a2_mn_major) {
                            tma_load_2d_pair(sA, &tmA2, bar, mb * kBlockM, ab * 64);
                            tma_load_2d_pair(sA + 8192, &tmA2, bar, mb * kBlockM + 64, ab * 64);
                        } else {
                            tma_load_2d_pair(sA, &tmA2, bar, ab * 64, mb * kBlockM);
                        }
                        tma_load_2d_pair(sB, &tmB2, bar, ab * 64, n_row0);
                    }
                    ps.advance(stages, stage_bytes);
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (leader CTA only)
        if (cta == 0 && elect_one()) {
            RingState ps;
            bool ok = true;
            int it = 0;
            ClockProbe probe;
            if (pair_id == 0) probe.begin();
            for (int tile = pair_id; ok && tile < num_tiles; tile += num_pairs, ++it) {
                const int width = token_tile_width(p.Ntok, (tile / num_m) * p.width, p.width);
                const uint32_t idesc_sp = make_idesc_bf16(2 * kBlockM, width, false, false, true);
                const uint32_t idesc_ad = make_idesc_bf16(2 * kBlockM, width, p.a2_mn_major != 0, false, false);
                const int acc = it & 1;
                const uint32_t acc_phase = static_cast<uint32_t>(it >> 1) & 1u;
                if (!mbar_wait(&tempty_bar[acc], acc_phase ^ 1u, abort_flag)) { ok = false; break; }
                tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + acc * kMaxTokenTile;
                for (int kb = 0; kb < total_kb; ++kb) {
                    if (!mbar_wait(&full_bar[ps.stage], ps.phase, abort_flag)) { ok = false; break; }
                    tc_fence_after_sync();
                    const uint32_t sA = smem_u32(smem + ps.off);
                    const uint32_t sB = sA + Cfg::kABytes;
                    const uint32_t sE = sB + 2 * b_half;
                    if (kb < num_kb) {
                        const uint32_t e_tmem = tmem_base + Cfg::kECol + (kb & 1) * 4;
                        tmem_cp_128x128b_pair(e_tmem, make_smem_desc(sE, 128, 128, kSwizzleNone));
                        // (a step along K adds to the start address, the descriptor's lowest field, in 16-byte units)
                        const uint64_t a0 = make_smem_desc(sA, 16, 1024, kSwizzle128B);
                        const uint64_t b0 = make_smem_desc(sB, 16, 1024, kSwizzle128B);
                        const uint64_t b2 = b0 + (b_half >> 4);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint64_t ad = a0 + 2 * j, bd = (j < 2 ? b0 : b2) + 4 * (j & 1);
                            umma_bf16_sp_pair(d_tmem, ad, bd, e_tmem + (j & 2), idesc_sp | (j & 1),
                                              (kb | j) != 0 ? 1u : 0u);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint64_t ad = p.a2_mn_major
                                                    ? make_smem_desc(sA + j * 2048, 8192, 1024, kSwizzle128B)
                                                    : make_smem_desc(sA + j * 32, 16, 1024, kSwizzle128B);
                            const uint64_t bd = make_smem_desc(sB + j * 32, 16, 1024, kSwizzle128B);
                            umma_bf16_pair(d_tmem, ad, bd, idesc_ad, 1u);
                        }
                    }
                    umma_commit_pair(&empty_bar[ps.stage], 3);
                    ps.advance(stages, stage_bytes);
                }
                if (ok) umma_commit_pair(&tfull_bar[acc], 3);
            }
            if (pair_id == 0) probe.end(kClockSparse);
        }
    } else {
        // ------------------------------------------------------------ epilogue (warps 2..9, both CTAs)
        // Warp w drains lane quadrant w%4; the two warps of a quadrant take alternate 32-token
        // blocks.  A block (32 features x 32 tokens) is read from tensor memory as accumulator
        // fragments, packed to bf16 pairs of adjacent tokens, and written transposed into the
        // warp's private staging buffer by four stmatrix instructions ([token][32 features],
        // 16-byte pieces XOR-swizzled as the store's tensor map expects); it leaves as a TMA store
        // of 32 tokens x 32 features, so no warp waits for another.
        const int q = warp & 3;
        const int ew = warp - 2;
        const int half = ew >> 2;
        uint8_t* my_buf = staging + ew * 2 * Cfg::kStoreBytes;
        const uint64_t stream_out = l2_policy_evict_first();
        bool ok = true;
        int it = 0;
        uint32_t buf = 0;
        for (int tile = pair_id; ok && tile < num_tiles; tile += num_pairs, ++it) {
            const int m_pair = tile % num_m, n_blk = tile / num_m;
            const int acc = it & 1;
            const uint32_t acc_phase = static_cast<uint32_t>(it >> 1) & 1u;
            if (!mbar_wait(&tfull_bar[acc], acc_phase, abort_flag)) { ok = false; break; }
            tc_fence_after_sync();
            const uint32_t t_row = tmem_base + acc * kMaxTokenTile + (static_cast<uint32_t>(q * 32) << 16);
            const int m0 = (m_pair * 2 + static_cast<int>(cta)) * kBlockM + q * 32;
            const int width = token_tile_width(p.Ntok, n_blk * p.width, p.width);
            // (rows past M are not staged either: the wait for a staging buffer counts stores)
#pragma unroll 1
            for (int c0 = half * Cfg::kStoreRows; m0 < p.M && c0 < width; c0 += 2 * Cfg::kStoreRows) {
                uint32_t block[16];
                load_packed_block(t_row + c0, block);
                // the staging buffer about to be overwritten must have been read by its TMA store
                if (lane == 0) tma_store_wait_read<1>();
                __syncwarp();
                stage_packed_block(smem_u32(my_buf + buf * Cfg::kStoreBytes), lane, block);
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    tma_store_2d_hint(&tmO, my_buf + buf * Cfg::kStoreBytes, m0, n_blk * p.width + c0, stream_out);
                    tma_store_commit();
                }
                buf ^= 1u;
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(mapa_shared(smem_u32(&tempty_bar[acc]), 0));
        }
        if (lane == 0) tma_store_wait_all<0>();
    }

    __syncwarp();
    if (*abort_flag) drain_after_abort();
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync_all();                                      // nobody signals or reads the peer after this
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc_pair(tmem_base, 512);
    }
}

// Tile order for GEMMs whose two operands are both streamed once per tile (dW: dY^T X with the
// tokens as reduction).  The ~74 tiles in flight should form a near-square patch of the output:
// a patch of gm x gn tiles reads (gm + gn) operand panels, a gm x 1 strip reads gm + 1 for 1/gn
// of the work.  Tiles are numbered in groups of kRasterGroupM tile rows, column by column.
//
// These GEMMs run at the power cap, where a byte from HBM costs what some 150 FLOP do, so what a wave can take from L2
// instead is time.  A wave's panels (17 x 256 x K) are more than L2 keeps from some 5500 steps of the reduction on.  From there,
// and with at least seven tile rows,
//   - a pair works on two tiles at a time, kInterleaveBlocks k-blocks of one, then of the other (it has two accumulators
//     anyway): the patch in flight is twice as large and reads a fifth fewer panels per tile, and each accumulator is
//     drained while the other one's k-blocks run;
//   - every other two tiles of a pair take the k-blocks from the end, where the reduction runs over tokens: the last part of a
//     wave's panels is still there when the next wave begins, and half of its panels are the next wave's too.  (Forward and input
//     gradient of a dense layer gain less than 1 % from it, and a token's outputs would have other bits elsewhere in the batch);
//   - every other group is walked backwards: the wave that straddles two groups has the columns of both in common.
// us under sustained load, one tile after the other / so, medians that repeat within 1 %:
//   weight gradient, 16384 tokens 4096 x 4096 425 / 406, 4096 -> 11008 1107 / 1076, 11008 -> 4096 1084 / 1055, 8192 tokens
//     5120 -> 13824 858 / 831; input gradient 4000 tokens 4096 <- 11008 287 / 277, forward 16384 tokens 11008 -> 4096 1130 / 1073;
//   length, weight gradients 4096 x 4096, 4096 -> 11008, 2560 -> 7680, 11008 -> 4096: 4608 tokens 115.9 / 115.2, 303.2 / 301.6,
//     138.0 / 138.1, 304.1 / 304.8; 5632 142.1 / 140.2, 375.2 / 367.5, 170.7 / 168.4, 372.0 / 369.4; 7000 181.2 / 177.0, 485.8 / 468.0,
//     215.5 / 209.7; forward 8192 tokens 5120 -> 4096 258.7 / 258.7, 5632 282.1 / 280.1, 7168 370.9 / 361.9;
//   tile rows, 16384 tokens 8192 -> 1024, 1536, 1792: 217.2 / 216.5, 323.6 / 318.7, 373.0 / 363.4; but with six 12000 tokens
//     7168 -> 1408 205.2 / 205.4, 8500 145.2 / 146.2, forward 1536 tokens 11008 -> 4096 115.2 / 116.0, 1792 138.5 / 136.7.
// DRAM reads in MB, one tile after the other / alternating ends only / so (captures differ by up to a seventh from GPU to GPU): 16384 tokens
// 4096 x 4096 631 / 534 / 430 to 440, 4096 -> 11008 2059 / 1554 / 1140 to 1300, 11008 -> 4096 1698 / 1452 / 1050 to 1230.  (32 k-blocks
// at a time instead of 16: 1 to 2 % longer in wide layers.)
constexpr int kRasterGroupM = 8;
constexpr int kLongFrom = 5632, kLongTileRows = 7;
constexpr int kInterleaveBlocks = 16;
// (`turn`: every other group backwards; `pos`: how many columns of tiles of the group come before the tile's)
__host__ __device__ __forceinline__ void raster_tile(int tile, int num_m, int num_n, bool turn, int& m, int& n, int& pos) {
    const int group_size = kRasterGroupM * num_n;
    const int g = tile / group_size;
    const int first_m = g * kRasterGroupM;
    const int gm = num_m - first_m < kRasterGroupM ? num_m - first_m : kRasterGroupM;
    const int local = tile - g * group_size;
    m = first_m + local % gm;
    pos = local / gm;
    n = turn && (g & 1) ? num_n - 1 - pos : pos;
}

// Work items of the persistent CTA-pair GEMM.  Items are tiles in raster order; when the tiles
// left over after the last full wave of the machine (num_tiles mod num_pairs) fill at most
// half of the pairs, each of them is cut into two half-width items, so that the last wave
// takes half the time instead of a full tile time on a half-empty machine (4096 x 4096 weight
// gradient: 256 tiles on 74 pairs = 3 waves + 34 tiles -> 68 half items: 3.5 instead of 4 waves).
struct PairWork {
    int m_pair, n0, width, pos;
};
__device__ __forceinline__ bool pair_work(int item, int num_pairs, int num_m, int num_n, int width, bool split_tail, bool turn,
                                          PairWork& w) {
    const int num_tiles = num_m * num_n;
    const int full = (num_tiles / num_pairs) * num_pairs, rem = num_tiles - full;
    const bool split = split_tail && rem > 0 && 2 * rem <= num_pairs;
    if (item >= (split ? full + 2 * rem : num_tiles)) return false;
    const bool halved = split && item >= full;
    const int tile = halved ? full + ((item - full) >> 1) : item;
    int n_blk;
    raster_tile(tile, num_m, num_n, turn, w.m_pair, n_blk, w.pos);
    w.width = halved ? width / 2 : width;
    w.n0 = n_blk * width + (halved && ((item - full) & 1) ? width / 2 : 0);
    return true;
}

// Dense CTA-pair GEMM: D[M x N] = A[M x K] * B[N x K]^T with a tile of 256 rows x 64 ... 256 columns per pair (each CTA:
// 128 rows of A, half of the columns of B, 128 accumulator rows).  The width is chosen per launch so that a small
// matrix has tiles for all pairs; a [K x N] operand is loaded in chunks of 64 columns (a width of 64 or 192
// leaves half of a chunk unused).
struct DensePairCfg {
    static constexpr int kABytes = kBlockM * 128;
    static constexpr int kMaxWidth = 256, kMaxStages = 8;
    __host__ __device__ static constexpr int chunks(int width) { return (width / 2 + 63) / 64; }
    __host__ __device__ static constexpr int b_bytes(bool b_mn, int width) { return b_mn ? chunks(width) * 8192 : width * 64; }
    __host__ __device__ static constexpr int stage_bytes(bool b_mn, int width) { return kABytes + b_bytes(b_mn, width); }
    static constexpr int kStoreBytes = 32 * 32 * 2;               // kEpiStore: 32 rows x 32 columns per TMA store
    __host__ __device__ static constexpr int staging_bytes(int epi) { return epi == kEpiStore ? kDenseEpiWarps * 2 * kStoreBytes : 0; }
    __host__ __device__ static constexpr int smem_bytes(bool b_mn, int epi, int width, int stages) {
        return stages * stage_bytes(b_mn, width) + staging_bytes(epi) + 256 + 1024;
    }
};

// LONG: two tiles in turn, in the weight gradient from alternating ends (see raster_tile); a kernel of its own, whose loops do not
// cost the others.
template <bool A_MN, bool B_MN, int EPI, bool LONG>
__global__ void __launch_bounds__(kDenseThreads, 1)
dense_gemm_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                       const __grid_constant__ CUtensorMap tmO /* kEpiStore */, const DenseGemmParams p) {
    using Cfg = DensePairCfg;
    constexpr int kTmemCols = 2 * Cfg::kMaxWidth;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int stages = p.stages, stage_bytes = Cfg::stage_bytes(B_MN, p.width);
    uint8_t* staging = smem + stages * stage_bytes;
    uint64_t* full_bar = reinterpret_cast<uint64_t*>(staging + Cfg::staging_bytes(EPI));
    uint64_t* empty_bar = full_bar + Cfg::kMaxStages;
    uint64_t* tfull_bar = empty_bar + Cfg::kMaxStages;
    uint64_t* tempty_bar = tfull_bar + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty_bar + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t cta = cluster_ctarank();
    const int pair_id = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;
    const int num_m = (p.M + 2 * kBlockM - 1) / (2 * kBlockM);
    const int num_n = (p.N + p.width - 1) / p.width;
    const int num_kb = (p.K + 63) / 64;
    // halving needs B loads of any width: the [K x N] operand is loaded in 64-column chunks
    const bool split_tail = B_MN && p.width == 256;
    constexpr int at_a_time = LONG ? 2 : 1;       // items that a pair works on in turn
    constexpr bool kAlternate = LONG && A_MN;     // every other two from the end of the reduction

    if (threadIdx.x == 0) {
#pragma unroll
        for (int s = 0; s < Cfg::kMaxStages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(&tfull_bar[a], 1); mbar_init(&tempty_bar[a], 2 * kDenseEpiWarps); }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 2 && elect_one()) {
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }
    if (warp == 1) {
        tmem_alloc_pair(tmem_slot, kTmemCols);
        tmem_relinquish_pair();
    }
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync_all();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    // Programmatic dependent launch: the set-up above may overlap the tail of the previous kernel in
    // the stream; no thread touches global memory before that kernel has completed.
    griddep_launch_dependents();
    griddep_wait();

    if (warp == 0) {
        if (elect_one()) {
            RingState ps;
            bool ok = true, backwards = kAlternate;   // (what ran before, the input gradient, read the last tokens last)
            const uint32_t leader_bar = mapa_shared(smem_u32(full_bar), 0);
            // k-blocks [kb0, kb1) of an item
            auto load = [&](const PairWork& w, int kb0, int kb1) {
                const int half_w = w.width / 2;                       // B rows (columns of D) this CTA stages
                const int m0 = (w.m_pair * 2 + static_cast<int>(cta)) * kBlockM;
                const int n0 = w.n0 + static_cast<int>(cta) * half_w;
                const bool two_chunks = Cfg::chunks(w.width) == 2;
                const uint32_t stage_tx = 2 * (dense_a_bytes(A_MN, p.M) + Cfg::b_bytes(B_MN, w.width));
                const int step = kAlternate && backwards ? -64 : 64;
                int k0 = kAlternate && backwards ? (num_kb - 1 - kb0) * 64 : kb0 * 64;
                for (int kb = kb0; kb < kb1; ++kb, k0 += step) {
                    if (!mbar_wait(&empty_bar[ps.stage], ps.phase ^ 1u, abort_flag)) { ok = false; break; }
                    uint8_t* sA = smem + ps.off;
                    uint8_t* sB = sA + Cfg::kABytes;
                    const uint32_t bar = leader_bar + 8 * ps.stage;
                    if (cta == 0) mbar_expect_tx(&full_bar[ps.stage], stage_tx);
                    if (A_MN) {
                        tma_load_2d_pair(sA, &tmA, bar, m0, k0);
                        tma_load_2d_pair(sA + 8192, &tmA, bar, m0 + 64, k0);
                    } else {
                        tma_load_2d_pair(sA, &tmA, bar, k0, m0);
                    }
                    if (B_MN) {
                        tma_load_2d_pair(sB, &tmB, bar, n0, k0);
                        if (two_chunks) tma_load_2d_pair(sB + 8192, &tmB, bar, n0 + 64, k0);
                    } else {
                        tma_load_2d_pair(sB, &tmB, bar, k0, n0);
                    }
                    ps.advance(stages, stage_bytes);
                }
            };
            PairWork w0;
            for (int item = pair_id; ok && pair_work(item, num_pairs, num_m, num_n, p.width, split_tail, LONG, w0);
                 item += at_a_time * num_pairs) {
                if constexpr (LONG) {
                    PairWork w1;
                    const bool two = pair_work(item + num_pairs, num_pairs, num_m, num_n, p.width, split_tail, LONG, w1);
                    for (int kb = 0; ok && kb < num_kb; kb += kInterleaveBlocks) {
                        load(w0, kb, min(kb + kInterleaveBlocks, num_kb));
                        if (two && ok) load(w1, kb, min(kb + kInterleaveBlocks, num_kb));
                    }
                    backwards ^= kAlternate;
                } else {
                    load(w0, 0, num_kb);
                }
            }
        }
    } else if (warp == 1) {
        if (cta == 0 && elect_one()) {
            RingState ps;
            bool ok = true;
            int it = 0;
            ClockProbe probe;
            if (pair_id == 0) probe.begin();
            // k-blocks [kb0, kb1) of a pair's item number `it`
            auto multiply = [&](const PairWork& w, int it, int kb0, int kb1) {
                const uint32_t idesc = make_idesc_bf16(2 * kBlockM, w.width, A_MN, B_MN, false);
                const int acc = it & 1;
                if (kb0 == 0) {
                    const uint32_t acc_phase = static_cast<uint32_t>(it >> 1) & 1u;
                    if (!mbar_wait(&tempty_bar[acc], acc_phase ^ 1u, abort_flag)) { ok = false; return; }
                    tc_fence_after_sync();
                }
                const uint32_t d_tmem = tmem_base + acc * Cfg::kMaxWidth;
                for (int kb = kb0; kb < kb1; ++kb) {
                    if (!mbar_wait(&full_bar[ps.stage], ps.phase, abort_flag)) { ok = false; return; }
                    tc_fence_after_sync();
                    const uint32_t sA = smem_u32(smem + ps.off);
                    const uint32_t sB = sA + Cfg::kABytes;
                    const uint64_t a0 = A_MN ? make_smem_desc(sA, 8192, 1024, kSwizzle128B) : make_smem_desc(sA, 16, 1024, kSwizzle128B);
                    const uint64_t b0 = B_MN ? make_smem_desc(sB, 8192, 1024, kSwizzle128B) : make_smem_desc(sB, 16, 1024, kSwizzle128B);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {              // steps along K, in 16-byte units of the start address
                        const uint64_t ad = a0 + j * (A_MN ? 128 : 2), bd = b0 + j * (B_MN ? 128 : 2);
                        umma_bf16_pair(d_tmem, ad, bd, idesc, (kb | j) != 0 ? 1u : 0u);
                    }
                    umma_commit_pair(&empty_bar[ps.stage], 3);
                    ps.advance(stages, stage_bytes);
                }
                if (kb1 == num_kb) umma_commit_pair(&tfull_bar[acc], 3);
            };
            PairWork w0;
            for (int item = pair_id; ok && pair_work(item, num_pairs, num_m, num_n, p.width, split_tail, LONG, w0);
                 item += at_a_time * num_pairs, it += at_a_time) {
                if constexpr (LONG) {
                    PairWork w1;
                    const bool two = pair_work(item + num_pairs, num_pairs, num_m, num_n, p.width, split_tail, LONG, w1);
                    for (int kb = 0; ok && kb < num_kb; kb += kInterleaveBlocks) {
                        multiply(w0, it, kb, min(kb + kInterleaveBlocks, num_kb));
                        if (two && ok) multiply(w1, it + 1, kb, min(kb + kInterleaveBlocks, num_kb));
                    }
                } else {
                    multiply(w0, it, 0, num_kb);
                }
            }
            if (pair_id == 0) probe.end(kClockDense);
        }
    } else {
        const int q = warp & 3, half = (warp - 2) >> 2;
        bool ok = true;
        int it = 0;
        uint32_t buf = 0;
        const uint32_t my_buf = smem_u32(staging + (warp - 2) * 2 * Cfg::kStoreBytes);
        PairWork w;
        for (int item = pair_id; ok && pair_work(item, num_pairs, num_m, num_n, p.width, split_tail, LONG, w);
             item += num_pairs, ++it) {
            const int acc = it & 1;
            const uint32_t acc_phase = static_cast<uint32_t>(it >> 1) & 1u;
            const int m = (w.m_pair * 2 + static_cast<int>(cta)) * kBlockM + q * 32 + lane;
            const int cols = w.width / 2, n0 = w.n0 + half * cols;
            // columns inside the matrix: N is a multiple of 128, so a part of them only at a width of 192 (kEpiStore)
            const int left = min(cols, p.N - n0);
            const bool live = m < p.M && left > 0;           // (kEpiMasked: the same for all rows of a CTA)
            uint32_t mw[4];
            if (EPI == kEpiMasked && live)
                load_mask_bits(p.mask + static_cast<size_t>(m) * (p.N >> 3) + (n0 >> 3), cols, mw);
            if (!mbar_wait(&tfull_bar[acc], acc_phase, abort_flag)) { ok = false; break; }
            tc_fence_after_sync();
            const uint32_t t_row = tmem_base + acc * Cfg::kMaxWidth + half * cols + (static_cast<uint32_t>(q * 32) << 16);
            if (EPI == kEpiMasked) {
                if (live) drain_row<EPI>(t_row, left, p, m, n0, mw);
            } else if (m - lane < p.M) {
                // 32 columns at a time through a private staging buffer (64-byte rows, 16-byte pieces XOR-swizzled as the
                // store's tensor map expects) and out as a TMA store, which leaves out rows past M.  (Stored straight from
                // the registers, 16 bytes in each of 32 rows per instruction, the drain paced small and short products: us,
                // before -> after, forward 8192 tokens 768 -> 3072 37.4 -> 31.4, 700 tokens 2048 -> 6144 17.8 -> 15.8, weight
                // gradient 300 tokens 2560 -> 7680 22.7 -> 13.7; 2048 tokens 4096 -> 4096 49.6 -> 48.4.)
#pragma unroll 1
                for (int c0 = 0; c0 < left; c0 += 32) {
                    uint32_t v[2][16];
                    tmem_ld_16(t_row + c0, v[0]);
                    tmem_ld_16(t_row + c0 + 16, v[1]);
                    if (lane == 0) tma_store_wait_read<1>();          // the store before last has read this buffer
                    __syncwarp();
                    tmem_ld_wait();
                    const uint32_t row = my_buf + buf * Cfg::kStoreBytes + lane * 64;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint32_t* e = v[k >> 1] + 8 * (k & 1);
                        st_shared_v4(row + ((k ^ ((lane >> 1) & 3)) << 4),
                                     make_uint4(pack_bf16x2(__uint_as_float(e[0]), __uint_as_float(e[1])),
                                                pack_bf16x2(__uint_as_float(e[2]), __uint_as_float(e[3])),
                                                pack_bf16x2(__uint_as_float(e[4]), __uint_as_float(e[5])),
                                                pack_bf16x2(__uint_as_float(e[6]), __uint_as_float(e[7]))));
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_2d(&tmO, my_buf + buf * Cfg::kStoreBytes, n0 + c0, m);
                        tma_store_commit();
                    }
                    buf ^= 1u;
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(mapa_shared(smem_u32(&tempty_bar[acc]), 0));
        }
        if (EPI == kEpiStore && lane == 0) tma_store_wait_all<0>();
    }

    __syncwarp();
    if (*abort_flag) drain_after_abort();
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync_all();
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc_pair(tmem_base, kTmemCols);
    }
}

// =====================================================================================
// Sparse CTA-pair GEMM with a 512-row tile: the pair runs TWO 256-row MMA sub-tiles against
// ONE staged activation tile, so every activation byte pulled from L2 feeds twice as many
// MMAs (L2 -> SM bytes per FLOP drop by 31 % against the 256-row tile; that fabric, not DRAM
// or the tensor pipe, is what bounds these GEMMs).  Tensor memory then holds one accumulator
// per sub-tile (2 x 224 columns) plus the metadata columns, so accumulators are single
// buffered; the epilogue is made short instead: accumulator rows are transposed through
// shared memory and leave as TMA stores of 32 tokens x 32 features.
//   128-row block of A handled by CTA c for sub-tile s of tile mt:  4*mt + 2*s + c.
// =====================================================================================
constexpr int kPrefetchAhead = 8;          // k-blocks of L2 prefetch distance for activation boxes

struct SparseQuadCfg {
    static constexpr int kABytes = kBlockM * 128;                 // per sub-tile
    static constexpr int kEBytes = 2048;                          // per sub-tile
    static constexpr int kOffB = 2 * kABytes;
    static constexpr int kStoreRows = 32;                         // tokens per TMA store
    static constexpr int kStoreCols = 32;                         // features per TMA store (one warp's lanes)
    static constexpr int kStoreBytes = kStoreRows * kStoreCols * 2;
    static constexpr int kEpiWarps = 8;                           // two warps per tensor-memory lane quadrant
    static constexpr int kThreads = 64 + 32 * kEpiWarps;
    static constexpr int kStagingBytes = kEpiWarps * 2 * kStoreBytes;
    static constexpr int kECol = 2 * kMaxTokenTile;
    __host__ __device__ static constexpr int stage_bytes(int width) { return kOffB + width * 128 + 2 * kEBytes; }
    __host__ __device__ static constexpr int smem_bytes(int width, int stages) {
        return stages * stage_bytes(width) + kStagingBytes + 256 + 1024;
    }
    static_assert(2 * kMaxTokenTile + 16 <= 512, "tile does not fit tensor memory");
};

// Tile order of the 512-row-tile kernel: row tiles fastest inside a group of `group_m` row tiles,
// then token blocks, then the next group.  The pairs that work on one token block side by side
// share its activation tile; a group's share of the compressed weight is what has to stay in L2
// while the token blocks sweep by.  `first` marks the tile that prefetches the block's
// activations into L2 for its group.  Every tile takes the k-blocks from the first to the last: a token's outputs then have
// the same bits wherever in the batch it stands.  (Where a group's weights are more than L2 keeps, tiles that took them from
// alternating ends found some 180 of 795 MB still there -- 16384 tokens 11008 -> 4096 631 -> 619 us, 8192 tokens 13824 -> 5120
// 485 -> 476 -- but two equal tokens could then differ in the last bit.)
__device__ __forceinline__ void quad_tile(int tile, int num_m, int num_n, int group_m, int& mt, int& n_blk,
                                          bool& first) {
    const int group_size = group_m * num_n;
    const int g = tile / group_size;
    const int first_m = g * group_m;
    const int gm = min(num_m - first_m, group_m);
    const int local = tile - g * group_size;
    mt = first_m + local % gm;
    n_blk = local / gm;
    first = local % gm == 0;
}

__global__ void __launch_bounds__(SparseQuadCfg::kThreads, 1)
sparse_gemm_quad_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                        const __grid_constant__ CUtensorMap tmE, const __grid_constant__ CUtensorMap tmA2,
                        const __grid_constant__ CUtensorMap tmB2, const __grid_constant__ CUtensorMap tmO,
                        const SparseGemmParams p) {
    using Cfg = SparseQuadCfg;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int stages = p.stages, stage_bytes = Cfg::stage_bytes(p.width);
    const uint32_t b_half = p.width * 64;                    // bytes of one 64-column half of the activation tile
    const uint32_t off_e = Cfg::kOffB + 2 * b_half;
    uint8_t* staging = smem + stages * stage_bytes;
    uint64_t* full_bar = reinterpret_cast<uint64_t*>(staging + Cfg::kStagingBytes);
    uint64_t* empty_bar = full_bar + kMaxTileStages;
    uint64_t* tfull_bar = empty_bar + kMaxTileStages;
    uint64_t* tempty_bar = tfull_bar + 2;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty_bar + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t cta = cluster_ctarank();
    const int pair_id = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;
    const int num_mb = p.M / kBlockM;
    const int num_m = (num_mb + 3) / 4;                      // 512-row tiles
    const int num_n = p.num_n;
    const int num_tiles = num_m * num_n;
    const int num_kb = p.K / 128;
    const int num_ab = (p.r + 63) / 64;
    const int total_kb = num_kb + num_ab;
    const int group_m = p.group_m > 0 && p.group_m < num_m ? p.group_m : num_m;

    if (threadIdx.x == 0) {
#pragma unroll
        for (int s = 0; s < kMaxTileStages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        mbar_init(&tfull_bar[0], 1);
        mbar_init(&tfull_bar[1], 1);
        mbar_init(&tempty_bar[0], 2 * Cfg::kEpiWarps);
        mbar_init(&tempty_bar[1], 2 * Cfg::kEpiWarps);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 2 && elect_one()) {
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
        tma_prefetch_desc(&tmE);
    }
    if (warp == 1) {
        tmem_alloc_pair(tmem_slot, 512);
        tmem_relinquish_pair();
    }
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync_all();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    // Programmatic dependent launch: the set-up above may overlap the tail of the previous kernel in
    // the stream; no thread touches global memory before that kernel has completed.
    // (consumer of a fused pair of launches, pdl_mode 2: only the producer thread waits, before its
    // first load of the adapter operand T)
    griddep_launch_dependents();
    if (p.pdl_mode != 2) griddep_wait();

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer (both CTAs)
        if (elect_one()) {
            const uint64_t keep = l2_policy_evict_last();
            PipeState ps;
            bool ok = true;
            bool waited = false;
            for (int tile = pair_id; ok && tile < num_tiles; tile += num_pairs) {
                int mt, n_blk, next_mt, next_n_blk;
                bool first, next_first = false;
                quad_tile(tile, num_m, num_n, group_m, mt, n_blk, first);
                const int nsub = (4 * mt + 2 < num_mb) ? 2 : 1;              // second sub-tile may lie past M
                const int width = token_tile_width(p.Ntok, n_blk * p.width, p.width);
                const int n_row0 = n_blk * p.width + static_cast<int>(cta) * (width / 2);
                // The pairs working on the same token block (same n_blk, different mt) run side by
                // side and would all wait on the same first-touch DRAM fetch of an activation box.
                // One of them (mt == 0) pulls the boxes into L2 kPrefetchAhead k-blocks early.
                const int next_tile = tile + num_pairs;
                if (next_tile < num_tiles) quad_tile(next_tile, num_m, num_n, group_m, next_mt, next_n_blk, next_first);
                const int next_row0 =
                    next_first ? next_n_blk * p.width +
                                     static_cast<int>(cta) * (token_tile_width(p.Ntok, next_n_blk * p.width, p.width) / 2)
                               : 0;
                for (int kb = 0; kb < total_kb; ++kb) {
                    if (kb < num_kb) {
                        const int pk = kb + kPrefetchAhead;
                        if (pk < num_kb) {
                            if (first) {
                                tma_prefetch_l2_2d(&tmB, pk * 128, n_row0);
                                tma_prefetch_l2_2d(&tmB, pk * 128 + 64, n_row0);
                            }
                        } else if (next_first && pk - num_kb < num_kb) {
                            tma_prefetch_l2_2d(&tmB, (pk - num_kb) * 128, next_row0);
                            tma_prefetch_l2_2d(&tmB, (pk - num_kb) * 128 + 64, next_row0);
                        }
                    }
                    if (!mbar_wait(&empty_bar[ps.stage], ps.phase ^ 1u, abort_flag)) { ok = false; break; }
                    uint8_t* st = smem + ps.stage * stage_bytes;
                    uint8_t* sB = st + Cfg::kOffB;
                    const uint32_t bar = mapa_shared(smem_u32(&full_bar[ps.stage]), 0);
                    if (kb < num_kb) {
                        if (cta == 0)
                            mbar_expect_tx(&full_bar[ps.stage],
                                           2 * (2 * b_half + nsub * (Cfg::kABytes + Cfg::kEBytes)));
                        tma_load_2d_pair(sB, &tmB, bar, kb * 128, n_row0);
                        tma_load_2d_pair(sB + b_half, &tmB, bar, kb * 128 + 64, n_row0);
                        for (int s = 0; s < nsub; ++s) {
                            const int mb = 4 * mt + 2 * s + static_cast<int>(cta);
                            const int mb_e = mb < num_mb ? mb : num_mb - 1;
                            tma_load_2d_pair_hint(st + s * Cfg::kABytes, &tmA, bar, kb * 64, mb * kBlockM, keep);
                            tma_load_2d_pair_hint(st + off_e + s * Cfg::kEBytes, &tmE, bar, 0, mb_e * num_kb + kb,
                                                  keep);
                        }
                    } else {
                        const int ab = kb - num_kb;
                        if (p.pdl_mode == 2 && !waited) {
                            griddep_wait();
                            waited = true;
                        }
                        if (cta == 0)
                            mbar_expect_tx(&full_bar[ps.stage], 2 * (b_half + nsub * Cfg::kABytes));
                        tma_load_2d_pair(sB, &tmB2, bar, ab * 64, n_row0);
                        for (int s = 0; s < nsub; ++s) {
                            const int m0 = (4 * mt + 2 * s + static_cast<int>(cta)) * kBlockM;
                            uint8_t* sA = st + s * Cfg::kABytes;
                            if (p.a2_mn_major) {
                                tma_load_2d_pair(sA, &tmA2, bar, m0, ab * 64);
                                tma_load_2d_pair(sA + 8192, &tmA2, bar, m0 + 64, ab * 64);
                            } else {
                                tma_load_2d_pair(sA, &tmA2, bar, ab * 64, m0);
                            }
                        }
                    }
                    ps.advance(stages);
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer (leader CTA only)
        if (cta == 0 && elect_one()) {
            uint32_t idesc_sp = 0, idesc_ad = 0;              // set per tile: N is the tile's width
            // the MMAs of sub-tile s for k-block kb out of pipeline stage `stage`
            auto issue = [&](int s, int kb, int stage) {
                const uint32_t st = smem_u32(smem + stage * stage_bytes);
                const uint32_t sB = st + Cfg::kOffB;
                const uint32_t d_tmem = tmem_base + s * kMaxTokenTile;
                const uint32_t sA = st + s * Cfg::kABytes;
                if (kb < num_kb) {
                    const uint32_t e_tmem = tmem_base + Cfg::kECol + (kb & 1) * 8 + s * 4;
                    tmem_cp_128x128b_pair(e_tmem, make_smem_desc(st + off_e + s * Cfg::kEBytes, 128, 128,
                                                                 kSwizzleNone));
                    const uint64_t a0 = make_smem_desc(sA, 16, 1024, kSwizzle128B);
                    const uint64_t b0 = make_smem_desc(sB, 16, 1024, kSwizzle128B);
                    const uint64_t b2 = b0 + (b_half >> 4);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint64_t ad = a0 + 2 * j, bd = (j < 2 ? b0 : b2) + 4 * (j & 1);
                        umma_bf16_sp_pair(d_tmem, ad, bd, e_tmem + (j & 2), idesc_sp | (j & 1), (kb | j) != 0 ? 1u : 0u);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint64_t ad = p.a2_mn_major ? make_smem_desc(sA + j * 2048, 8192, 1024, kSwizzle128B)
                                                          : make_smem_desc(sA + j * 32, 16, 1024, kSwizzle128B);
                        const uint64_t bd = make_smem_desc(sB + j * 32, 16, 1024, kSwizzle128B);
                        umma_bf16_pair(d_tmem, ad, bd, idesc_ad, 1u);
                    }
                }
                // sub-tile s is complete with its last k-block: its drain may start while the other
                // sub-tile's last MMAs still run
                if (kb == total_kb - 1) umma_commit_pair(&tfull_bar[s], 3);
            };
            PipeState ps;                                     // stage that sub-tile 0 consumes next
            bool ok = true;
            int it = 0;
            ClockProbe probe;
            if (pair_id == 0) probe.begin();
            for (int tile = pair_id; ok && tile < num_tiles; tile += num_pairs, ++it) {
                int mt, n_blk;
                bool first_unused;
                quad_tile(tile, num_m, num_n, group_m, mt, n_blk, first_unused);
                const int nsub = (4 * mt + 2 < num_mb) ? 2 : 1;
                const int width = token_tile_width(p.Ntok, n_blk * p.width, p.width);
                idesc_sp = make_idesc_bf16(2 * kBlockM, width, false, false, true);
                idesc_ad = make_idesc_bf16(2 * kBlockM, width, p.a2_mn_major != 0, false, false);
                const uint32_t acc_parity = (static_cast<uint32_t>(it) & 1u) ^ 1u;
                if (!mbar_wait(&tempty_bar[0], acc_parity, abort_flag)) { ok = false; break; }
                tc_fence_after_sync();
                // The epilogue hands the second accumulator back a little after the first.  Until
                // then sub-tile 0 runs ahead through the stages that are already full (they cannot
                // be released before sub-tile 1 has used them too); then sub-tile 1 catches up.
                PipeState pc = ps;                            // stage that sub-tile 1 consumes (and releases) next
                int kb0 = 0;
                bool ready1 = nsub == 1;
                while (ok && !ready1) {
                    ready1 = mbar_test(&tempty_bar[1], acc_parity);
                    if (ready1) break;
                    if (kb0 < total_kb && kb0 < stages) {
                        if (!mbar_wait(&full_bar[ps.stage], ps.phase, abort_flag)) { ok = false; break; }
                        tc_fence_after_sync();
                        issue(0, kb0, ps.stage);
                        ps.advance(stages);
                        ++kb0;
                    } else {
                        ok = mbar_wait(&tempty_bar[1], acc_parity, abort_flag);
                        ready1 = true;
                    }
                }
                if (!ok) break;
                tc_fence_after_sync();
                if (nsub == 2) {
                    for (int kb1 = 0; kb1 < kb0; ++kb1) {       // catch up
                        issue(1, kb1, pc.stage);
                        umma_commit_pair(&empty_bar[pc.stage], 3);
                        pc.advance(stages);
                    }
                }
                for (int kb = kb0; kb < total_kb; ++kb) {        // in step
                    if (!mbar_wait(&full_bar[ps.stage], ps.phase, abort_flag)) { ok = false; break; }
                    tc_fence_after_sync();
                    issue(0, kb, ps.stage);
                    if (nsub == 2) issue(1, kb, ps.stage);
                    umma_commit_pair(&empty_bar[ps.stage], 3);
                    ps.advance(stages);
                }
                if (ok && nsub == 1) umma_commit_pair(&tfull_bar[1], 3);        // keep both barriers in phase
            }
            if (pair_id == 0) probe.end(kClockSparse);
        }
    } else {
        // ------------------------------------------------------------ epilogue (warps 2..9, both CTAs)
        // Warp w drains lane quadrant w%4; the two warps of a quadrant take alternate 32-token
        // blocks.  Phase 1 empties both accumulators into registers (packed bf16) and hands them
        // back to the MMA issuer at once -- the accumulators are single buffered, so this is
        // what the next tile waits for.  Phase 2 runs under the next tile's main loop: each warp
        // transposes its 32 x 32 blocks through a private staging buffer and sends them with its
        // own TMA stores; the warps never wait for one another.  Nothing hides the last tile's phase 2: with one tile
        // per pair (500 tokens, 4096 -> 11008) it took 7000 of 38000 clocks while a block was staged by 32 two-byte
        // stores per lane instead of four stmatrix.  Now the last tile goes block by block from tensor memory to its store, in
        // one loop whose code stays cached: 27.9 -> 25.9 us, 700 tokens 4096 -> 5120 21.9 -> 20.8.
        constexpr int kBlocks = kMaxTokenTile / Cfg::kStoreRows;   // 32-token blocks per accumulator
        constexpr int kMyBlocks = (kBlocks + 1) / 2;              // at most this many per warp
        const int q = warp & 3;
        const int ew = warp - 2;
        const int half = ew >> 2;
        uint8_t* my_buf = staging + ew * 2 * Cfg::kStoreBytes;
        const uint64_t stream_out = l2_policy_evict_first();
        bool ok = true;
        int it = 0;
        uint32_t buf = 0;
        auto store_block = [&](const uint32_t (&block)[16], int m0, int n0) {
            // (Rows past M are not staged either: the wait below counts stores, and a block that is staged but not stored
            // would let the one after it overwrite a buffer whose store is still reading.)
            if (m0 >= p.M) return;
            // the staging buffer about to be overwritten must have been read by its TMA store
            if (lane == 0) tma_store_wait_read<1>();
            __syncwarp();
            stage_packed_block(smem_u32(my_buf + buf * Cfg::kStoreBytes), lane, block);
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                tma_store_2d_hint(&tmO, my_buf + buf * Cfg::kStoreBytes, m0, n0, stream_out);
                tma_store_commit();
            }
            buf ^= 1u;
        };
        for (int tile = pair_id; ok && tile < num_tiles; tile += num_pairs, ++it) {
            int mt, n_blk;
            bool first_unused;
            quad_tile(tile, num_m, num_n, group_m, mt, n_blk, first_unused);
            const int nsub = (4 * mt + 2 < num_mb) ? 2 : 1;
            const int width = token_tile_width(p.Ntok, n_blk * p.width, p.width);
            if (tile + num_pairs >= num_tiles) {
                // the pair's last tile: nothing waits for the accumulators and nothing hides phase 2, so one short loop
                // takes every block from tensor memory to its store
                for (int s = 0; ok && s < nsub; ++s) {
                    ok = mbar_wait(&tfull_bar[s], static_cast<uint32_t>(it) & 1u, abort_flag);
                    if (!ok) break;
                    tc_fence_after_sync();
                    const uint32_t t_row = tmem_base + s * kMaxTokenTile + (static_cast<uint32_t>(q * 32) << 16);
                    const int m0 = (4 * mt + 2 * s + static_cast<int>(cta)) * kBlockM + q * 32;
#pragma unroll 1
                    for (int c0 = half * Cfg::kStoreRows; c0 < width; c0 += 2 * Cfg::kStoreRows) {
                        uint32_t block[16];
                        load_packed_block(t_row + c0, block);
                        store_block(block, m0, n_blk * p.width + c0);
                    }
                }
                break;
            }
            uint32_t pk[2][kMyBlocks][16];
            // ---- first accumulator (its drain is what the next tile's first MMA waits for).  One load of 16 registers at a
            //      time: the warps of a 320-thread CTA are allocated registers as twelve, which caps a thread at 168, and
            //      128 of them hold the two packed accumulators.
            if (!mbar_wait(&tfull_bar[0], static_cast<uint32_t>(it) & 1u, abort_flag)) { ok = false; break; }
            tc_fence_after_sync();
            {
                const uint32_t t_row = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
#pragma unroll
                for (int j = 0; j < kMyBlocks; ++j) {
                    const int c0 = (2 * j + half) * Cfg::kStoreRows;
                    if (c0 < width) {
                        load_packed_block(t_row + c0, pk[0][j]);
                    }
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(mapa_shared(smem_u32(&tempty_bar[0]), 0));
            // ---- second accumulator
            if (!mbar_wait(&tfull_bar[1], static_cast<uint32_t>(it) & 1u, abort_flag)) { ok = false; break; }
            tc_fence_after_sync();
            if (nsub == 2) {
                const uint32_t t_row = tmem_base + kMaxTokenTile + (static_cast<uint32_t>(q * 32) << 16);
#pragma unroll
                for (int j = 0; j < kMyBlocks; ++j) {
                    const int c0 = (2 * j + half) * Cfg::kStoreRows;
                    if (c0 < width) {
                        load_packed_block(t_row + c0, pk[1][j]);
                    }
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(mapa_shared(smem_u32(&tempty_bar[1]), 0));
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                if (s < nsub) {
                    const int m0 = (4 * mt + 2 * s + static_cast<int>(cta)) * kBlockM + q * 32;
#pragma unroll
                    for (int j = 0; j < kMyBlocks; ++j) {
                        const int c0 = (2 * j + half) * Cfg::kStoreRows;
                        if (c0 < width) store_block(pk[s][j], m0, n_blk * p.width + c0);
                    }
                }
            }
        }
        if (lane == 0) tma_store_wait_all<0>();
    }

    __syncwarp();
    if (*abort_flag) drain_after_abort();
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync_all();
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc_pair(tmem_base, 512);
    }
}

// =====================================================================================
// Sparse GEMM for few tokens (inference / decode sizes, Ntok <= BLOCK_N <= 128).
// With so few tokens the GEMM is a stream of compressed weights from HBM, and the big-tile
// kernels above would occupy only a handful of SMs.  Here one CTA owns a 128-row slab of the
// weights (1-CTA tcgen05.mma.sp, M = 128) and a slice of the reduction: a cluster of S CTAs
// splits K, each accumulates its partial tile in tensor memory, parks it in its own shared
// memory, and after a cluster barrier every CTA sums one share of the token rows over all S
// partials through distributed shared memory -- in rank order, so the result is
// deterministic and needs no global workspace.  The adapter K-steps ride on the last rank.
//
// What bounds the kernel is the number of weight bytes in flight, so the weights (values +
// metadata, from HBM, read once) and the activations (from L2, re-read by every slab) travel
// in two separate rings with their own producer threads: a deep one for the weights, a
// shallow one for the activations.
// =====================================================================================
constexpr int kSkinnyPrefetchBlocks = 6;   // k-blocks whose first-byte latency is otherwise exposed (6 x 0.23 us)

template <int BLOCK_N, int A_STAGES, int B_STAGES>
struct SparseSkinnyCfg {
    static constexpr int kABytes = kBlockM * 128;                    // compressed values of one k-block
    static constexpr int kEBytes = 2048;                             // their metadata
    static constexpr int kAStage = kABytes + kEBytes;
    static constexpr int kBStage = BLOCK_N * 256;
    static constexpr int kOffB = A_STAGES * kAStage;
    static constexpr int kOffBar = kOffB + B_STAGES * kBStage;
    static constexpr int kPartialBytes = BLOCK_N * kBlockM * 4;      // fp32 [token][feature], reuses the rings
    static constexpr int kSmemBytes = kOffBar + 512 + 1024;
    static constexpr int kTmemCols = BLOCK_N + 8 <= 32 ? 32 : (BLOCK_N + 8 <= 128 ? 128 : (BLOCK_N + 8 <= 256 ? 256 : 512));
    static_assert(BLOCK_N % 16 == 0 && BLOCK_N >= 16 && BLOCK_N <= 128, "token tile");
    static_assert(kPartialBytes <= kOffBar, "partial tile must fit in the pipeline buffers");
    static_assert(kAStage % 1024 == 0 && kBStage % 1024 == 0 && kSmemBytes <= 232448, "shared memory layout");
    static_assert(2 * (A_STAGES + B_STAGES) * 8 + 16 <= 512, "barrier block");
};

template <int BLOCK_N, int A_STAGES, int B_STAGES>
__global__ void __launch_bounds__(kGemmThreads, 1)
sparse_gemm_skinny_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                          const __grid_constant__ CUtensorMap tmE, const __grid_constant__ CUtensorMap tmA2,
                          const __grid_constant__ CUtensorMap tmB2, const SparseGemmParams p) {
    using Cfg = SparseSkinnyCfg<BLOCK_N, A_STAGES, B_STAGES>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* fullA = reinterpret_cast<uint64_t*>(smem + Cfg::kOffBar);
    uint64_t* emptyA = fullA + A_STAGES;
    uint64_t* fullB = emptyA + A_STAGES;
    uint64_t* emptyB = fullB + B_STAGES;
    uint64_t* tfull_bar = emptyB + B_STAGES;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tfull_bar + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int splits = static_cast<int>(cluster_nctarank());
    const int rank = static_cast<int>(cluster_ctarank());
    const int m_blk = blockIdx.x / splits;
    const int num_kb = p.K / 128;
    const int kb_per = (num_kb + splits - 1) / splits;
    const int kb0 = min(num_kb, rank * kb_per), kb1 = min(num_kb, kb0 + kb_per);
    const int num_sb = kb1 - kb0;                                            // sparse k-blocks of this rank
    // Dense K-steps (64 wide): the adapter product rides on the last rank.
    const int num_ab = rank == splits - 1 ? (p.r + 63) / 64 : 0;
    const int total_kb = num_sb + num_ab;

    if (threadIdx.x == 0) {
        for (int s = 0; s < A_STAGES; ++s) { mbar_init(&fullA[s], 1); mbar_init(&emptyA[s], 1); }
        for (int s = 0; s < B_STAGES; ++s) { mbar_init(&fullB[s], 1); mbar_init(&emptyB[s], 1); }
        mbar_init(&tfull_bar[0], 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, Cfg::kTmemCols);
        tmem_relinquish();
    }
    if (warp == 2 && elect_one()) {
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmE);
    }
    if (warp == 2 && elect_one()) tma_prefetch_desc(&tmB);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    // Everything above overlaps the tail of the previous kernel in the stream when the launch
    // allows it; nothing below may touch global memory before that kernel has finished.  One
    // thing is safe earlier: asking L2 to fetch this CTA's first weight tiles.  A prefetch moves no
    // data into the SM, and L2 is the point of coherence, so a line the previous kernel is still
    // writing stays correct; the first loads after the wait then come at L2 instead of HBM latency.
    //
    // Two launches issued together by one call (T = X L, then the forward that adds T R) use the
    // dependency more finely.  The producer (adapter_gemm_kernel, pdl_mode 1) waits first and releases
    // its dependents afterwards: when the consumer starts, everything that preceded the pair in the
    // stream is complete.  The consumer (pdl_mode 2) therefore streams its weights and activations
    // and runs its whole sparse reduction without waiting; only the thread that loads the producer's
    // output T waits, right before the first such load.  Everything that follows in the consumer
    // (the adapter MMAs, the cluster reduction, the stores) is ordered behind that load.
    griddep_launch_dependents();
    if (warp == 0 && elect_one()) {
        // (4 linears of a decoder block of width 1280 at one token, slices of 2 ... 5 k-blocks: 19.3 -> 18.1 us)
        const int n_pf = p.pdl_mode == 0 ? min(num_sb, kSkinnyPrefetchBlocks) : 0;
        for (int i = 0; i < n_pf; ++i) {
            tma_prefetch_l2_2d(&tmA, (kb0 + i) * 64, m_blk * kBlockM);
            tma_prefetch_l2_2d(&tmE, 0, m_blk * num_kb + kb0 + i);
        }
    }
    __syncwarp();
    if (p.pdl_mode != 2) griddep_wait();

    if (warp == 0) {
        // ---------------------------------------------------------- weight ring (values + metadata)
        if (elect_one()) {
            const uint64_t stream_once = l2_policy_evict_first();        // weights are read exactly once
            PipeState ps;
            for (int i = 0; i < total_kb; ++i) {
                if (!mbar_wait(&emptyA[ps.stage], ps.phase ^ 1u, abort_flag)) break;
                uint8_t* sA = smem + ps.stage * Cfg::kAStage;
                uint64_t* bar = &fullA[ps.stage];
                if (i < num_sb) {
                    const int kb = kb0 + i;
                    mbar_expect_tx(bar, Cfg::kAStage);
                    tma_load_2d_hint(sA, &tmA, bar, kb * 64, m_blk * kBlockM, stream_once);
                    tma_load_2d_hint(sA + Cfg::kABytes, &tmE, bar, 0, m_blk * num_kb + kb, stream_once);
                } else {
                    const int ab = i - num_sb;
                    mbar_expect_tx(bar, Cfg::kABytes);
                    if (p.a2_mn_major) {
                        tma_load_2d(sA, &tmA2, bar, m_blk * kBlockM, ab * 64);
                        tma_load_2d(sA + 8192, &tmA2, bar, m_blk * kBlockM + 64, ab * 64);
                    } else {
                        tma_load_2d(sA, &tmA2, bar, ab * 64, m_blk * kBlockM);
                    }
                }
                ps.advance(A_STAGES);
            }
        }
    } else if (warp == 1) {
        // ---------------------------------------------------------- MMA issue
        if (elect_one()) {
            constexpr uint32_t idesc_sp = make_idesc_bf16(kBlockM, BLOCK_N, false, false, true);
            const uint32_t idesc_ad = make_idesc_bf16(kBlockM, BLOCK_N, p.a2_mn_major != 0, false, false);
            PipeState pa, pb;
            bool ok = true;
            for (int i = 0; i < total_kb; ++i) {
                if (!mbar_wait(&fullB[pb.stage], pb.phase, abort_flag)) { ok = false; break; }
                if (!mbar_wait(&fullA[pa.stage], pa.phase, abort_flag)) { ok = false; break; }
                tc_fence_after_sync();
                const uint32_t sA = smem_u32(smem + pa.stage * Cfg::kAStage);
                const uint32_t sE = sA + Cfg::kABytes;
                const uint32_t sB = smem_u32(smem + Cfg::kOffB + pb.stage * Cfg::kBStage);
                if (i < num_sb) {
                    const uint32_t e_tmem = tmem_base + BLOCK_N + (i & 1) * 4;
                    tmem_cp_128x128b(e_tmem, make_smem_desc(sE, 128, 128, kSwizzleNone));
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint64_t ad = make_smem_desc(sA + j * 32, 16, 1024, kSwizzle128B);
                        const uint64_t bd =
                            make_smem_desc(sB + (j >> 1) * (BLOCK_N * 128) + (j & 1) * 64, 16, 1024, kSwizzle128B);
                        umma_bf16_sp(tmem_base, ad, bd, e_tmem + (j & 2), idesc_sp | (j & 1), (i | j) != 0 ? 1u : 0u);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint64_t ad = p.a2_mn_major ? make_smem_desc(sA + j * 2048, 8192, 1024, kSwizzle128B)
                                                          : make_smem_desc(sA + j * 32, 16, 1024, kSwizzle128B);
                        const uint64_t bd = make_smem_desc(sB + j * 32, 16, 1024, kSwizzle128B);
                        umma_bf16(tmem_base, ad, bd, idesc_ad, (i | j) != 0 ? 1u : 0u);
                    }
                }
                umma_commit(&emptyA[pa.stage]);
                umma_commit(&emptyB[pb.stage]);
                pa.advance(A_STAGES);
                pb.advance(B_STAGES);
            }
            if (ok) umma_commit(&tfull_bar[0]);
        }
    } else if (warp == 2) {
        // ---------------------------------------------------------- activation ring
        if (elect_one()) {
            PipeState ps;
            const uint32_t half_bytes = p.width * 128;                   // p.width token rows (see launch_sparse_skinny)
            for (int i = 0; i < total_kb; ++i) {
                if (!mbar_wait(&emptyB[ps.stage], ps.phase ^ 1u, abort_flag)) break;
                uint8_t* sB = smem + Cfg::kOffB + ps.stage * Cfg::kBStage;
                uint64_t* bar = &fullB[ps.stage];
                if (i < num_sb) {
                    const int kb = kb0 + i;
                    mbar_expect_tx(bar, 2 * half_bytes);
                    tma_load_2d(sB, &tmB, bar, kb * 128, 0);
                    tma_load_2d(sB + BLOCK_N * 128, &tmB, bar, kb * 128 + 64, 0);
                } else {
                    if (p.pdl_mode == 2 && i == num_sb) griddep_wait();      // T comes from the launch before this one
                    mbar_expect_tx(bar, half_bytes);
                    tma_load_2d(sB, &tmB2, bar, (i - num_sb) * 64, 0);
                }
                ps.advance(B_STAGES);
            }
        }
        __syncwarp();
    }

    // ---------------------------------------------------------------- epilogue (warps 2..5)
    // Park the fp32 partial tile in shared memory as [token][feature]; the pipeline buffers are
    // free once the last MMA has completed (tfull).  A rank with no k-block contributes zeros.
    // A CTA that has a slab to itself (no split) stores straight from tensor memory instead: the four linears of a
    // decoder block, two of them unsplit, at one token, width 4096 / 1280: 51.5 -> 49.8 / 18.0 -> 16.9 us.
    float* partial = reinterpret_cast<float*>(smem);
    bool ok = true;
    if (warp >= 2) {
        const int q = warp & 3;
        if (total_kb > 0) ok = mbar_wait(&tfull_bar[0], 0u, abort_flag);
        tc_fence_after_sync();
        const uint32_t t_row = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
        const int ncols = min(BLOCK_N, (p.Ntok + 15) & ~15);         // columns past the last token are never read
#pragma unroll 1
        for (int c0 = 0; c0 < ncols; c0 += 16) {
            uint32_t v[16];
            if (total_kb > 0 && ok) {
                tmem_ld_16(t_row + c0, v);
                tmem_ld_wait();
            } else {
#pragma unroll
                for (int c = 0; c < 16; ++c) v[c] = 0u;
            }
            if (splits == 1) {
                uint16_t* o = p.out + static_cast<size_t>(c0) * p.M + m_blk * kBlockM + q * 32 + lane;
#pragma unroll
                for (int c = 0; c < 16; ++c)
                    if (ok && c0 + c < p.Ntok) o[static_cast<size_t>(c) * p.M] = to_bf16(__uint_as_float(v[c]));
            } else {
#pragma unroll
                for (int c = 0; c < 16; ++c) partial[(c0 + c) * kBlockM + q * 32 + lane] = __uint_as_float(v[c]);
            }
        }
        tc_fence_before_sync();
    }
    if (splits == 1) {
        __syncthreads();
        if (*abort_flag) drain_after_abort();
        if (warp == 1) {
            tc_fence_after_sync();
            tmem_dealloc(tmem_base, Cfg::kTmemCols);
        }
        return;
    }
    cluster_sync_all();                                       // every rank's partial tile is in place

    // Token rows are dealt round-robin to the ranks.  One warp sums one token row at a time: a
    // lane owns four consecutive features, fetches its 16 bytes from every rank's partial tile
    // (all S loads in flight together) and adds them in rank order.
    if (!*abort_flag) {
        const int ntok = min(p.Ntok, BLOCK_N);
        const int mine = ntok > rank ? (ntok - rank + splits - 1) / splits : 0;
        const uint32_t my_partial = smem_u32(partial);
        for (int i = warp; i < mine; i += kGemmThreads / 32) {
            const int n = rank + i * splits;
            const uint32_t off = my_partial + static_cast<uint32_t>(n * kBlockM + lane * 4) * 4u;
            float4 v[8];
#pragma unroll
            for (int s = 0; s < 8; ++s)
                if (s < splits) v[s] = ld_shared_cluster_v4(mapa_shared(off, s));
            float4 acc = v[0];
#pragma unroll
            for (int s = 1; s < 8; ++s)
                if (s < splits) { acc.x += v[s].x; acc.y += v[s].y; acc.z += v[s].z; acc.w += v[s].w; }
            uint2 o;
            o.x = pack_bf16x2(acc.x, acc.y);
            o.y = pack_bf16x2(acc.z, acc.w);
            const int m = m_blk * kBlockM + lane * 4;
            if (m < p.M) *reinterpret_cast<uint2*>(p.out + static_cast<size_t>(n) * p.M + m) = o;
        }
    }
    if (*abort_flag) drain_after_abort();
    cluster_sync_all();                                       // peers may still be reading this CTA's tile
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, Cfg::kTmemCols);
    }
}

}  // namespace slope
