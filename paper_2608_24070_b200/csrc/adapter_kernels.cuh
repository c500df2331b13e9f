// The adapter's low-rank products on sm_100a: T = X L, dT = dY R^T, dL = X^T dT, dR = T^T dY.
//
// All four are D[M x N] = A[M x K] * B[N x K]^T with N = r <= 256: one operand (activations or
// output gradients) is large and read once, everything else is small.  What bounds them is the
// read of the large operand: HBM at training sizes, and at inference sizes the number of SMs that
// pull at the same time (a CTA takes in ~130 GB/s; 500 tokens are four 128-row tiles, which alone
// walked a reduction of 4096 in 12 us and one of 11008 in 28 us).  So
//   - a cluster of S CTAs splits the reduction of a tile; the partial tiles are summed in rank
//     order through distributed shared memory, so there is no workspace, no second launch, and
//     the result is deterministic;
//   - the column tile is 64, 128 or 256 wide: a wide one reads the large operand once whatever r
//     is, narrow ones bring more CTAs to a small problem;
//   - a CTA has an SM's shared memory to itself (deep ring) when a launch fits the machine that way,
//     otherwise two CTAs share it and overlap each other's set-up, drain and reduction.
// adapter_plan() weighs these by estimate.  Measured (us, cold, in a graph; 128-row tiles without a
// split and split-K partial sums in global memory before): T at 500 tokens, 4096 / 11008 wide, r = 64:
// 12.3 / 28.3 -> 6.2 / 8.6; dT + dL + dR at 8192 tokens, 5120 -> 13824, r = 128: 115 -> 92 (82 at the
// HBM peak); at 1000 tokens, 768 -> 2304, r = 256: 29.8 -> 13.4; T at 16384 x 4096, r = 256: 45 -> 36.
#pragma once
#include <type_traits>

#include "gemm_kernels.cuh"

namespace slope {

// Rows of a K-contiguous operand's box: no more than the matrix has.  An SM takes about one 128-byte row of any box per two clocks,
// inside the matrix or not; what the MMAs read behind the last row only reaches accumulator rows or columns that are
// never stored.
__host__ __device__ constexpr int adapter_box_rows(int rows, int tile) { return rows < tile ? rows : tile; }

struct AdapterProblem {
    int M, N, K;
    uint16_t* out;                // bf16 [M x N], or [N x M] when `transposed`
    int transposed;
};

template <int N_TILE>
struct AdapterCfg {
    static constexpr int kABytes = kBlockM * 128;                // 128 x 64 bf16 of the large operand
    static constexpr int kStageBytes = kABytes + N_TILE * 128;
    static constexpr int kMaxStages = 9;
    // The fp32 partial tile, reusing the stages: [row][column] with four floats of padding (lanes that
    // hold consecutive rows then store 16 bytes without bank conflicts), or [column][row] for an
    // output that is stored transposed.
    static constexpr int kPitch = N_TILE + 4;
    static constexpr int kPartialBytes = kBlockM * kPitch * 4;
    static constexpr int smem_bytes(int stages) { return stages * kStageBytes + 1024 + 1024; }
    // stages of a CTA that has the SM to itself / shares it with another one (0: does not fit)
    static constexpr int kDeep = (232448 - 2048) / kStageBytes < kMaxStages ? (232448 - 2048) / kStageBytes : kMaxStages;
    static constexpr int kShared = N_TILE > 128 ? 0 : (232448 / 2 - 1024 - 2048) / kStageBytes;
    static_assert(N_TILE == 64 || N_TILE == 128 || N_TILE == 256, "column tile = tensor memory columns");
    static_assert(kPartialBytes <= (kShared ? kShared : kDeep) * kStageBytes, "partial tile must fit in the stages");
};

// Sums the parked partial tiles of the SPLITS ranks in rank order and stores this rank's share.  A unit is
// four consecutive outputs (columns of a row, or rows of a column; both counts are multiples of
// four except the rows of a ragged token tile, which is never stored transposed).
template <int SPLITS, int PITCH>
__device__ __forceinline__ void adapter_reduce(const AdapterProblem& p, uint32_t base, int rank, int m_blk, int n0,
                                               int rows, int cols) {
    const int per_line = (p.transposed ? rows : cols) / 4, units = rows * cols / 4;
    const int pitch = p.transposed ? kBlockM : PITCH;
    const int step = SPLITS * kGemmThreads;
#pragma unroll (SPLITS <= 2 ? 4 : 2)
    for (int u = rank * kGemmThreads + threadIdx.x; u < units; u += step) {
        const int i = u / per_line, j = 4 * (u - i * per_line);
        const uint32_t off = base + static_cast<uint32_t>(i * pitch + j) * 4u;
        float4 v[SPLITS];
#pragma unroll
        for (int s = 0; s < SPLITS; ++s)
            v[s] = SPLITS == 1 ? ld_shared_v4(off) : ld_shared_cluster_v4(mapa_shared(off, s));
        float4 acc = v[0];
#pragma unroll
        for (int s = 1; s < SPLITS; ++s) { acc.x += v[s].x; acc.y += v[s].y; acc.z += v[s].z; acc.w += v[s].w; }
        const size_t at = p.transposed ? static_cast<size_t>(n0 + i) * p.M + m_blk * kBlockM + j
                                       : static_cast<size_t>(m_blk * kBlockM + i) * p.N + n0 + j;
        *reinterpret_cast<uint2*>(p.out + at) = make_uint2(pack_bf16x2(acc.x, acc.y), pack_bf16x2(acc.z, acc.w));
    }
}

// Weights of the few-token forward that a T launch is the producer of.  That forward's CTAs come up only when T has let them in, i.e.
// when everything before the pair is complete, and their first loads 1 to 1.5 us later, in which HBM would have nothing to do;
// `blocks` further CTAs of the T launch, on SMs that T does not need, ask L2 for the first k-blocks of every slice meanwhile.
// (4 linears of a block of width 4096 / 11008, r = 64, 8 tokens, us: none 56.96, 3 k-blocks 55.40, 6 55.66, 12 58.19.)
constexpr int kPairPrefetchBlocks = 3;     // k-blocks of a slice
struct WeightPrefetch {
    const uint8_t *vals, *meta;   // compressed values [M x K/2] and their metadata
    int K, splits, slices;        // K-slices of a 128-row slab; slices of all slabs
    int blocks;                   // at the end of the grid, whole clusters; 0: none
};
__device__ __forceinline__ void prefetch_weights(const WeightPrefetch& w, int block) {
    const int num_kb = w.K / 128, kb_per = (num_kb + w.splits - 1) / w.splits;
    for (int slice = block; slice < w.slices; slice += w.blocks) {
        const int slab = slice / w.splits, kb0 = slice % w.splits * kb_per;
        const int n = min(kPairPrefetchBlocks, min(num_kb, kb0 + kb_per) - kb0);
        const uint8_t* v = w.vals + static_cast<size_t>(slab) * kBlockM * w.K + kb0 * 128;
        for (int i = threadIdx.x; i < kBlockM * n; i += kGemmThreads) prefetch_l2(v + static_cast<size_t>(i / n) * w.K + i % n * 128);
        const uint8_t* m = w.meta + (static_cast<size_t>(slab) * num_kb + kb0) * 2048;
        for (int i = threadIdx.x; i < 16 * n; i += kGemmThreads) prefetch_l2(m + i * 128);
    }
}

struct NoPrefetch {};                      // (launches without such CTAs do not pay for the test)

template <bool A_MN, bool B_MN, int N_TILE, typename Prefetch>
__global__ void __launch_bounds__(kGemmThreads, 2)
adapter_gemm_kernel(const __grid_constant__ CUtensorMap tmA0, const __grid_constant__ CUtensorMap tmB0,
                    const AdapterProblem p0, const __grid_constant__ CUtensorMap tmA1,
                    const __grid_constant__ CUtensorMap tmB1, const AdapterProblem p1, const int stages,
                    const int pdl_mode, const Prefetch next) {
    if constexpr (std::is_same<Prefetch, WeightPrefetch>::value) {
        if (blockIdx.x >= gridDim.x - next.blocks) {
            griddep_wait();
            griddep_launch_dependents();
            prefetch_weights(next, blockIdx.x - (gridDim.x - next.blocks));
            return;
        }
    }
    // One cluster per tile of 128 rows x N_TILE columns, column tiles of a row tile next to each other.  Up to
    // two problems with the same N and K share a launch (p1.M == 0: only one): the row tiles
    // [0, tiles0) belong to problem 0, the rest to problem 1.
    using Cfg = AdapterCfg<N_TILE>;
    __shared__ uint64_t full_bar[Cfg::kMaxStages], empty_bar[Cfg::kMaxStages], tfull_bar[1];
    __shared__ uint32_t tmem_slot[1];
    __shared__ int abort_word;
    volatile int* abort_flag = &abort_word;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int splits = static_cast<int>(cluster_nctarank());
    const int rank = static_cast<int>(cluster_ctarank());
    const int col_tiles = (p0.N + N_TILE - 1) / N_TILE;
    const int tile = blockIdx.x / splits;
    int m_blk = tile / col_tiles;
    const int n0 = (tile - m_blk * col_tiles) * N_TILE;
    const int tiles0 = (p0.M + kBlockM - 1) / kBlockM;
    const bool second = m_blk >= tiles0;
    if (second) m_blk -= tiles0;
    const AdapterProblem& p = second ? p1 : p0;
    const CUtensorMap* tmA = second ? &tmA1 : &tmA0;
    const CUtensorMap* tmB = second ? &tmB1 : &tmB0;
    const int cols = min(N_TILE, p.N - n0);                                  // a multiple of 16
    const int all_kb = (p.K + 63) / 64;
    const int kb_per = (all_kb + splits - 1) / splits;
    const int kb0 = min(all_kb, rank * kb_per), num_kb = min(all_kb, kb0 + kb_per) - kb0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
        mbar_init(&tfull_bar[0], 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, N_TILE);
        tmem_relinquish();
    }
    if (warp == 0 && elect_one()) {
        tma_prefetch_desc(tmA);
        tma_prefetch_desc(tmB);
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    // Programmatic dependent launch, as in the few-token kernel: the producer of a fused pair
    // (pdl_mode 1) waits first, so that its dependent may rely on all earlier work.  As the consumer
    // of such a pair (pdl_mode 2: dR and dL behind dT) only problem 1 reads what the producer writes;
    // the CTAs of problem 0 run beside it.
    if (pdl_mode == 1) {
        griddep_wait();
        griddep_launch_dependents();
    } else {
        griddep_launch_dependents();
        if (pdl_mode == 0 || second) griddep_wait();
    }

    if (warp == 0) {
        if (elect_one()) {
            PipeState ps;
            const int chunks = (cols + 63) / 64;                             // chunks of 64 columns past N are not loaded
            const uint32_t stage_tx = 128 * ((A_MN ? kBlockM : adapter_box_rows(p.M, kBlockM)) +
                                             (B_MN ? 64 * chunks : adapter_box_rows(p.N, N_TILE)));
            for (int i = 0; i < num_kb; ++i) {
                if (!mbar_wait(&empty_bar[ps.stage], ps.phase ^ 1u, abort_flag)) break;
                uint8_t* sA = smem + ps.stage * Cfg::kStageBytes;
                uint8_t* sB = sA + Cfg::kABytes;
                uint64_t* bar = &full_bar[ps.stage];
                const int k0 = (kb0 + i) * 64;
                mbar_expect_tx(bar, stage_tx);
                if (A_MN) {
                    tma_load_2d(sA, tmA, bar, m_blk * kBlockM, k0);
                    tma_load_2d(sA + 8192, tmA, bar, m_blk * kBlockM + 64, k0);
                } else {
                    tma_load_2d(sA, tmA, bar, k0, m_blk * kBlockM);
                }
                if (B_MN) {
                    for (int h = 0; h < chunks; ++h) tma_load_2d(sB + h * 8192, tmB, bar, n0 + h * 64, k0);
                } else {
                    tma_load_2d(sB, tmB, bar, k0, n0);
                }
                ps.advance(stages);
            }
        }
    } else if (warp == 1) {
        if (elect_one()) {
            const uint32_t idesc = make_idesc_bf16(kBlockM, cols, A_MN, B_MN, false);
            PipeState ps;
            bool ok = true;
            for (int i = 0; i < num_kb; ++i) {
                if (!mbar_wait(&full_bar[ps.stage], ps.phase, abort_flag)) { ok = false; break; }
                tc_fence_after_sync();
                const uint32_t sA = smem_u32(smem + ps.stage * Cfg::kStageBytes);
                const uint32_t sB = sA + Cfg::kABytes;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint64_t ad = A_MN ? make_smem_desc(sA + j * 2048, 8192, 1024, kSwizzle128B)
                                             : make_smem_desc(sA + j * 32, 16, 1024, kSwizzle128B);
                    const uint64_t bd = B_MN ? make_smem_desc(sB + j * 2048, 8192, 1024, kSwizzle128B)
                                             : make_smem_desc(sB + j * 32, 16, 1024, kSwizzle128B);
                    umma_bf16(tmem_base, ad, bd, idesc, (i | j) != 0 ? 1u : 0u);
                }
                umma_commit(&empty_bar[ps.stage]);
                ps.advance(stages);
            }
            if (ok) umma_commit(&tfull_bar[0]);
        }
    }

    // ---------------------------------------------------------------- drain and reduction
    // The fp32 partial tile is parked in shared memory (the stages are free once the last MMA has
    // completed; a rank without a k-block contributes zeros); after a cluster barrier the ranks share
    // the sums.  A wide tile that is not split goes the same way: stores straight from tensor memory
    // touch a row per lane, which costs the store unit 32 times the accesses (a 64-column tile is
    // through sooner without the detour).
    float* partial = reinterpret_cast<float*>(smem);
    const int rows = min(kBlockM, p.M - m_blk * kBlockM);
    const bool direct = N_TILE == 64 && splits == 1 && !p.transposed;
    if (warp >= 2) {
        const int q = warp & 3;
        bool ok = num_kb > 0;
        if (ok) ok = mbar_wait(&tfull_bar[0], 0u, abort_flag);
        tc_fence_after_sync();
        const uint32_t t_row = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
        const int row = q * 32 + lane;
        if (q * 32 < rows) {
#pragma unroll 1
            for (int c0 = 0; c0 < cols; c0 += 16) {
                uint32_t v[16];
                if (ok) {
                    tmem_ld_16(t_row + c0, v);
                    tmem_ld_wait();
                } else {
#pragma unroll
                    for (int c = 0; c < 16; ++c) v[c] = 0u;
                }
                if (direct) {
                    if (row < rows) {
                        uint4* dst = reinterpret_cast<uint4*>(p.out + static_cast<size_t>(m_blk * kBlockM + row) * p.N + n0 + c0);
                        uint32_t w[8];
#pragma unroll
                        for (int c = 0; c < 8; ++c) w[c] = pack_bf16x2(__uint_as_float(v[2 * c]), __uint_as_float(v[2 * c + 1]));
                        dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
                        dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
                    }
                } else if (!p.transposed) {
                    uint4* dst = reinterpret_cast<uint4*>(partial + row * Cfg::kPitch + c0);
#pragma unroll
                    for (int c = 0; c < 4; ++c) dst[c] = make_uint4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
                } else {
#pragma unroll
                    for (int c = 0; c < 16; ++c) partial[(c0 + c) * kBlockM + row] = __uint_as_float(v[c]);
                }
            }
        }
        tc_fence_before_sync();
    }
    __syncthreads();
    if (splits > 1) cluster_sync_all();                       // every rank's partial tile is in place

    if (!direct && !*abort_flag) {
        const uint32_t base = smem_u32(partial);
        switch (splits) {
            case 2: adapter_reduce<2, Cfg::kPitch>(p, base, rank, m_blk, n0, rows, cols); break;
            case 4: adapter_reduce<4, Cfg::kPitch>(p, base, rank, m_blk, n0, rows, cols); break;
            case 8: adapter_reduce<8, Cfg::kPitch>(p, base, rank, m_blk, n0, rows, cols); break;
            default: adapter_reduce<1, Cfg::kPitch>(p, base, rank, m_blk, n0, rows, cols); break;
        }
    }
    if (*abort_flag) drain_after_abort();
    if (splits > 1) cluster_sync_all();                       // peers may still be reading this CTA's tile
    else __syncthreads();
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, N_TILE);
    }
}

}  // namespace slope
