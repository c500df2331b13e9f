// General N:M magnitude pruning to masked-dense matrices (emulation of N:M sparsity for
// accuracy studies, and the matrices A^R and A^{R,C} of Lemma 1 / Eq. (sparsity_ratio)).
// HBM-bound streaming kernels: every element is read once and written once.
//
// Selection rule, as for 2:4: in a group of M entries keep the N of largest 15-bit bf16
// magnitude, the lower position winning ties: u beats t when key[u] > key[t], or
// key[u] == key[t] and u < t, and entry t is kept iff fewer than N entries beat it.
#pragma once
#include "ptx.cuh"

namespace slope {

// Two groups at once: entry i of one in the low and of the other in the high half-word of E[i].  These kernels are
// bound by the integer / logic pipe (64 lanes per clock and SM) long before HBM unless the selection costs
// few instructions per entry.  Magnitudes have 15 bits, so (E[i] | 0x8000) - |E[j]| leaves "i beats j" (i < j,
// ties to the lower position) in bits 15 and 31: one instruction per pair of entries for both groups; a
// byte permute replicates the two signs over their half-words, and three-operand adds of these masks count
// how often an entry is beaten.  A mask of the low half-word is 65536 - 1: every -1 below comes with a +1
// above, which a multiplication by 65537 takes out again.  Twice the count less (2n - 1) is odd, so the borrow
// that a negative low half-word takes from the high one never changes the high one's sign.
// 4096 x 4096, us, first / second pass, before (32-bit compares, adds and sorting networks, one group at a time) ->
// now: 1:2 12.3 / 15.3 -> 12.0 / 12.3, 2:4 14.2 / 16.8 -> 12.0 / 12.8, 2:8 18.6 / 23.7 -> 12.5 / 13.7, 4:16 22.2 /
// 37.5 -> 17.5 / 23.3 (10.6 / 10.9 at the HBM rate).
// keep[i]: 0xFFFF in the half-words of the groups that keep entry i.
template <int M>
__device__ __forceinline__ void keep_n_of_m_packed(const uint32_t (&E)[M], int n, uint32_t (&keep)[M]) {
    static_assert(M == 2 || M == 4 || M == 8 || M == 16, "group size");
    uint32_t cnt[M] = {};                                  // (entries after i that i beats) - (entries before i that beat it)
#pragma unroll
    for (int i = 0; i < M; i += 2) {
#pragma unroll
        for (int j = i; j < M; j += 2) {                   // 2 x 2 blocks of pairs: one three-operand add per pair
            uint32_t c[2][2] = {};
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b)
                    if (i + a < j + b) c[a][b] = prmt((E[i + a] | 0x80008000u) - (E[j + b] & 0x7FFF7FFFu), 0u, 0xBB99u);
            cnt[i] -= c[0][0] + c[0][1];
            cnt[i + 1] -= c[1][0] + c[1][1];
            cnt[j] += c[0][0] + c[1][0];
            cnt[j + 1] += c[0][1] + c[1][1];
        }
    }
#pragma unroll
    for (int i = 0; i < M; ++i)
        keep[i] = prmt(static_cast<uint32_t>(2 * (M - 1 - i) + 1 - 2 * n) * 0x10001u - 0x20002u * cnt[i], 0u, 0xBB99u);
}

// First pass: groups of M consecutive entries along a row.  A thread owns chunks of 16 consecutive entries (two 16-byte
// loads): one, or for M = 16 two, 32 chunks apart, since the selection works on pairs of groups.  It writes
// them back with the pruned entries zeroed (+0) and, when asked, a chunk's 16 mask bits (bit j % 8 of
// byte j / 8: one aligned 16-bit store).  n_chunks is a multiple of 64.  `out` may be `W` itself.
template <int M>
__global__ void __launch_bounds__(256)
prune_nm_kernel(const uint4* W, size_t n_chunks, int n, uint4* out, uint16_t* __restrict__ mask) {
    constexpr int kChunks = M == 16 ? 2 : 1;
    griddep_stream(8);
    const size_t stride = static_cast<size_t>(gridDim.x) * blockDim.x;
    for (size_t t0 = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; t0 < n_chunks / kChunks; t0 += stride) {
        const size_t c = kChunks == 1 ? t0 : (t0 & ~size_t(31)) * 2 + (t0 & 31);
        uint32_t w[8 * kChunks];
#pragma unroll
        for (int k = 0; k < kChunks; ++k) {
            const uint4 a = ld_stream_v4(W + 2 * (c + 32 * k)), b = ld_stream_v4(W + 2 * (c + 32 * k) + 1);
            w[8 * k] = a.x; w[8 * k + 1] = a.y; w[8 * k + 2] = a.z; w[8 * k + 3] = a.w;
            w[8 * k + 4] = b.x; w[8 * k + 5] = b.y; w[8 * k + 6] = b.z; w[8 * k + 7] = b.w;
        }
        uint32_t kept[2] = {0, 0};
#pragma unroll
        for (int g = 0; g < 16 * kChunks / M; g += 2) {        // groups g and g + 1: words wa[0 .. M/2) and wb[0 .. M/2)
            uint32_t *wa = w + g * (M / 2), *wb = wa + M / 2, E[M], m[M], bits = 0;
#pragma unroll
            for (int k = 0; k < M / 2; ++k) {
                E[2 * k] = prmt(wa[k], wb[k], 0x5410u);
                E[2 * k + 1] = prmt(wa[k], wb[k], 0x7632u);
            }
            keep_n_of_m_packed<M>(E, n, m);
#pragma unroll
            for (int k = 0; k < M / 2; ++k) {
                wa[k] &= prmt(m[2 * k], m[2 * k + 1], 0x5410u);
                wb[k] &= prmt(m[2 * k], m[2 * k + 1], 0x7632u);
            }
#pragma unroll
            for (int t = 0; t < M; ++t) bits |= m[t] & (0x00010001u << t);
            if (M == 16) {
                kept[0] = bits & 0xFFFFu;
                kept[1] = bits >> 16;
            } else {
                kept[0] |= ((bits & 0xFFFFu) | ((bits >> 16) << (M & 15))) << (g * M);
            }
        }
#pragma unroll
        for (int k = 0; k < kChunks; ++k) {
            __stcs(out + 2 * (c + 32 * k), make_uint4(w[8 * k], w[8 * k + 1], w[8 * k + 2], w[8 * k + 3]));
            __stcs(out + 2 * (c + 32 * k) + 1, make_uint4(w[8 * k + 4], w[8 * k + 5], w[8 * k + 6], w[8 * k + 7]));
            if (mask != nullptr) mask[c + 32 * k] = static_cast<uint16_t>(kept[k]);
        }
    }
}

// Second pass: groups of M consecutive entries down a column of the already pruned matrix (entries outside the
// first-pass mask count as zeros).  Groups run down the columns, so a word of a row (two adjacent columns) is
// a packed pair as it is.  A thread owns M rows x 8 columns (M <= 8: 16-byte loads at row pitch, a warp reads
// 512 contiguous bytes of a row) or 16 rows x 4 columns (8-byte loads; two neighbours share a mask byte), which
// keeps the registers of the 16-row pattern under 128; output in the same orientation.  mask2 = kept by
// both passes.  `out` may be `W` itself.
// (Ordinary loads through unrestricted pointers: they stay behind griddep_stream, and unlike volatile ones the
// compiler may place them, without which the kernel spills.)
template <int WORDS>
__device__ __forceinline__ void load_words(const uint32_t* p, uint32_t (&w)[WORDS]) {
    if constexpr (WORDS == 4) {
        const uint4 v = *reinterpret_cast<const uint4*>(p);
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    } else {
        const uint2 v = *reinterpret_cast<const uint2*>(p);
        w[0] = v.x; w[1] = v.y;
    }
}
template <int M>
__global__ void __launch_bounds__(256, M == 16 ? 2 : M == 8 ? 3 : 4)
double_prune_nm_kernel(const uint4* W, const uint8_t* mask1, int d_out, int d_in, int n, uint4* out, uint8_t* mask2) {
    constexpr int kWords = M == 16 ? 2 : 4;
    const int per_row = d_in / (2 * kWords);                   // threads per row: a multiple of 16, of 32 for M = 16
    const size_t total = static_cast<size_t>(d_out / M) * per_row;
    griddep_stream(M == 16 ? 2 : M == 8 ? 3 : 4);
    const size_t stride = static_cast<size_t>(gridDim.x) * blockDim.x;
    for (size_t idx = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; idx < total; idx += stride) {
        const size_t h = idx / per_row, c = idx % per_row;
        const size_t at = (h * M * per_row + c) * kWords, mask_at = h * M * (d_in / 8) + c * kWords / 4;
        const int first_bit = kWords == 4 ? 0 : 4 * (static_cast<int>(c) & 1);   // of this thread's columns in the mask byte
        const uint32_t* src = reinterpret_cast<const uint32_t*>(W) + at;
        uint32_t* dst = reinterpret_cast<uint32_t*>(out) + at;
        const size_t pitch = static_cast<size_t>(per_row) * kWords, mask_pitch = d_in / 8;
        uint32_t w[M][kWords], m1[M], sel[M];
#pragma unroll
        for (int t = 0; t < M; ++t) {
            load_words(src + t * pitch, w[t]);
            m1[t] = (mask1[mask_at + t * mask_pitch] >> first_bit) & (kWords == 4 ? 0xFFu : 0xFu);
            sel[t] = 0;
        }
#pragma unroll
        for (int q = 0; q < kWords; ++q) {
            uint32_t E[M], m[M];
#pragma unroll
            for (int t = 0; t < M; ++t) {
                // mask bits 2q and 2q + 1 over the half-words: pruned by the first pass -> +0
                // (one multiply for two shifts and an or: the shifted bytes do not overlap)
                const uint32_t z = m1[t] * ((1u << (15 - 2 * q)) + (1u << (30 - 2 * q)));
                E[t] = w[t][q] & prmt(z, 0u, 0xBB99u);
            }
            keep_n_of_m_packed<M>(E, n, m);
#pragma unroll
            for (int t = 0; t < M; ++t) {
                w[t][q] = E[t] & m[t];
                sel[t] |= m[t] & ((1u << (2 * q)) | (0x10000u << (2 * q + 1)));
            }
        }
#pragma unroll
        for (int t = 0; t < M; ++t) {
            uint32_t both = (sel[t] | (sel[t] >> 16)) & m1[t];
            if constexpr (kWords == 4) {
                __stcs(reinterpret_cast<uint4*>(dst + t * pitch), make_uint4(w[t][0], w[t][1], w[t][2], w[t][3]));
                if (mask2 != nullptr) mask2[mask_at + t * mask_pitch] = static_cast<uint8_t>(both);
            } else {
                __stcs(reinterpret_cast<uint2*>(dst + t * pitch), make_uint2(w[t][0], w[t][1]));
                both <<= first_bit;
                both |= __shfl_xor_sync(0xFFFFFFFFu, both, 1);                    // (whole warps run the loop)
                if (mask2 != nullptr && first_bit == 0) mask2[mask_at + t * mask_pitch] = static_cast<uint8_t>(both);
            }
        }
    }
}

// out = G where the mask bit is set, +0 elsewhere (a dense gradient restricted to a static
// N:M pattern).  A thread owns 16 consecutive entries; `out` may be `G` itself.
__global__ void __launch_bounds__(256)
apply_mask_kernel(const uint4* G, const uint16_t* __restrict__ mask, size_t n_chunks, uint4* out) {
    griddep_stream(8);
    const size_t stride = static_cast<size_t>(gridDim.x) * blockDim.x;
    for (size_t c = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; c < n_chunks; c += stride) {
        const uint4 a = ld_stream_v4(G + 2 * c), b = ld_stream_v4(G + 2 * c + 1);
        uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        const uint32_t keep = ld_u16(mask + c);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const uint32_t lo = (keep >> (2 * q)) & 1u ? 0x0000FFFFu : 0u;
            const uint32_t hi = (keep >> (2 * q + 1)) & 1u ? 0xFFFF0000u : 0u;
            w[q] &= lo | hi;
        }
        __stcs(out + 2 * c, make_uint4(w[0], w[1], w[2], w[3]));
        __stcs(out + 2 * c + 1, make_uint4(w[4], w[5], w[6], w[7]));
    }
}

// Number of element positions in which two bit masks differ (the per-iteration mask change
// that the comparison with dynamically re-selected masks plots).  16-byte loads, popcount of the
// XOR, one integer atomic per warp: the count is exact whatever the order.
__global__ void __launch_bounds__(256)
mask_difference_kernel(const uint4* __restrict__ a, const uint4* __restrict__ b, size_t n_vec,
                       unsigned long long* __restrict__ count) {
    unsigned int local = 0;
    const size_t stride = static_cast<size_t>(gridDim.x) * blockDim.x;
    for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n_vec; i += stride) {
        const uint4 x = __ldcs(a + i), y = __ldcs(b + i);
        local += __popc(x.x ^ y.x) + __popc(x.y ^ y.y) + __popc(x.z ^ y.z) + __popc(x.w ^ y.w);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) local += __shfl_xor_sync(0xFFFFFFFFu, local, o);
    if ((threadIdx.x & 31) == 0 && local != 0) atomicAdd(count, static_cast<unsigned long long>(local));
}

}  // namespace slope
