// The N:M step on eight consecutive saliency values, and how the kernels that stream a weight-shaped tensor cut it
// into work items.  Shared by the mask projection and the fused saliency kernel.
#pragma once

#include "crisp_internal.h"

namespace crisp {

constexpr int kM1Threads = 256;
constexpr int kM1ChunkK = 256;           // k-elements covered by one warp pass (32 lanes x 8)

// |s| as an order-preserving uint32 key: NaN -> 0, Inf -> FLT_MAX.
__device__ __forceinline__ uint32_t canonical_key(float s) {
    uint32_t u = __float_as_uint(s) & 0x7FFFFFFFu;
    if (u > 0x7F800000u) return 0u;
    if (u == 0x7F800000u) return 0x7F7FFFFFu;
    return u;
}

// |s| with NaN -> 0 and Inf -> FLT_MAX in two instructions: max(|s|, 0) drops a NaN (the maximum of a NaN and a
// number is the number), min(., FLT_MAX) caps infinity; -0 becomes +0, denormals pass unchanged.
__device__ __forceinline__ uint32_t canonical_bits(uint32_t u) {
    return __float_as_uint(fminf(fmaxf(fabsf(__uint_as_float(u)), 0.f), 3.402823466e+38f));
}

// Bit i of the result is set iff element i is among the N largest of its group of M
// (ties to the lower index).  M is 4 or 8; the 8 keys hold two groups or one.
// For i < j, element i beats element j iff key[i] >= key[j].
template <int M>
__device__ __forceinline__ uint32_t top_n_bits(const uint32_t key[8], int n) {
    uint32_t bits = 0u;
#pragma unroll
    for (int g = 0; g < 8 / M; ++g) {
        int rank[M];
#pragma unroll
        for (int i = 0; i < M; ++i) rank[i] = 0;
#pragma unroll
        for (int i = 0; i < M; ++i)
#pragma unroll
            for (int j = i + 1; j < M; ++j) {
                const int i_wins = key[g * M + i] >= key[g * M + j];
                rank[j] += i_wins;
                rank[i] += 1 - i_wins;
            }
#pragma unroll
        for (int i = 0; i < M; ++i) bits |= (rank[i] < n ? 1u : 0u) << (g * M + i);
    }
    return bits;
}

// Groups of 4: the six pairwise outcomes index a 64-entry table of keep masks (built per CTA for
// the layer's n by keep_mask_of_outcomes), which replaces the rank arithmetic.
__device__ __forceinline__ uint32_t outcomes4(const uint32_t *k) {
    return (uint32_t)(k[0] >= k[1]) | ((uint32_t)(k[0] >= k[2]) << 1) | ((uint32_t)(k[0] >= k[3]) << 2) |
           ((uint32_t)(k[1] >= k[2]) << 3) | ((uint32_t)(k[1] >= k[3]) << 4) | ((uint32_t)(k[2] >= k[3]) << 5);
}
__device__ __forceinline__ uint32_t keep_mask_of_outcomes(uint32_t o, int n) {
    const int w01 = o & 1, w02 = (o >> 1) & 1, w03 = (o >> 2) & 1, w12 = (o >> 3) & 1, w13 = (o >> 4) & 1,
              w23 = (o >> 5) & 1;
    const int r0 = (1 - w01) + (1 - w02) + (1 - w03);
    const int r1 = w01 + (1 - w12) + (1 - w13);
    const int r2 = w02 + w12 + (1 - w23);
    const int r3 = w03 + w13 + w23;
    return (uint32_t)(r0 < n) | ((uint32_t)(r1 < n) << 1) | ((uint32_t)(r2 < n) << 2) | ((uint32_t)(r3 < n) << 3);
}

constexpr int kM1Rows = 32;              // rows per work item of K-M1a / K-M1b (divides every block height)
constexpr int kM1RowsPerWarp = kM1Rows / (kM1Threads / 32);

// One work item = 32 rows x 256 k-elements.  Warp w takes rows 4w..4w+3 (all loads issued first); lane l owns
// the 8 elements at k = chunk*256 + 8*l of each row, so a lane stays inside one block column.  Items are dealt
// out to a grid of resident CTAs (grid-stride), chunk fastest, so that a CTA streams along rows.
struct M1Item { int64_t row0; int chunk; };
__device__ __forceinline__ M1Item m1_item(int64_t it, int chunks) {
    M1Item x;
    const int64_t rg = it / chunks;
    x.chunk = (int)(it - rg * chunks);
    x.row0 = rg * kM1Rows;
    return x;
}

}  // namespace crisp
