// Mask projection kernels: saliency -> hybrid (block + N:M) mask.
//
// Algorithm 1 of the paper, restricted to one layer with the block keep count given:
//   K-M1a per group of M: keep the N largest (fine-grained N:M step), and the layer-wide maximum
//         of the canonical saliency (it sets the fixed-point scale): one pass over S from HBM
//   K-M1b block scores s_j = sum |T_w| as exact fixed-point integers: second pass over S, which
//         for layers up to the size of L2 is served from there
//   K-M2  per row of the block grid: keep the kkeep highest-scored blocks and clear the
//         bits of the pruned ones (blocks keep their positions)
// Coalesced 32-byte-per-lane accesses; K-M1a is bound by HBM bandwidth.
#include <atomic>

#include "crisp_internal.h"
#include "mask_common.cuh"

namespace crisp {

namespace {

constexpr int kScoreFractionBits = 40;
constexpr int kMaxDevices = 64;

// Raw bits of eight consecutive saliency values; the caller guarantees row < rows, k0 + 8 <= k and
// 16-byte alignment.  Kept free of branches so that several of these can be in flight per lane.
__device__ __forceinline__ void load8_raw(const float *s, int64_t ld, int64_t row, int64_t k0, uint32_t key[8]) {
    const uint4 *p = reinterpret_cast<const uint4 *>(s + row * ld + k0);
    const uint4 a = p[0], b = p[1];
    key[0] = a.x; key[1] = a.y; key[2] = a.z; key[3] = a.w;
    key[4] = b.x; key[5] = b.y; key[6] = b.z; key[7] = b.w;
}
// Eight consecutive saliency values of one row, zero beyond the matrix.
__device__ __forceinline__ void load8(const float *s, int64_t ld, int rows, int k, int64_t row, int64_t k0, bool vec_ok,
                                      uint32_t key[8]) {
    if (row >= rows || k0 >= k) {
#pragma unroll
        for (int i = 0; i < 8; ++i) key[i] = 0u;
        return;
    }
    const float *p = s + row * ld + k0;
    if (vec_ok && k0 + 8 <= k) {
        const float4 a = *reinterpret_cast<const float4 *>(p);
        const float4 b = reinterpret_cast<const float4 *>(p)[1];
        key[0] = canonical_key(a.x); key[1] = canonical_key(a.y);
        key[2] = canonical_key(a.z); key[3] = canonical_key(a.w);
        key[4] = canonical_key(b.x); key[5] = canonical_key(b.y);
        key[6] = canonical_key(b.z); key[7] = canonical_key(b.w);
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) key[i] = (k0 + i < k) ? canonical_key(p[i]) : 0u;
    }
}

// Exponent of a positive finite float given by its bits (ilogb), denormals included.
__device__ __forceinline__ int key_exponent(uint32_t key) {
    const int e = (int)(key >> 23);
    return e ? e - 127 : (31 - __clz(key)) - 149;
}

// floor(value * 2^(40 - e_max)) for a non-negative finite float given by its bits, in integer
// arithmetic: the mantissa shifted by the exponent difference (exact, no rounding mode involved).
__device__ __forceinline__ unsigned long long fixed_point_score(uint32_t key, int e_max) {
    const int e = (int)(key >> 23);
    const uint32_t mant = e ? ((key & 0x7FFFFFu) | 0x800000u) : key;           // value = mant * 2^(max(e,1) - 150)
    const int sh = max(e, 1) - 150 + kScoreFractionBits - e_max;                 // <= 17 because value <= layer maximum
    const uint32_t down = mant >> min(max(-sh, 0), 31);                          // mant < 2^24: shifts >= 24 give 0
    const int up = max(sh, 0);                                                   // only one of the two shifts is non-zero
    return ((unsigned long long)__funnelshift_l(down, 0u, up) << 32) | (unsigned long long)(down << up);
}

// The 8 canonical keys of the lane's elements of row `row` (zero beyond the matrix).  kCap = false leaves infinities in.
template <bool kCap = true>
__device__ __forceinline__ void m1_load_rows(const float *s, int64_t ld, const Geometry &g, bool vec_ok,
                                             const M1Item &x, int warp, int64_t k0, uint32_t key[kM1RowsPerWarp][8]) {
    if (vec_ok && x.row0 + kM1Rows <= g.rows && (int64_t)(x.chunk + 1) * kM1ChunkK <= g.k) {   // interior item
#pragma unroll
        for (int i = 0; i < kM1RowsPerWarp; ++i) load8_raw(s, ld, x.row0 + warp * kM1RowsPerWarp + i, k0, key[i]);
#pragma unroll
        for (int i = 0; i < kM1RowsPerWarp; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j)
                key[i][j] = kCap ? canonical_bits(key[i][j]) : __float_as_uint(fmaxf(fabsf(__uint_as_float(key[i][j])), 0.f));
    } else {
#pragma unroll
        for (int i = 0; i < kM1RowsPerWarp; ++i)
            load8(s, ld, g.rows, g.k, x.row0 + warp * kM1RowsPerWarp + i, k0, vec_ok, key[i]);
    }
}

// K-M1a: the fine-grained N:M step (which does not depend on the score scale) and the layer maximum (which fixes
// the scale) in ONE pass over S, the pass that comes from HBM: per group of M the N largest are marked, a lane
// stores its eight mask bits as one byte, and the largest key goes to max_key (one atomic per CTA).
// find_max = false when the caller already knows the maximum.
template <int M>
__global__ void __launch_bounds__(kM1Threads)
group_bits_kernel(const float *s, int64_t ld, Geometry g, bool vec_ok, int64_t items, int chunks, bool find_max,
                  uint32_t *max_key, uint32_t *nm_bits) {
    __shared__ uint8_t s_keep[64];
    __shared__ uint32_t s_best[kM1Threads / 32];
    chain_kernels();
    if (M == 4 && threadIdx.x < 64) s_keep[threadIdx.x] = (uint8_t)keep_mask_of_outcomes(threadIdx.x, g.n);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t best = 0u;
    for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
        const M1Item x = m1_item(it, chunks);
        const int64_t k0 = (int64_t)x.chunk * kM1ChunkK + lane * 8;
        uint32_t key[kM1RowsPerWarp][8];
        m1_load_rows(s, ld, g, vec_ok, x, warp, k0, key);
        const bool in_kp = k0 < g.kp();
#pragma unroll
        for (int i = 0; i < kM1RowsPerWarp; ++i) {
            const int64_t row = x.row0 + warp * kM1RowsPerWarp + i;
            uint32_t bits;
            if constexpr (M == 4)
                bits = (uint32_t)s_keep[outcomes4(key[i])] | ((uint32_t)s_keep[outcomes4(key[i] + 4)] << 4);
            else
                bits = top_n_bits<M>(key[i], g.n);
            // the lane's eight bits are byte (k0 / 8) mod 4 of their little-endian mask word: a warp stores 32
            // consecutive bytes of the row
            if (in_kp) reinterpret_cast<uint8_t *>(nm_bits + row * g.wpr)[k0 >> 3] = (uint8_t)bits;
#pragma unroll
            for (int j = 0; j < 8; ++j) best = max(best, key[i][j]);
        }
    }
    if (find_max) {
        best = __reduce_max_sync(0xFFFFFFFFu, best);
        if (lane == 0) s_best[warp] = best;
        __syncthreads();
        if (threadIdx.x == 0) {
#pragma unroll
            for (int w = 1; w < kM1Threads / 32; ++w) best = max(best, s_best[w]);
            if (best) atomicMax(max_key, best);
        }
    }
}

// Two fp32 values in one 64-bit register and the packed fp32 instructions of sm_100 on them (one instruction
// per pair; each half is rounded as the scalar instruction would round it).
__device__ __forceinline__ uint64_t f32x2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float f32x2_sum(uint64_t v) {       // lo + hi
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
    return __fadd_rn(lo, hi);
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) { uint64_t r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) { uint64_t r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) { uint64_t r; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t add2_down(uint64_t a, uint64_t b) { uint64_t r; asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }

// floor(v) of fp32 values 0 <= v < 2^41, two at a time, without a float-to-integer conversion per element (those
// run at a fraction of the fp32 rate and were what bound this kernel): v = r + d with r = v rounded DOWN to a
// multiple of 2^20 (add 1.5 * 2^43 rounding toward minus infinity: the sum lies in [2^43, 2^44), where fp32 steps
// by 2^20; subtracting the constant again is exact) and d = v - r exact, 0 <= d < 2^20; floor(d) by the same device
// with 1.5 * 2^23, where fp32 steps by 1.  r and floor(d) are then added up in fp32 over the eight elements of a
// row, which is exact (r / 2^20 <= 2^21 each, floor(d) < 2^20 each), and converted once.
__device__ __forceinline__ void floor_parts2(uint64_t v, uint64_t &r, uint64_t &fd) {
    const uint64_t big = f32x2(13194139533312.f, 13194139533312.f);            // 1.5 * 2^43
    const uint64_t mid = f32x2(12582912.f, 12582912.f);                        // 1.5 * 2^23
    r = sub2(add2_down(v, big), big);
    fd = sub2(add2_down(sub2(v, r), mid), mid);
}

// The two largest of four values (as a pair; equal values count as often as they occur).
struct Two { float a, b; };
__device__ __forceinline__ Two top2_of4(float x0, float x1, float x2, float x3) {
    const float h0 = fmaxf(x0, x1), l0 = fminf(x0, x1), h1 = fmaxf(x2, x3), l1 = fminf(x2, x3);
    return Two{fmaxf(h0, h1), fmaxf(fminf(h0, h1), fmaxf(l0, l1))};
}

// K-M1b: the block scores s_j = sum |T_w| as exact fixed-point integers, once the scale is known.  Second pass
// over S (for layers that fit, out of L2, where K-M1a left it).  Warps are independent (no shared memory, no
// barrier): a lane adds floor(|s| * 2^(40 - e_max)) of its counted elements over its warp's four rows, the four lanes of a
// 32-element word add up (a mask word never straddles a block: block_k is a multiple of 32), and one lane per word adds the
// partial score to the block's 64-bit total with an atomic (integer addition: any order gives the same sum).
// Which elements count: TOP = 0, the N:M survivors, read back as the byte K-M1a stored, or all of them.  TOP = 1 or 2
// (score mode 0 and n = TOP): a group contributes the sum of its n largest values, whichever of equal ones the mask keeps,
// so the values themselves are selected with minima and maxima and only they are scaled and floored: half of the
// elements for 2:4, an eighth for 1:8.  Measured (4096 x 4096, 2:4, S of 64 MiB): 18.2 -> 14.4 us under ncu with a cold L2,
// 4.4 us off the mask phase in a stream; what is left is mostly the wait between an item's loads and the next item's.
template <int CAP, int M, int TOP>
__global__ void __launch_bounds__(kM1Threads)
block_score_kernel(const __grid_constant__ Batch<ScoreLayer, CAP> batch) {
    chain_kernels();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t unit = blockIdx.x; unit < batch.first[batch.n]; unit += gridDim.x) {
    const int l = batch.find(unit);
    const ScoreLayer &L = batch.layer[l];
    const Geometry &g = L.g;
    const float *s = L.s;
    const int64_t ld = L.ld;
    const uint32_t *nm_bits = L.nm_bits;
    const uint32_t mk = *L.max_key;
    if (!mk) continue;                                       // an all-zero layer: every score stays 0
    const int e_max = key_exponent(mk);
    // floor(value * 2^(40 - e_max)): when that power of two is an fp32 number, the product is exact
    // (value <= layer maximum, so it stays below 2^41)
    const int scale_exp = kScoreFractionBits - e_max;
    const bool float_scale = scale_exp >= -126 && scale_exp <= 127;
    const float scale = float_scale ? __uint_as_float((uint32_t)(127 + scale_exp) << 23) : 0.f;
        const M1Item x = m1_item(unit - batch.first[l], L.chunks);
        const int64_t k0 = (int64_t)x.chunk * kM1ChunkK + lane * 8;
        const int rt = (int)(x.row0 / g.bm);
        uint32_t key[kM1RowsPerWarp][8];
        m1_load_rows<TOP == 0>(s, ld, g, L.vec_ok != 0, x, warp, k0, key);
        const bool in_kp = k0 < g.kp();
        unsigned long long acc = 0ull;
        if (TOP != 0 && float_scale) {
            uint64_t r_sum = f32x2(0.f, 0.f), d_sum = r_sum;                     // exact for eight values: see floor_parts2
            auto count = [&](float a, float b) {
                uint64_t r, fd;
                floor_parts2(mul2(f32x2(fminf(a, 3.402823466e+38f), fminf(b, 3.402823466e+38f)), f32x2(scale, scale)), r, fd);
                r_sum = add2(r_sum, r);
                d_sum = add2(d_sum, fd);
            };
            auto flush = [&]() {
                acc += ((unsigned long long)__float2uint_rn(f32x2_sum(r_sum) * 9.5367431640625e-07f) << 20) +
                       (unsigned long long)__float2uint_rn(f32x2_sum(d_sum));
                r_sum = d_sum = f32x2(0.f, 0.f);
            };
            float best_before = 0.f;
#pragma unroll
            for (int i = 0; i < kM1RowsPerWarp; ++i) {
                float v[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(key[i][j]);
                const Two p = top2_of4(v[0], v[1], v[2], v[3]), q = top2_of4(v[4], v[5], v[6], v[7]);
                if constexpr (TOP == 2 && M == 4) {
                    count(p.a, p.b);
                    count(q.a, q.b);
                    if (i & 1) flush();
                } else if constexpr (TOP == 1 && M == 4) {
                    count(p.a, q.a);
                } else if constexpr (TOP == 2) {
                    count(fmaxf(p.a, q.a), fmaxf(fminf(p.a, q.a), fmaxf(p.b, q.b)));
                } else {
                    if (i & 1) count(best_before, fmaxf(p.a, q.a));
                    best_before = fmaxf(p.a, q.a);
                }
            }
            if (!(TOP == 2 && M == 4)) flush();
        } else if (float_scale) {
#pragma unroll
            for (int i = 0; i < kM1RowsPerWarp; ++i) {
                const int64_t row = x.row0 + warp * kM1RowsPerWarp + i;
                uint32_t counted = 0xFFu;
                if (g.score_mode == 0) counted = in_kp ? reinterpret_cast<const uint8_t *>(nm_bits + row * g.wpr)[k0 >> 3] : 0u;
                // an element that is not counted is multiplied by zero instead of by the scale: its parts are zero
                uint64_t r_sum = f32x2(0.f, 0.f), d_sum = r_sum;             // exact: see floor_parts2
#pragma unroll
                for (int j = 0; j < 8; j += 2) {
                    const uint64_t sc = f32x2((counted >> j) & 1u ? scale : 0.f, (counted >> (j + 1)) & 1u ? scale : 0.f);
                    uint64_t r, fd;
                    floor_parts2(mul2(f32x2(__uint_as_float(key[i][j]), __uint_as_float(key[i][j + 1])), sc), r, fd);
                    r_sum = add2(r_sum, r);
                    d_sum = add2(d_sum, fd);
                }
                acc += ((unsigned long long)__float2uint_rn(f32x2_sum(r_sum) * 9.5367431640625e-07f) << 20) +
                       (unsigned long long)__float2uint_rn(f32x2_sum(d_sum));
            }
        } else {
#pragma unroll
            for (int i = 0; i < kM1RowsPerWarp; ++i) {
                const int64_t row = x.row0 + warp * kM1RowsPerWarp + i;
                uint32_t counted = 0xFFu;
                if (g.score_mode == 0) counted = in_kp ? reinterpret_cast<const uint8_t *>(nm_bits + row * g.wpr)[k0 >> 3] : 0u;
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if ((counted >> j) & 1u) acc += fixed_point_score(canonical_bits(key[i][j]), e_max);
            }
        }
        acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 1);
        acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 2);
        // lanes that share a block column (block_k / 8 of them, 4, 8, 12 or 16): add up as far as the lane groups
        // of a power of two allow, then one atomic per group
        if (g.bk % 64 == 0) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 4);
        if (g.bk % 128 == 0) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 8);
        const int grp = g.bk % 128 == 0 ? 15 : (g.bk % 64 == 0 ? 7 : 3);
        if ((lane & grp) == 0 && in_kp && acc) {
            const int jb = (int)(k0 / g.bk);
            if (jb < g.nblk) atomicAdd(&L.score[(int64_t)rt * g.nblk + jb], acc);
        }
    }
}

// K-M2.  One CTA per 32 rows of a row tile.  Every CTA ranks its row tile's block scores (cheap)
// and clears the mask words of pruned blocks in its own 32 rows; the first CTA of a row tile also
// emits the kept columns in ascending order.
template <int CAP>
__global__ void __launch_bounds__(256)
block_select_kernel(const __grid_constant__ Batch<ScoreLayer, CAP> batch) {
    extern __shared__ unsigned long long sm[];
    chain_kernels();
    const int l = batch.find(blockIdx.x);
    const ScoreLayer &L = batch.layer[l];
    const Geometry &g = L.g;
    const unsigned long long *score = L.score;
    int32_t *blk_col = L.blk_col;
    uint32_t *nm_bits = L.nm_bits;
    unsigned long long *sc = sm;                                   // [nblk]
    int *kept = reinterpret_cast<int *>(sm + g.nblk);              // [nblk]
    __shared__ int s_warp_tot[8];
    __shared__ int s_base;
    const int cta = (int)(blockIdx.x - batch.first[l]), slabs = g.bm / 32;
    const int rt = cta / slabs, slab = cta - rt * slabs;
    for (int j = threadIdx.x; j < g.nblk; j += blockDim.x) sc[j] = score[(int64_t)rt * g.nblk + j];
    if (threadIdx.x == 0) s_base = 0;
    __syncthreads();
    for (int j = threadIdx.x; j < g.nblk; j += blockDim.x) {
        const unsigned long long mine = sc[j];
        int rank = 0;
        for (int t = 0; t < g.nblk; ++t) {
            const unsigned long long o = sc[t];
            rank += (o > mine) || (o == mine && t < j);
        }
        kept[j] = rank < g.kkeep;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (slab == 0) {
        // ascending compaction: block-wide exclusive scan over chunks of blockDim.x flags
        for (int j0 = 0; j0 < g.nblk; j0 += blockDim.x) {
            const int j = j0 + threadIdx.x;
            const int f = (j < g.nblk) ? kept[j] : 0;
            const uint32_t ballot = __ballot_sync(0xFFFFFFFFu, f);
            const int before = __popc(ballot & ((1u << lane) - 1u));
            if (lane == 0) s_warp_tot[warp] = __popc(ballot);
            __syncthreads();
            int warp_off = 0, tot = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
                if (w < warp) warp_off += s_warp_tot[w];
                tot += s_warp_tot[w];
            }
            if (f) blk_col[(int64_t)rt * g.kkeep + s_base + warp_off + before] = j;
            __syncthreads();
            if (threadIdx.x == 0) s_base += tot;
            __syncthreads();
        }
    }
    // final mask = group bits AND block kept: one warp per row, lanes stride over the row's words
    const int wpb = g.bk / 32;
    for (int r = warp; r < 32; r += 8) {
        uint32_t *row_words = nm_bits + ((int64_t)rt * g.bm + slab * 32 + r) * g.wpr;
        for (int wc = lane; wc < g.wpr; wc += 32)
            if (!kept[wc / wpb]) row_words[wc] = 0u;
    }
}

// The whole projection of a small layer in one launch: a cluster of up to eight CTAs, each with whole row tiles, so that all that
// crosses between them is the layer maximum.  Group bits and the maximum in a first pass over S, scores in a second (out of L1 and L2)
// summed in shared memory, then the selection: what the kernels above compute, from the same definitions.  What bounds it is instructions on
// one SM (some 250 for eight elements), and for the smallest layers the two passes' round trips.  A memset and three kernels in its place
// take the device 10 to 15 us and the host about as long.
constexpr int kSmallThreads = 1024, kSmallMaxBlocks = 512, kSmallCluster = 8;
template <int M>
__global__ void __launch_bounds__(kSmallThreads)
mask_small_kernel(const float *s, int64_t ld, Geometry g, bool vec_ok, bool max_known, uint32_t *max_key, unsigned long long *score,
                  uint32_t *nm_bits, int32_t *blk_col, int ctas) {
    __shared__ unsigned long long s_score[kSmallMaxBlocks];
    __shared__ uint32_t s_part[3][kSmallMaxBlocks];          // a score in pieces of 22 bits: 32-bit shared atomics are native, 64-bit ones a loop
    __shared__ int s_kept[kSmallMaxBlocks];
    __shared__ uint32_t s_best[kSmallThreads / 32];
    __shared__ uint32_t s_max;
    __shared__ uint8_t s_keep[64];
    chain_kernels();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, cta = blockIdx.x;
    if (M == 4 && tid < 64) s_keep[tid] = (uint8_t)keep_mask_of_outcomes(tid, g.n);
    __syncthreads();
    const int chunks = g.wpr * 4, units = g.bm * chunks;     // chunks of eight elements: of a row, of a row tile
    // a thread takes every kSmallThreads-th chunk of a row tile: (row, chunk) of the first, and the step
    const int r_first = tid / chunks, c_first = tid - r_first * chunks, r_step = kSmallThreads / chunks, c_step = kSmallThreads - r_step * chunks;
    auto load = [&](int64_t row, int c, uint32_t (&key)[8]) {
        if (vec_ok && row < g.rows && 8 * c + 8 <= g.k) {
            load8_raw(s, ld, row, 8 * c, key);
#pragma unroll
            for (int j = 0; j < 8; ++j) key[j] = canonical_bits(key[j]);
        } else {
            load8(s, ld, g.rows, g.k, row, 8 * c, vec_ok, key);
        }
    };
    // group bits and the maximum
    uint32_t best = 0u;
    for (int rt = cta; rt < g.nrt; rt += ctas)
        for (int u = tid, r = r_first, c = c_first; u < units; u += kSmallThreads) {
            const int64_t row = (int64_t)rt * g.bm + r;
            uint32_t key[8];
            load(row, c, key);
            uint32_t bits;
            if constexpr (M == 4) bits = (uint32_t)s_keep[outcomes4(key)] | ((uint32_t)s_keep[outcomes4(key + 4)] << 4);
            else bits = top_n_bits<M>(key, g.n);
            reinterpret_cast<uint8_t *>(nm_bits + row * g.wpr)[c] = (uint8_t)bits;
#pragma unroll
            for (int j = 0; j < 8; ++j) best = max(best, key[j]);
            r += r_step; c += c_step;
            if (c >= chunks) { c -= chunks; ++r; }
        }
    best = __reduce_max_sync(0xFFFFFFFFu, best);
    if (lane == 0) s_best[warp] = best;
    __syncthreads();
    if (warp == 0) {
        best = __reduce_max_sync(0xFFFFFFFFu, s_best[lane]);
        if (lane == 0) s_max = best;
    }
    if (ctas > 1) {
        cluster_arrive();
        cluster_wait();
        best = lane < ctas ? lds32_peer(peer_address((uint32_t)__cvta_generic_to_shared(&s_max), (uint32_t)lane)) : 0u;
    } else {
        __syncthreads();
        best = s_max;
    }
    best = max_known ? *max_key : __reduce_max_sync(0xFFFFFFFFu, best);
    if (!max_known && cta == 0 && tid == 0) *max_key = best;
    const int e_max = best ? key_exponent(best) : 0, scale_exp = kScoreFractionBits - e_max;
    const bool float_scale = scale_exp >= -126 && scale_exp <= 127;
    const float scale = float_scale ? __uint_as_float((uint32_t)(127 + scale_exp) << 23) : 0.f;
    for (int rt = cta; rt < g.nrt; rt += ctas) {
        // block scores
        for (int j = tid; j < g.nblk; j += kSmallThreads) s_part[0][j] = s_part[1][j] = s_part[2][j] = 0u;
        __syncthreads();
        for (int u0 = 0, r = r_first, c = c_first; u0 < units; u0 += kSmallThreads) {        // (chunks of a row come in fours, so the lanes of a mask word stay together)
            const int64_t row = (int64_t)rt * g.bm + r;
            unsigned long long acc = 0ull;
            if (u0 + tid < units && best) {
                uint32_t key[8];
                load(row, c, key);
                uint32_t counted = 0xFFu;
                if (g.score_mode == 0) counted = reinterpret_cast<const uint8_t *>(nm_bits + row * g.wpr)[c];       // (this thread's own byte)
                if (float_scale) {                           // (as in block_score_kernel)
                    uint64_t r_sum = f32x2(0.f, 0.f), d_sum = r_sum;
#pragma unroll
                    for (int j = 0; j < 8; j += 2) {
                        uint64_t whole, part;
                        floor_parts2(mul2(f32x2(__uint_as_float(key[j]), __uint_as_float(key[j + 1])),
                                          f32x2((counted >> j) & 1u ? scale : 0.f, (counted >> (j + 1)) & 1u ? scale : 0.f)), whole, part);
                        r_sum = add2(r_sum, whole);
                        d_sum = add2(d_sum, part);
                    }
                    acc = ((unsigned long long)__float2uint_rn(f32x2_sum(r_sum) * 9.5367431640625e-07f) << 20) + (unsigned long long)__float2uint_rn(f32x2_sum(d_sum));
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if ((counted >> j) & 1u) acc += fixed_point_score(key[j], e_max);
                }
            }
            acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 1);
            acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 2);
            if (g.bk % 64 == 0) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 4);
            if (g.bk % 128 == 0) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 8);
            // (at most 384 such sums make a block, each below 2^48: no piece overflows)
            if ((lane & (g.bk % 128 == 0 ? 15 : g.bk % 64 == 0 ? 7 : 3)) == 0 && acc) {
                const int j = 8 * c / g.bk;
                atomicAdd(&s_part[0][j], (uint32_t)acc & 0x3FFFFFu);
                atomicAdd(&s_part[1][j], (uint32_t)(acc >> 22) & 0x3FFFFFu);
                atomicAdd(&s_part[2][j], (uint32_t)(acc >> 44));
            }
            r += r_step; c += c_step;
            if (c >= chunks) { c -= chunks; ++r; }
        }
        __syncthreads();
        for (int j = tid; j < g.nblk; j += kSmallThreads)
            s_score[j] = (unsigned long long)s_part[0][j] + ((unsigned long long)s_part[1][j] << 22) + ((unsigned long long)s_part[2][j] << 44);
        __syncthreads();
        // selection
        for (int j = tid; j < g.nblk; j += kSmallThreads) {
            const unsigned long long mine = s_score[j];
            int rank = 0;
            for (int t = 0; t < g.nblk; ++t) rank += s_score[t] > mine || (s_score[t] == mine && t < j);
            s_kept[j] = rank < g.kkeep;
            score[(int64_t)rt * g.nblk + j] = mine;
        }
        __syncthreads();
        if (warp == 0) {                                     // kept columns in ascending order
            int base = 0;
            for (int j0 = 0; j0 < g.nblk; j0 += 32) {
                const int f = j0 + lane < g.nblk ? s_kept[j0 + lane] : 0;
                const uint32_t ballot = __ballot_sync(0xFFFFFFFFu, f);
                if (f) blk_col[(int64_t)rt * g.kkeep + base + __popc(ballot & ((1u << lane) - 1u))] = j0 + lane;
                base += __popc(ballot);
            }
        }
        const int wpb = g.bk / 32;
        for (int i = tid; i < g.bm * g.wpr; i += kSmallThreads)
            if (!s_kept[i % g.wpr / wpb]) nm_bits[(int64_t)rt * g.bm * g.wpr + i] = 0u;
        __syncthreads();                                     // (the scores are cleared for the next row tile)
    }
    if (ctas > 1) {                                          // no CTA's shared memory goes before all have read it
        cluster_arrive();
        cluster_wait();
    }
}
// Layers that it takes: up to 2^14 elements a CTA.  Mask phase replayed from a graph, and mask, encoding and decoding called in a row, us, this kernel and
// the others: 256 x 256 (2^13 a CTA) 6.3 and 10.4, 14.3 and 19; 128 x 256 (2^14) 8.0 and 10.4, 15.6 and 19; 25 x 489 (2^14, one CTA) 9.2
// and 13.1, 19.5 and 21; 256 x 512 in four CTAs (2^15) 12.1 and 10.5, 19.9 and 19.  A CTA takes its row tiles one after the other, so of two at most (mask
// phase: two, 435 x 35 9.0 and 13.2, 464 x 218 12.2 and 12.6; four, 1949 x 46 15.3 and 13.2; six, 1497 x 58 19.0 and 12.4).
constexpr int64_t kSmallPerCta = 1 << 14;
int small_ctas(const Geometry &g) {
    const int ctas = g.nrt < kSmallCluster ? g.nrt : kSmallCluster;
    const int row_tiles = (g.nrt + ctas - 1) / ctas;
    return g.nblk <= kSmallMaxBlocks && row_tiles <= 2 && (int64_t)row_tiles * g.bm * g.kp() <= kSmallPerCta ? ctas : 0;
}

// Scores and maxima of a batch, cleared (one CTA per layer; a memset per layer costs a launch each).
template <int CAP>
__global__ void __launch_bounds__(256)
clear_scores_kernel(const __grid_constant__ Batch<ScoreLayer, CAP> batch) {
    chain_kernels();
    const ScoreLayer &L = batch.layer[blockIdx.x];
    if (threadIdx.x == 0) *const_cast<uint32_t *>(L.max_key) = 0u;
    const int64_t n = (int64_t)L.g.nrt * L.g.nblk;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) L.score[i] = 0ull;
}

// Grids of resident CTAs: every CTA is on an SM from the start and takes its share of the items.  What a device holds of a
// kernel does not change, so it is asked for once (the queries take a microsecond or two of every call).
template <typename... Params>
int resident_grid(void (*kern)(Params...), std::atomic<int> *capacity, int64_t items) {
    int dev = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) dev = 0;
    int cap = dev >= 0 && dev < kMaxDevices ? capacity[dev].load(std::memory_order_relaxed) : 0;
    if (cap <= 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kM1Threads, 0) != cudaSuccess || per_sm <= 0) per_sm = 4;
        cap = sm_count_of(dev) * per_sm;
        if (dev >= 0 && dev < kMaxDevices) capacity[dev].store(cap, std::memory_order_relaxed);
    }
    return (int)(items < cap ? items : cap);
}
template <int M>
int group_bits_grid(int64_t items) {
    static std::atomic<int> capacity[kMaxDevices];
    return resident_grid(group_bits_kernel<M>, capacity, items);
}

bool saliency_vec_ok(const float *s, int64_t ld) { return (ld % 4 == 0) && ((reinterpret_cast<uintptr_t>(s) & 15u) == 0); }
int saliency_chunks(const Geometry &g) { return (int)((g.kp() + kM1ChunkK - 1) / kM1ChunkK); }

// Layers [0, n) in launches of up to kBatchLayers; units(layer) = work units of a layer, launch(batch, units of the batch).
template <typename Units, typename Launch>
cudaError_t for_batches(const ScoreLayer *layers, int n, Units units, Launch launch) {
    for (int at = 0; at < n; at += kBatchLayers) {
        Batch<ScoreLayer, kBatchLayers> b;
        b.n = n - at < kBatchLayers ? n - at : kBatchLayers;
        b.first[0] = 0;
        for (int i = 0; i < b.n; ++i) {
            b.layer[i] = layers[at + i];
            b.layer[i].chunks = saliency_chunks(b.layer[i].g);
            b.layer[i].vec_ok = saliency_vec_ok(b.layer[i].s, b.layer[i].ld);
            b.first[i + 1] = b.first[i] + units(b.layer[i].g);
        }
        if (b.first[b.n] > 0x7FFFFFFFll) return cudaErrorInvalidValue;
        cudaError_t e = launch(b);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
Batch<ScoreLayer, 1> batch_of_one(const ScoreLayer &L, int64_t units) {
    Batch<ScoreLayer, 1> b;
    b.n = 1; b.first[0] = 0; b.first[1] = units;
    b.layer[0] = L;
    b.layer[0].chunks = saliency_chunks(L.g);
    b.layer[0].vec_ok = saliency_vec_ok(L.s, L.ld);
    return b;
}

template <int CAP, int M, int TOP>
cudaError_t run_block_scores(const Batch<ScoreLayer, CAP> &b, cudaStream_t st) {
    static std::atomic<int> capacity[kMaxDevices];
    const int grid = resident_grid(block_score_kernel<CAP, M, TOP>, capacity, b.first[b.n]);
    return launch_chained(block_score_kernel<CAP, M, TOP>, (unsigned)grid, kM1Threads, 0, st, b);
}
// The selecting forms where n is 1 or 2 and only survivors count (all layers of a launch share n and m); from n = 3 on the
// selection network is longer than the work it saves.
template <int CAP>
cudaError_t run_block_scores_any(const Batch<ScoreLayer, CAP> &b, cudaStream_t st) {
    const Geometry &g = b.layer[0].g;
    bool survivors = true;
    for (int i = 0; i < b.n; ++i) survivors = survivors && b.layer[i].g.score_mode == 0;
    if (survivors && g.n == 1) return g.m == 4 ? run_block_scores<CAP, 4, 1>(b, st) : run_block_scores<CAP, 8, 1>(b, st);
    if (survivors && g.n == 2) return g.m == 4 ? run_block_scores<CAP, 4, 2>(b, st) : run_block_scores<CAP, 8, 2>(b, st);
    return run_block_scores<CAP, 4, 0>(b, st);
}

size_t select_smem(int nblk) { return (size_t)nblk * (sizeof(unsigned long long) + sizeof(int)); }
int64_t select_ctas(const Geometry &g) { return (int64_t)g.nrt * (g.bm / 32); }

template <int CAP>
cudaError_t run_block_select(const Batch<ScoreLayer, CAP> &b, cudaStream_t st) {
    size_t smem = 0;
    for (int i = 0; i < b.n; ++i) smem = select_smem(b.layer[i].g.nblk) > smem ? select_smem(b.layer[i].g.nblk) : smem;
    if (smem + 64 > 48 * 1024) {     // the longest rows (nblk near 4096) need the opt-in shared-memory size
        // (the same limit at every call: it belongs to the function, which several host threads may be launching)
        cudaError_t e = cudaFuncSetAttribute(block_select_kernel<CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)select_smem(kMaxBlocksPerRowTile));
        if (e != cudaSuccess) return e;
    }
    if (b.first[b.n] == 0) return cudaSuccess;
    return launch_chained(block_select_kernel<CAP>, (unsigned)b.first[b.n], 256, smem, st, b);
}

}  // namespace

// workspace: [0] max key (uint32), padded to 256 B; then score[nrt * nblk] uint64.
size_t mask_workspace_bytes(const Geometry &g) {
    return kAlign + align_up((size_t)g.nrt * g.nblk * sizeof(unsigned long long));
}

cudaError_t launch_clear_scores(const ScoreLayer *layers, int n, cudaStream_t st) {
    return for_batches(layers, n, [](const Geometry &) { return (int64_t)1; }, [&](const Batch<ScoreLayer, kBatchLayers> &b) {
        return launch_chained(clear_scores_kernel<kBatchLayers>, (unsigned)b.n, 256, 0, st, b);
    });
}

cudaError_t launch_block_scores(const ScoreLayer *layers, int n, cudaStream_t st) {
    return for_batches(layers, n, [](const Geometry &g) { return (g.mp() / kM1Rows) * (int64_t)saliency_chunks(g); },
                       [&](const Batch<ScoreLayer, kBatchLayers> &b) { return run_block_scores_any(b, st); });
}

cudaError_t launch_block_selects(const ScoreLayer *layers, int n, cudaStream_t st) {
    return for_batches(layers, n, select_ctas, [&](const Batch<ScoreLayer, kBatchLayers> &b) { return run_block_select(b, st); });
}

cudaError_t launch_block_select(const Geometry &g, const void *d_workspace, int32_t *d_blk_col, uint32_t *d_nm_bits,
                                cudaStream_t st) {
    ScoreLayer L = {};
    L.g = g; L.nm_bits = d_nm_bits; L.blk_col = d_blk_col;
    L.score = reinterpret_cast<unsigned long long *>(const_cast<uint8_t *>(reinterpret_cast<const uint8_t *>(d_workspace)) + kAlign);
    return run_block_select(batch_of_one(L, select_ctas(g)), st);
}

cudaError_t launch_build_mask(const float *d_s, int64_t ld, const Geometry &g, int32_t *d_blk_col,
                              uint32_t *d_nm_bits, void *d_workspace, size_t workspace_bytes, bool max_known,
                              cudaStream_t st) {
    uint32_t *max_key = reinterpret_cast<uint32_t *>(d_workspace);
    unsigned long long *score =
        reinterpret_cast<unsigned long long *>(reinterpret_cast<uint8_t *>(d_workspace) + kAlign);
    if (const int ctas = small_ctas(g)) {
        auto launch = [&](auto kern) {
            return launch_clusters(kern, (unsigned)ctas, kSmallThreads, 0, st, (unsigned)ctas, d_s, ld, g, saliency_vec_ok(d_s, ld), max_known, max_key,
                                   score, d_nm_bits, d_blk_col, ctas);
        };
        return g.m == 4 ? launch(mask_small_kernel<4>) : launch(mask_small_kernel<8>);
    }
    // max_known: the first word already holds the layer's largest canonical |s| (written by the saliency kernel
    // that produced S), so only the scores are cleared and the pass over S that finds the maximum is skipped
    cudaError_t e = max_known ? cudaMemsetAsync(score, 0, workspace_bytes - kAlign, st)
                              : cudaMemsetAsync(d_workspace, 0, workspace_bytes, st);
    if (e != cudaSuccess) return e;
    const bool vec_ok = saliency_vec_ok(d_s, ld);

    // work items of 32 rows x 256 k-elements, dealt out to resident CTAs
    const int chunks = saliency_chunks(g);
    const int64_t items = (g.mp() / kM1Rows) * chunks;
    if (g.m == 4)
        group_bits_kernel<4><<<group_bits_grid<4>(items), kM1Threads, 0, st>>>(
            d_s, ld, g, vec_ok, items, chunks, !max_known, max_key, d_nm_bits);
    else
        group_bits_kernel<8><<<group_bits_grid<8>(items), kM1Threads, 0, st>>>(
            d_s, ld, g, vec_ok, items, chunks, !max_known, max_key, d_nm_bits);
    ScoreLayer L = {};
    L.g = g; L.s = d_s; L.ld = ld; L.max_key = max_key; L.nm_bits = d_nm_bits; L.score = score; L.blk_col = d_blk_col;
    e = cudaGetLastError();
    if (e == cudaSuccess) e = run_block_scores_any(batch_of_one(L, items), st);
    if (e != cudaSuccess) return e;
    return run_block_select(batch_of_one(L, select_ctas(g)), st);
}

}  // namespace crisp
