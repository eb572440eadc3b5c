// Mask projection kernels: saliency -> hybrid (block + N:M) mask.
//
// Algorithm 1 of the paper, restricted to one layer with the block keep count given:
//   K-M1a per group of M: keep the N largest (fine-grained N:M step), the layer-wide maximum of the canonical saliency (it sets
//         the fixed-point scale of the scores), and sums of 32 x 32 elements in their own scale: the one pass over S
//   K-M1b block scores s_j = sum |T_w| as exact fixed-point integers, from those sums
//   K-M2  per row of the block grid: keep the kkeep highest-scored blocks and clear the
//         bits of the pruned ones (blocks keep their positions)
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

// Eight consecutive fp32 values from a 32-byte boundary, one load.
__device__ __forceinline__ void load8_wide(const float *p, uint32_t key[8]) {
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(key[0]), "=r"(key[1]), "=r"(key[2]), "=r"(key[3]), "=r"(key[4]), "=r"(key[5]), "=r"(key[6]), "=r"(key[7]) : "l"(p) : "memory");
}
// Canonical bits of the lane's elements of a patch, zero beyond the matrix; vec_ok: S and its rows lie on 16-byte boundaries.
__device__ __forceinline__ void load_patch(const float *s, int64_t ld, const Geometry &g, bool vec_ok, int64_t row0, int64_t col0, int lane,
                                           uint32_t (&key)[kM1LaneRows][8]) {
    const int64_t row = row0 + (lane >> 2), k0 = col0 + 8 * (lane & 3);
    if (vec_ok && row0 + kM1Rows <= g.rows && k0 + 8 <= g.k) {
#pragma unroll
        for (int i = 0; i < kM1LaneRows; ++i) load8_raw(s, ld, row + 8 * i, k0, key[i]);
#pragma unroll
        for (int i = 0; i < kM1LaneRows; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) key[i][j] = canonical_bits(key[i][j]);
    } else {
#pragma unroll
        for (int i = 0; i < kM1LaneRows; ++i) load8(s, ld, g.rows, g.k, row + 8 * i, k0, vec_ok, key[i]);
    }
}

// K-M1a: the one pass over S.  The fine-grained N:M step does not depend on the score scale, and the sums of bits_and_record wait for it with a
// shift, so mask bits, layer maximum (one partial maximum a CTA, in `maxima`; nullptr: known) and the records of the scores come from the same load.
// What bounds it is DRAM: S comes in while the results of the calls in front, dirty in L2, leave for it (67 MB read and some 40 written back in 17 us; 13 instructions an
// element fill 45 % of the issue slots).  Copies of the next patch into shared memory while this one is worked on (cp.async, two stages) gained nothing, 18.2 to
// 18.5 us where this took 18.0; nor did 2 or 4 resident CTAs, 20.5 and 18.0.
// align: of S and its rows, 32 bytes (one load for eight elements), 16 or less.
template <int M, int TOP>
__global__ void __launch_bounds__(kM1Threads, 3)
group_bits_kernel(const float *s, int64_t ld, Geometry g, int align, int64_t items, uint32_t *maxima, uint32_t *nm_bits,
                  unsigned long long *records) {
    __shared__ uint8_t s_keep[64];
    __shared__ uint32_t s_best[kM1Warps];
    chain_kernels();
    if (M == 4 && threadIdx.x < 64) s_keep[threadIdx.x] = (uint8_t)keep_mask_of_outcomes(threadIdx.x, g.n);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t best = 0u;
    for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
        const Patch x = patch_of(it, warp, g);
        if (!x.any) continue;
        const int64_t row = x.row0 + (lane >> 2), k0 = (int64_t)x.word * 32 + 8 * (lane & 3);
        auto reload = [&](int i, uint32_t (&q)[8]) { load8(s, ld, g.rows, g.k, row + 8 * i, k0, align >= 16, q); };
        uint32_t key[kM1LaneRows][8];
        if (align >= 16 && x.row0 + kM1Rows <= g.rows && k0 + 8 <= g.k) {
            const float *p = s + row * ld + k0;
            if (align >= 32) {
#pragma unroll
                for (int i = 0; i < kM1LaneRows; ++i) load8_wide(p + 8 * i * ld, key[i]);
            } else {
#pragma unroll
                for (int i = 0; i < kM1LaneRows; ++i) load8_raw(s, ld, row + 8 * i, k0, key[i]);
            }
        } else {
#pragma unroll
            for (int i = 0; i < kM1LaneRows; ++i) reload(i, key[i]);
        }
        unsigned long long record;
        const uint32_t bits = mask_words(bits_and_record<M, TOP>(key, g.n, g.score_mode != 0, s_keep, reload, best, record), lane);
        nm_bits[(x.row0 + mask_word_row(lane)) * g.wpr + x.word] = bits;
        if (lane == 0) records[x.at] = record;
    }
    if (maxima) {
        if (lane == 0) s_best[warp] = best;
        __syncthreads();
        if (threadIdx.x == 0) {
#pragma unroll
            for (int w = 1; w < kM1Warps; ++w) best = max(best, s_best[w]);
            maxima[blockIdx.x] = best;
        }
    }
}

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

// K-M1b: the block scores from the records of K-M1a, once the scale is known: a warp a block, a lane a record.  A record whose sum does
// not stand (see bits_and_record) has its 32 x 32 elements counted again, the mask bits telling which.
// Measured (us, 4096 x 4096, 2:4, S of 64 MiB): the pass over S and this kernel 17.0 + 3.8, where a memset, a pass for bits and maximum and a second one
// for the scores took 1.8 + 16.2 + 11.4; mask, encoding and decoding in a row 59.3 -> 47.2.  The mask phase alone, in a row: 28.8 -> 18.5, 4:8 in blocks of 32 x 32
// 41.1 -> 39.8.  Where no record stands (elements spread over 20 binades evenly) this kernel is a second pass over S: 28.8 -> 31.5 and 41.1 -> 52.6.
// Where all elements count (score mode 1, n = m) the small ones decide: 2 % of the records of normal S do not stand, 36 % of those of products of two normals; calls
// with 64 x 64 blocks in a row, 4:4 35.6 -> 30.7 and 35.2 -> 36.8, 8:8 42.4 -> 39.9 and 42.5 -> 46.2, mode 1 of 2:4 33.9 -> 29.7 and 33.9 -> 35.9; smaller
// layers gain in all of them (256 x 2304, 4:4, 12.5 -> 12.4 for products).
template <int CAP>
__global__ void __launch_bounds__(kM1Threads)
block_score_kernel(const __grid_constant__ Batch<ScoreLayer, CAP> batch) {
    __shared__ uint32_t s_best[kM1Threads / 32];
    chain_kernels();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int l = batch.find(blockIdx.x);
    const ScoreLayer &L = batch.layer[l];
    const Geometry &g = L.g;
    const int64_t cta = blockIdx.x - batch.first[l], block = cta * (kM1Threads / 32) + warp;
    uint32_t mk;
    if (L.maxima) {
        mk = 0u;
        for (int i = threadIdx.x; i < L.n_maxima; i += kM1Threads) mk = max(mk, L.maxima[i]);
        mk = __reduce_max_sync(0xFFFFFFFFu, mk);
        if (lane == 0) s_best[warp] = mk;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kM1Threads / 32; ++w) mk = max(mk, s_best[w]);
        if (cta == 0 && threadIdx.x == 0) *L.max_key = mk;
    } else {
        mk = *L.max_key;
    }
    if (block >= (int64_t)g.nrt * g.nblk) return;
    const int rt = (int)(block / g.nblk), jb = (int)(block - (int64_t)rt * g.nblk);
    const int wpb = g.bk / 32, parts = g.bm / kM1Rows * wpb;                   // at most 16
    const int64_t rec0 = (int64_t)rt * (g.bm / kM1Rows) * g.wpr + jb * wpb;    // (a record a mask word of every 32nd row)
    unsigned long long acc = 0ull;
    bool stands = true;
    if (lane < parts) {
        const unsigned long long rec = L.records[rec0 + lane / wpb * g.wpr + lane % wpb];
        const int d = (int)(mk >> 23) - (int)(rec >> kRecordExpShift), code = (int)(rec >> kRecordCodeShift) & 31;
        const unsigned long long sum = rec & kRecordSum;
        // nothing counted; all elements below one unit; or a sum that stands
        if (code == 18 && sum == 0ull) acc = 0ull;
        else if (d >= kScoreFractionBits + 1) acc = 0ull;
        else if (d >= 0 && d < code) acc = sum >> d;
        else stands = false;
    }
    if (const uint32_t again = __ballot_sync(0xFFFFFFFFu, !stands)) {
        // The elements of these records once more, the next record's on their way while one is counted.  floor(value * 2^(40 - e_max)): when that
        // power of two is an fp32 number, the product is exact (value <= layer maximum, so it stays below 2^41).
        const int e_max = mk ? key_exponent(mk) : 0, scale_exp = kScoreFractionBits - e_max;
        const bool float_scale = scale_exp >= -126 && scale_exp <= 127;
        const float scale = float_scale ? __uint_as_float((uint32_t)(127 + scale_exp) << 23) : 0.f;
        auto load = [&](uint32_t left, uint32_t (&key)[kM1LaneRows][8], uint32_t &counted) {
            const int part = __ffs(left) - 1, word = jb * wpb + part % wpb;
            const int64_t row0 = (int64_t)rt * g.bm + part / wpb * kM1Rows;
            load_patch(L.s, L.ld, g, L.vec_ok != 0, row0, (int64_t)word * 32, lane, key);
            counted = 0xFFFFFFFFu;
            if (g.score_mode == 0) {
                const uint8_t *bits = reinterpret_cast<const uint8_t *>(L.nm_bits + (row0 + (lane >> 2)) * g.wpr + word) + (lane & 3);
                counted = 0u;
#pragma unroll
                for (int i = 0; i < kM1LaneRows; ++i) counted |= (uint32_t)bits[(int64_t)32 * i * g.wpr] << (8 * i);
            }
        };
        auto count = [&](const uint32_t (&key)[kM1LaneRows][8], uint32_t counted) {
#pragma unroll
            for (int i = 0; i < kM1LaneRows; ++i) {
                if (float_scale) {
                    // an element that does not count is multiplied by zero instead of by the scale: its parts are zero
                    uint64_t r_sum = f32x2(0.f, 0.f), d_sum = r_sum;             // exact for eight values: see floor_parts2
#pragma unroll
                    for (int j = 0; j < 8; j += 2) {
                        const uint32_t two = counted >> (8 * i + j);
                        uint64_t r, fd;
                        floor_parts2(mul2(f32x2(__uint_as_float(key[i][j]), __uint_as_float(key[i][j + 1])),
                                          f32x2(two & 1u ? scale : 0.f, two & 2u ? scale : 0.f)), r, fd);
                        r_sum = add2(r_sum, r);
                        d_sum = add2(d_sum, fd);
                    }
                    acc += ((unsigned long long)__float2uint_rn(f32x2_sum(r_sum) * 9.5367431640625e-07f) << 20) +
                           (unsigned long long)__float2uint_rn(f32x2_sum(d_sum));
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if ((counted >> (8 * i + j)) & 1u) acc += fixed_point_score(key[i][j], e_max);
                }
            }
        };
        uint32_t key[2][kM1LaneRows][8], counted[2], left = again;
        load(left, key[0], counted[0]);
        for (;;) {
            left &= left - 1u;
            if (left) load(left, key[1], counted[1]);
            count(key[0], counted[0]);
            if (!left) break;
            left &= left - 1u;
            if (left) load(left, key[0], counted[0]);
            count(key[1], counted[1]);
            if (!left) break;
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
    if (lane == 0) L.score[block] = acc;
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
// one SM (some 250 for eight elements), and for the smallest layers the two passes' round trips.  Three kernels in its place take the device 5.5 to
// 10 us and the host more.
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
// Layers that it takes: up to 2^14 elements a CTA, in two row tiles at most (a CTA takes them one after the other).  The line was drawn when the others were a memset
// and three kernels with two passes over S; since they are three with one, it lies on the high side.  Mask phase replayed from a graph, and mask, encoding and
// decoding called in a row, us, this kernel and the others, 2:4.  One row tile a CTA: 16 x 32 (2^10 elements) 3.7 and 6.8, 12.1 and 15.9; 64 x 64 (2^11)
// 5.1 and 5.5, 12.0 and 15.8; 17 x 140 (2^13.3) 5.5 and 8.2, 12.5 and 15.8; 25 x 489 (2^14) 8.8 and 9.6, 17.0 and 18.3; 128 x 256 (2^14) 8.0 and
// 5.8, 14.7 and 15.7; 374 x 248, 3:4 (2^14) 8.8 and 7.5, 16.3 and 16.1.  Two: 435 x 35 (2^12) 8.7 and 7.8, 16.4 and 16.1; 464 x 218 (2^13.8) 11.6 and
// 9.6, 21.7 and 20.0; 941 x 103, 4:8 (2^14) 12.1 and 8.8, 20.9 and 18.0.  Beyond: 256 x 512 in four CTAs (2^15) 12.4 and 6.6, 19.5 and 15.6; four row
// tiles, 1949 x 46 15.5 and 8.3, 24.0 and 17.1.
constexpr int64_t kSmallPerCta = 1 << 14;
int small_ctas(const Geometry &g) {
    const int ctas = g.nrt < kSmallCluster ? g.nrt : kSmallCluster;
    const int row_tiles = (g.nrt + ctas - 1) / ctas;
    return g.nblk <= kSmallMaxBlocks && row_tiles <= 2 && (int64_t)row_tiles * g.bm * g.kp() <= kSmallPerCta ? ctas : 0;
}

// Maxima of a batch, cleared (a memset per layer costs a launch each).
template <int CAP>
__global__ void __launch_bounds__(kBatchLayers)
clear_scores_kernel(const __grid_constant__ Batch<ScoreLayer, CAP> batch) {
    chain_kernels();
    if ((int)threadIdx.x < batch.n) *batch.layer[threadIdx.x].max_key = 0u;
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
bool saliency_vec_ok(const float *s, int64_t ld) { return (ld % 4 == 0) && ((reinterpret_cast<uintptr_t>(s) & 15u) == 0); }

// Layers [0, n) in launches of up to kBatchLayers; units(layer) = work units of a layer, launch(batch, units of the batch).
template <typename Units, typename Launch>
cudaError_t for_batches(const ScoreLayer *layers, int n, Units units, Launch launch) {
    for (int at = 0; at < n; at += kBatchLayers) {
        Batch<ScoreLayer, kBatchLayers> b;
        b.n = n - at < kBatchLayers ? n - at : kBatchLayers;
        b.first[0] = 0;
        for (int i = 0; i < b.n; ++i) {
            b.layer[i] = layers[at + i];
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
    b.layer[0].vec_ok = saliency_vec_ok(L.s, L.ld);
    return b;
}

template <int M, int TOP>
cudaError_t run_group_bits(const ScoreLayer &L, int *ctas, cudaStream_t st) {
    static std::atomic<int> capacity[kMaxDevices];
    const int64_t items = patch_ctas(L.g);
    if (items > 0x0FFFFFFF) return cudaErrorInvalidValue;    // (patches are numbered in 32 bits: 2^31 of them are 2^41 elements)
    const int align = L.ld % 8 == 0 && reinterpret_cast<uintptr_t>(L.s) % 32 == 0 ? 32 : saliency_vec_ok(L.s, L.ld) ? 16 : 4;
    *ctas = resident_grid(group_bits_kernel<M, TOP>, capacity, items < kMaxMaxima ? items : kMaxMaxima);
    return launch_chained(group_bits_kernel<M, TOP>, (unsigned)*ctas, kM1Threads, 0, st, L.s, L.ld, L.g, align, items,
                          const_cast<uint32_t *>(L.maxima), L.nm_bits, const_cast<unsigned long long *>(L.records));
}

int64_t score_ctas(const Geometry &g) { return ((int64_t)g.nrt * g.nblk + kM1Threads / 32 - 1) / (kM1Threads / 32); }
template <int CAP>
cudaError_t run_block_scores(const Batch<ScoreLayer, CAP> &b, cudaStream_t st) {
    return launch_chained(block_score_kernel<CAP>, (unsigned)b.first[b.n], kM1Threads, 0, st, b);
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

// workspace: [0] max key (uint32), padded to 256 B; then score[nrt * nblk] uint64; the records of the pass over S, a uint64 for 32 x 32
// elements; and that pass's partial maxima.
static size_t score_bytes(const Geometry &g) { return align_up((size_t)g.nrt * g.nblk * sizeof(unsigned long long)); }
static size_t record_bytes(const Geometry &g) { return align_up((size_t)(g.mp() / kM1Rows) * g.wpr * sizeof(unsigned long long)); }
size_t mask_workspace_bytes(const Geometry &g) { return mask_score_bytes(g) + record_bytes(g) + kMaxMaxima * sizeof(uint32_t); }
size_t mask_score_bytes(const Geometry &g) { return kAlign + score_bytes(g); }
void set_workspace(ScoreLayer *L, void *d_workspace) {
    uint8_t *ws = reinterpret_cast<uint8_t *>(d_workspace);
    L->max_key = reinterpret_cast<uint32_t *>(ws);
    L->score = reinterpret_cast<unsigned long long *>(ws + kAlign);
    L->records = reinterpret_cast<unsigned long long *>(ws + mask_score_bytes(L->g));
}

cudaError_t launch_clear_scores(const ScoreLayer *layers, int n, cudaStream_t st) {
    return for_batches(layers, n, [](const Geometry &) { return (int64_t)1; }, [&](const Batch<ScoreLayer, kBatchLayers> &b) {
        return launch_chained(clear_scores_kernel<kBatchLayers>, 1u, kBatchLayers, 0, st, b);
    });
}

cudaError_t launch_block_scores(const ScoreLayer *layers, int n, cudaStream_t st) {
    return for_batches(layers, n, score_ctas, [&](const Batch<ScoreLayer, kBatchLayers> &b) { return run_block_scores(b, st); });
}

cudaError_t launch_block_selects(const ScoreLayer *layers, int n, cudaStream_t st) {
    return for_batches(layers, n, select_ctas, [&](const Batch<ScoreLayer, kBatchLayers> &b) { return run_block_select(b, st); });
}

cudaError_t launch_block_select(const Geometry &g, const void *d_workspace, int32_t *d_blk_col, uint32_t *d_nm_bits,
                                cudaStream_t st) {
    ScoreLayer L = {};
    L.g = g; L.nm_bits = d_nm_bits; L.blk_col = d_blk_col;
    set_workspace(&L, const_cast<void *>(d_workspace));
    return run_block_select(batch_of_one(L, select_ctas(g)), st);
}

cudaError_t launch_build_mask(const float *d_s, int64_t ld, const Geometry &g, int32_t *d_blk_col,
                              uint32_t *d_nm_bits, void *d_workspace, bool max_known, cudaStream_t st) {
    ScoreLayer L = {};
    L.g = g; L.s = d_s; L.ld = ld; L.nm_bits = d_nm_bits; L.blk_col = d_blk_col;
    set_workspace(&L, d_workspace);
    if (const int ctas = small_ctas(g)) {
        auto launch = [&](auto kern) {
            return launch_clusters(kern, (unsigned)ctas, kSmallThreads, 0, st, (unsigned)ctas, d_s, ld, g, saliency_vec_ok(d_s, ld), max_known, L.max_key,
                                   L.score, d_nm_bits, d_blk_col, ctas);
        };
        return g.m == 4 ? launch(mask_small_kernel<4>) : launch(mask_small_kernel<8>);
    }
    // max_known: the first word already holds the layer's largest canonical |s| (written by the saliency kernel that produced S)
    if (!max_known)
        L.maxima = reinterpret_cast<uint32_t *>(reinterpret_cast<uint8_t *>(d_workspace) + mask_score_bytes(g) + record_bytes(g));
    const int top = top_counted(g.n, g.score_mode != 0);
    cudaError_t e = g.m == 4 ? (top == 0 ? run_group_bits<4, 0>(L, &L.n_maxima, st) : top == 1 ? run_group_bits<4, 1>(L, &L.n_maxima, st)
                                                                                              : run_group_bits<4, 2>(L, &L.n_maxima, st))
                             : (top == 0 ? run_group_bits<8, 0>(L, &L.n_maxima, st) : top == 1 ? run_group_bits<8, 1>(L, &L.n_maxima, st)
                                                                                              : run_group_bits<8, 2>(L, &L.n_maxima, st));
    if (e == cudaSuccess) e = run_block_scores(batch_of_one(L, score_ctas(g)), st);
    if (e != cudaSuccess) return e;
    return run_block_select(batch_of_one(L, select_ctas(g)), st);
}

}  // namespace crisp
