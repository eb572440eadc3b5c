// The N:M step on eight consecutive saliency values, and how the kernels that stream a weight-shaped tensor cut it
// into work items.  Shared by the mask projection and the fused saliency kernel.
#pragma once

#include "crisp_internal.h"

namespace crisp {

constexpr int kM1Threads = 256;

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

constexpr int kM1Warps = kM1Threads / 32;
constexpr int kM1Rows = 32;              // rows of a patch (divides every block height)
constexpr int kM1LaneRows = 4;           // rows of a lane

// The kernels that stream a weight-shaped tensor give a warp a patch of 32 x 32 elements: one mask word of each row, inside one block
// (block_rows and block_k are multiples of 32), so that everything a warp adds up belongs to one score.  Lane l takes the eight elements at column
// 8 (l mod 4) of the rows l / 4 + 8 i, i = 0..3 (all loads issued first).  Patches are numbered along rows of patches, and the warps of a
// CTA take eight in a row, whatever the width of the layer.
struct Patch { int64_t row0, at; int word; bool any; };      // first row, number, mask word of its rows, and whether there is one
__device__ __forceinline__ Patch patch_of(int64_t cta, int warp, const Geometry &g) {
    Patch p;
    p.at = cta * kM1Warps + warp;
    const uint32_t at = (uint32_t)p.at, rg = at / (uint32_t)g.wpr;              // (2^31 patches would be 2^41 elements)
    p.word = (int)(at - rg * (uint32_t)g.wpr);
    p.row0 = (int64_t)rg * kM1Rows;
    p.any = p.row0 < g.mp();
    return p;
}
inline int64_t patch_ctas(const Geometry &g) { return (g.mp() / kM1Rows * g.wpr + kM1Warps - 1) / kM1Warps; }

// Two fp32 values in one 64-bit register and the packed fp32 instructions of sm_100 on them (one instruction
// per pair; each half is rounded as the scalar instruction would round it).
__device__ __forceinline__ uint64_t f32x2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 f32x2_halves(uint64_t v) {
    float2 h;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(h.x), "=f"(h.y) : "l"(v));
    return h;
}
__device__ __forceinline__ float f32x2_sum(uint64_t v) {       // lo + hi
    const float2 h = f32x2_halves(v);
    return __fadd_rn(h.x, h.y);
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) { uint64_t r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) { uint64_t r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) { uint64_t r; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ uint64_t add2_down(uint64_t a, uint64_t b) { uint64_t r; asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }

// The larger of two values, NaN if one of them is.
__device__ __forceinline__ float max_nan(float a, float b) { float r; asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b)); return r; }

// The two largest of four values that are not negative (equal values count as often as they occur); a is NaN if one of the four is.
struct Two { float a, b; };
__device__ __forceinline__ Two top2_of4(float x0, float x1, float x2, float x3) {
    const float h0 = max_nan(x0, x1), l0 = fminf(x0, x1), h1 = max_nan(x2, x3), l1 = fminf(x2, x3);
    return Two{max_nan(h0, h1), fmaxf(fminf(h0, h1), fmaxf(l0, l1))};
}

// What a warp adds up of its 32 x 32 elements of S before the scale of the layer is known, in 64 bits:
//   bits 63..56  biased exponent e of the largest element (0: all are zero or denormal)
//   bits 55..51  0: the sum does not stand; c > 0: it does if the layer's largest exponent is at most e + c - 1
//   bits 50..0   the sum of the counted elements in units of 2^(e - 127 - 40)
// A score counts floor(s * 2^(40 - e_max)).  An element has 24 bits, so that is exact, nothing is cut off, for every element whose
// exponent is at least e_max - 17; where that holds for all counted elements of the warp, its part of the score is its exact sum, in whichever unit
// it was formed, shifted by the difference of the two exponents.  e + c - 1 is the smallest counted exponent plus 17.  Of normal or of
// product-distributed weights less than one warp in 10^5 fails this for 2:4 (two of four elements count); the score kernel goes through those
// elements again, once e_max is known.
constexpr int kRecordCodeShift = 51, kRecordExpShift = 56;
constexpr unsigned long long kRecordSum = (1ull << kRecordCodeShift) - 1;

// The N:M step on a lane's rows.  `key`: the bits of its elements (signs, infinities and NaN among them).  Returns its mask bits, byte i for row i of R; v: the
// values that count in the scores, top: the bits of the largest.  TOP = 1 or 2: n is TOP and only survivors count, so a group's largest values are selected with
// minima and maxima, which serve both the mask (an element is kept if it reaches the smallest of them) and the sums (whichever of equal values is
// kept; ties, where more than n elements reach the smallest, go by rank).  TOP = 0: any n, and all elements where all_count is set.  reload(i, key) reads the
// canonical bits of the lane's row i again, for infinities and NaN, so that no register holds them until then.
template <int M, int TOP> constexpr int kCounted = TOP ? TOP * (8 / M) : 8;     // values that count, of a row of a lane
template <int M, int TOP, int R, typename Reload>
__device__ __forceinline__ uint32_t select_rows(uint32_t (&key)[R][8], int n, bool all_count, const uint8_t *s_keep, const Reload &reload,
                                                float (&v)[R][kCounted<M, TOP>], uint32_t &top) {
    constexpr int kGroups = 8 / M;
    // Ties of a row, while its elements are in registers, where those are not what there is too little of (4096 x 4096, 2:4, three of four elements zero: 26.3 us
    // for the mask, 31.7 with the rows read again; but 15.6 instead of 13.0 for the saliency of 35 small layers, two rows a lane at 40 registers).
    constexpr bool kTiesByRow = R == kM1LaneRows;
    uint32_t bits = 0u;
    auto ranked = [&](const uint32_t (&raw)[8]) -> uint32_t {
        uint32_t q[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) q[j] = raw[j] & 0x7FFFFFFFu;
        if constexpr (M == 4) return (uint32_t)s_keep[outcomes4(q)] | ((uint32_t)s_keep[outcomes4(q + 4)] << 4);
        else return top_n_bits<M>(q, TOP ? TOP : n);
    };
    top = 0u;
    if constexpr (TOP == 0) {
#pragma unroll
        for (int i = 0; i < R; ++i) {
#pragma unroll
            for (int j = 0; j < 8; ++j) { key[i][j] = canonical_bits(key[i][j]); top = max(top, key[i][j]); }
            const uint32_t b = ranked(key[i]);
            bits |= b << (8 * i);
#pragma unroll
            for (int j = 0; j < 8; ++j) v[i][j] = all_count || ((b >> j) & 1u) ? __uint_as_float(key[i][j]) : 0.f;
        }
    } else {
        float top_f = 0.f;
        auto select = [&](int i, const uint32_t (&q8)[8]) {
            float x[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] = fabsf(__uint_as_float(q8[j]));
            const Two p = top2_of4(x[0], x[1], x[2], x[3]), q = top2_of4(x[4], x[5], x[6], x[7]);
            top_f = max_nan(top_f, max_nan(p.a, q.a));
            if constexpr (M == 4) {
                v[i][0] = p.a; v[i][TOP] = q.a;
                if constexpr (TOP == 2) { v[i][1] = p.b; v[i][3] = q.b; }
            } else {
                v[i][0] = fmaxf(p.a, q.a);
                if constexpr (TOP == 2) v[i][1] = fmaxf(fminf(p.a, q.a), fmaxf(p.b, q.b));
            }
            uint32_t row = 0u;
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (x[j] >= v[i][(M == 4 ? j / 4 : 0) * TOP + TOP - 1]) row |= 1u << j;
            if (kTiesByRow && __popc(row) != kGroups * TOP) row = ranked(q8);
            bits |= row << (8 * i);
        };
#pragma unroll
        for (int i = 0; i < R; ++i) select(i, key[i]);
        if (__float_as_uint(top_f) >= 0x7F800000u) {
            bits = 0u; top_f = 0.f;
#pragma unroll
            for (int i = 0; i < R; ++i) {
                uint32_t q[8];
                reload(i, q);
                select(i, q);
            }
        }
        if (kTiesByRow) {
        } else if (top_f == 0.f) {                           // (zeros: columns beyond the matrix, blocks pruned before)
            bits = (M == 4 ? 0x11111111u : 0x01010101u) * ((1u << TOP) - 1u) >> (32 - 8 * R);
        } else if (__popc(bits) != R * kGroups * TOP) {
            uint32_t q[R][8];
            bits = 0u;
#pragma unroll
            for (int i = 0; i < R; ++i) reload(i, q[i]);
#pragma unroll
            for (int i = 0; i < R; ++i) bits |= ranked(q[i]) << (8 * i);
        }
        top = __float_as_uint(top_f);
    }
    return bits;
}

// A lane's share of a record whose largest element has the biased exponent e: sums in units of 2^(e - 127 - 20) and 2^(e - 127 - 40), the
// smallest counted value that is not zero (all ones: none).  v = r + d with r the nearest multiple of the first unit (adding 1.5 * 2^(e - 127 + 3) makes fp32 step
// by that much) and d exact; r is at most 2^21 and |d| half a unit of r, so that 16 values of each half add up exactly, eight for r.
struct LaneSums { uint32_t r, low; int d; };
__device__ __forceinline__ bool record_in_range(int e) { return e >= 41 && e <= 240; }         // all constants are fp32 numbers
template <int M, int TOP, int R>
__device__ __forceinline__ LaneSums sum_rows(const float (&v)[R][kCounted<M, TOP>], int e) {
    constexpr int kRow = kCounted<M, TOP>, kAll = R * kRow;
    LaneSums out;
    // the last value of each group is its smallest, unless that is zero
    out.low = 0xFFFFFFFFu;
#pragma unroll
    for (int c = TOP ? TOP - 1 : 0; c < kAll; c += TOP ? TOP : 1) out.low = min(out.low, __float_as_uint(v[c / kRow][c % kRow]) - (TOP ? 0u : 1u));
    if (TOP == 0) {
        if (out.low != 0xFFFFFFFFu) ++out.low;
    } else if (out.low == 0u) {
        out.low = 0xFFFFFFFFu;
#pragma unroll
        for (int c = 0; c < kAll; ++c) out.low = min(out.low, __float_as_uint(v[c / kRow][c % kRow]) - 1u);      // (zero: the largest of all)
        if (out.low != 0xFFFFFFFFu) ++out.low;
    }
    const bool in_range = record_in_range(e);
    const float step = __uint_as_float(((uint32_t)(in_range ? e + 3 : 130) << 23) | 0x400000u);
    const uint64_t step2 = f32x2(step, step);
    const float r_unit = __uint_as_float((uint32_t)(in_range ? 274 - e : 127) << 23), d_unit = __uint_as_float((uint32_t)(in_range ? 294 - e : 127) << 23);
    uint64_t r_sum = f32x2(0.f, 0.f), d_sum = r_sum;
    out.r = 0u;
#pragma unroll
    for (int c = 0; c < kAll; c += 2) {
        const uint64_t x = f32x2(v[c / kRow][c % kRow], v[(c + 1) / kRow][(c + 1) % kRow]);
        const uint64_t r = sub2(add2(x, step2), step2);
        r_sum = add2(r_sum, r);
        d_sum = add2(d_sum, sub2(x, r));
        if (c % 16 == 14 || c + 2 == kAll) {
            const float2 h = f32x2_halves(r_sum);
            out.r += __float2uint_rn(h.x * r_unit) + __float2uint_rn(h.y * r_unit);
            r_sum = f32x2(0.f, 0.f);
        }
    }
    const float2 h = f32x2_halves(d_sum);
    out.d = __float2int_rn(h.x * d_unit) + __float2int_rn(h.y * d_unit);
    return out;
}
// The record of 32 x 32 elements: e of the largest, low the smallest counted that is not zero, sums over all lanes (r below 2^32, |d| below 2^30).
__device__ __forceinline__ unsigned long long make_record(int e, uint32_t low, uint32_t r, int d) {
    const int spare = (int)(low >> 23) - e + 17;             // how far above e the layer's exponent may lie
    const bool none = low == 0xFFFFFFFFu;
    const int code = none ? 18 : record_in_range(e) && low >= 0x800000u && spare >= 0 ? spare + 1 : 0;
    const unsigned long long sum = none ? 0ull : ((unsigned long long)r << 20) + (long long)d;
    return ((unsigned long long)e << kRecordExpShift) | ((unsigned long long)code << kRecordCodeShift) | (sum & kRecordSum);
}

// The N:M step and the record of a warp that holds 32 x 32 elements.
template <int M, int TOP, typename Reload>
__device__ __forceinline__ uint32_t bits_and_record(uint32_t (&key)[kM1LaneRows][8], int n, bool all_count, const uint8_t *s_keep,
                                                    const Reload &reload, uint32_t &best, unsigned long long &record) {
    float v[kM1LaneRows][kCounted<M, TOP>];
    uint32_t top;
    const uint32_t bits = select_rows<M, TOP>(key, n, all_count, s_keep, reload, v, top);
    top = __reduce_max_sync(0xFFFFFFFFu, top);
    best = max(best, top);
    const int e = (int)(top >> 23);
    const LaneSums s = sum_rows<M, TOP>(v, e);
    record = make_record(e, __reduce_min_sync(0xFFFFFFFFu, s.low), __reduce_add_sync(0xFFFFFFFFu, s.r), __reduce_add_sync(0xFFFFFFFFu, s.d));
    return bits;
}

// The mask words of a warp's 32 rows (byte i of lane l: columns 8 (l mod 4).. of row l / 4 + 8 i) from four lanes' bytes each: lane l gets the
// word of row l / 4 + 8 (l mod 4).
__device__ __forceinline__ uint32_t mask_words(uint32_t bits, int lane) {
    const uint32_t p = __shfl_xor_sync(0xFFFFFFFFu, bits, 1);
    bits = lane & 1 ? __byte_perm(bits, p, 0x3715) : __byte_perm(bits, p, 0x6240);
    const uint32_t o = __shfl_xor_sync(0xFFFFFFFFu, bits, 2);
    return lane & 2 ? __byte_perm(bits, o, 0x3276) : __byte_perm(bits, o, 0x5410);
}
__device__ __forceinline__ int mask_word_row(int lane) { return (lane >> 2) + 8 * (lane & 3); }

}  // namespace crisp
