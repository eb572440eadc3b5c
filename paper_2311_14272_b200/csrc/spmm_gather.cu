// Tensor-core product on layouts TMA cannot address (row pitches or bases that are not multiples of 16 bytes), bf16 results.
//
// It multiplies the same weight tiles as spmm_tc.cu (they come from the execution image, by TMA); what differs is how X gets
// into the operand tile and how Y leaves.  Rows of X that are eight apart start equally far from a 16-byte boundary, whatever
// the pitch (8 rows of 2-byte elements are a multiple of 16 bytes), so the rows of each residue modulo 8 are a matrix that TMA can
// address from the boundary in front of its first row.  Eight such loads bring a kept block as it lies in memory, 136 columns
// for 128; a warp per residue then moves its rows by the one distance that they share and writes them to the operand tile
// in the 128-byte swizzle that TMA would have used.  Rows and columns beyond the matrix arrive as zeros.  Two groups of eight such warps take
// alternate blocks, so that one group's chain (wait, shared-memory reads, writes, fence) does not set the pace alone.
// (Asynchronous 16-byte copies by the same warps instead of TMA: 0.55 us a block, of which the copies' issue alone took half.)
// Y goes through a staging tile and out in 4-byte stores, row by row.
// What bounds a long walk is the X warps' chain, 0.37 us a block; what a launch costs besides is set-up, the first load and the rows of
// Y, a third each.  Measured: 256 x 2304 x 6076, 1:4, keep 0.25: 51.2 us on the CUDA cores, 13.4 here; 512 x 4608 x 588, 2:4: 103 and 11.6.
//
// Few tiles and long walks leave most SMs without work: the walk of a tile is then split over a cluster of 2, 4 or 8 CTAs,
// each of which owns a slice of the tile's rows in the end.  The partial sums travel through distributed shared memory
// and are added in the order of the ranks, so results do not depend on timing.  (160 x 960 x 49, 28 blocks: 16.4 us on the CUDA
// cores, 8.2 with eight CTAs a tile.)
//
// Zeros in a weight tile (pruned places, row tiles that do not keep the block) multiply activations that the pattern does
// not touch: an infinity or a NaN there must not reach the result.  The warps that shift X notice one on the way (one fused
// multiply-add by zero per two elements), put 1 or -1 in its place and leave a note of the tile, the block and the row.  When a
// CTA has multiplied all its tiles, all its warps go through the noted ones: a result with such a term in the canonical format becomes
// what its terms that are not finite add up to, the others stay.  (us, clean, one infinity a column tile, all NaN, and the CUDA cores: 256 x 2304 x 6076, 1:4
// 13.1, 19.6, 31.3, 49.2; 160 x 960 x 49 8.1, 10.3, 11.8, 14.7; 64 x 64 x 50001, where a tile's work is little, 15.7, 31.3, 34.7, 23.0.)
#include <cuda.h>
#include <cuda_bf16.h>

#include <atomic>
#include <new>

#include "crisp_internal.h"
#include "tc_common.cuh"

namespace crisp {

using namespace tc;

namespace {

constexpr int kCols = 128;                               // columns per CTA tile
constexpr int kEpiWarps = 8, kGroups = 2, kGroupWarps = 8;
constexpr int kFirstX = 2 + kEpiWarps;                   // warp 0 weight tiles, warp 1 MMA issuer, epilogue warps, X warps
constexpr int kThreads = 32 * (kFirstX + kGroups * kGroupWarps);
constexpr int kRawCols = kCols + 8;                     // columns of X that hold 128 from any start, in whole 16-byte words
constexpr uint32_t kRawPitch = kRawCols * 2;
constexpr uint32_t kStagePitch = 144;                    // a row of 64 results in the staging tile (odd number of 16-byte words)
constexpr uint32_t kStageTile = 16 * kStagePitch;
constexpr int kMaxSplit = 8;
constexpr uint32_t kSumPitch = kCols * 4 + 16;           // a row of partial sums of a split tile (odd number of 16-byte words)
constexpr uint32_t kTileBitsAt = 768, kTileBits = 2048;   // (place among the barriers) notes of the tiles of a CTA that had a value that is not finite, by number modulo this

// Blocks as they lie in memory, of all warps: [group][slot][residue][bk / 8 rows], a residue's rows from a 128-byte boundary; `ahead`
// slots a group: 1 block of 128 or 96 rows, 2 of 64 or 4 of 32 (these take the most, 4 rows in 1152 bytes).
constexpr uint32_t kRawBytes = kGroups * 4 * 8 * 1152;
__host__ __device__ constexpr uint32_t raw_slot_bytes(int bk) { return ((uint32_t)bk / 8 * kRawPitch + 127u) & ~127u; }
static_assert(kGroups * 2 * 8 * raw_slot_bytes(64) <= kRawBytes && kGroups * 8 * raw_slot_bytes(96) <= kRawBytes &&
              kGroups * 8 * raw_slot_bytes(128) <= kRawBytes && kGroups * 4 * 8 * raw_slot_bytes(32) <= kRawBytes, "raw blocks");
static_assert(kRawBytes >= kTileM * kSumPitch, "partial sums take the place of the raw blocks");

// Maps of X by residue of the row modulo 8.
struct RowMaps { CUtensorMap m[8]; };

struct GatherParams {
    const int32_t *walk_col, *walk_len;
    // canonical format (tiles with activations that are not finite)
    const int32_t *blk_col;
    const uint16_t *vals;
    const uint32_t *idx;
    const uint16_t *x;
    int64_t ldx, ncols;
    uint16_t *y;
    int64_t ldy;
    const float *bias;
    int32_t *status;
    Geometry g;
    int relu;
    int nst, wcap, num_tiles, ahead;                     // ahead: blocks in flight per group of X warps
    int split, split_log2;                               // CTAs that share a tile's walk: a cluster
    uint32_t a_bytes, entry_bytes, stage_bytes, num_stages;
    unsigned long long wait_limit;
    int skip_fill;                                       // test hook: this fill gets no weight tile (-1 = none)
};

__device__ __forceinline__ uint32_t lds32(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint2 lds64(uint32_t a) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts32(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void sts64(uint32_t a, uint32_t x, uint32_t y) {
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void sts128(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
// acc + 0 * w on two bf16 values: stays a zero until w holds an infinity or a NaN
__device__ __forceinline__ uint32_t finite_probe(uint32_t w, uint32_t acc) {
    uint32_t r;
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(w), "r"(0u), "r"(acc));
    return r;
}
// Entries of a tile's walk that a rank of its cluster takes: rank, rank + split, ... (where they lie does not depend on the
// length of the walk, so a rank can ask for its block columns and for the length at the same time).
__device__ __forceinline__ int walk_share(const GatherParams &p, int st, int rank) {
    return (min(p.walk_len[st], p.wcap) - rank + p.split - 1) >> p.split_log2;
}

struct MmaArgs { uint32_t ring, bar_full, bar_empty, bar_tfull, bar_tempty, tmem_base; volatile int *abort_flag; int rank; };

template <bool kSparse, int NM>
__device__ __forceinline__ void mma_loop(const GatherParams &p, const MmaArgs &a) {
    constexpr uint32_t idesc = make_idesc(kCols, kSparse);
    constexpr uint32_t b_step = kSparse ? 256u : 128u;               // 32 or 16 rows of 128 bytes
    const uint64_t a_desc0 = make_smem_desc(a.ring, 2048, 128, kLayoutNone);
    const uint64_t b_desc0 = make_smem_desc(a.ring + p.entry_bytes, (uint32_t)(kBoxN * p.g.bk * 2), 1024, kLayoutSw128);
    const uint64_t m_desc0 = make_smem_desc(a.ring + p.a_bytes, 128, 128, kLayoutNone);
    const uint32_t stage_step = p.stage_bytes >> 4;
    uint32_t stage = 0, ph = 0, acc = 0, acc_ph = 0, meta_buf = 0;
    for (int t = blockIdx.x >> p.split_log2; t < p.num_tiles && !*a.abort_flag; t += gridDim.x >> p.split_log2) {
        const int count = walk_share(p, t % p.nst, a.rank);
        if (count <= 0) continue;                                    // (only a rank of a split tile: nothing to add)
        if (!mbar_wait(a.bar_tempty + 8 * acc, acc_ph ^ 1u, a.abort_flag, p.wait_limit)) return;
        tc_fence_after();
        const uint32_t d_tmem = a.tmem_base + acc * kCols;
        uint32_t accum = 0;
        for (int e = 0; e < count; ++e) {
            if (!mbar_wait(a.bar_full + 8 * stage, ph, a.abort_flag, p.wait_limit)) return;
            tc_fence_after();
            const uint32_t off = stage * stage_step;
            const uint64_t ad = a_desc0 + off, bd = b_desc0 + off;
            if constexpr (kSparse) {
                const uint32_t meta_tmem = a.tmem_base + 2 * kCols + 4 * meta_buf;
                tmem_copy_128x128b(meta_tmem, m_desc0 + off);
#pragma unroll
                for (int j = 0; j < NM; ++j)
                    mma_sparse(d_tmem, ad + j * 256, bd + j * b_step, idesc | (uint32_t)(j & 1), accum | (uint32_t)j, meta_tmem + (j & ~1));
                meta_buf ^= 1u;
            } else {
#pragma unroll
                for (int j = 0; j < NM; ++j) mma_dense(d_tmem, ad + j * 256, bd + j * b_step, idesc, accum | (uint32_t)j);
            }
            accum = 1u;
            mma_commit(a.bar_empty + 8 * stage);
            if (++stage == p.num_stages) { stage = 0; ph ^= 1u; }
        }
        mma_commit(a.bar_tfull + 8 * acc);
        if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
    }
}

// Blocks and rows of X that had a value that is not finite: block columns modulo 32, rows of a block modulo 32.
struct Notes { uint32_t blocks, rows; };

// One row of a tile with values that are not finite, 128 columns from col0, four a lane, one warp: what such terms of the row add up to takes
// the place of the result, which was made with 1 or -1 in their place.  A result that is not finite by itself (from a weight or the bias) is
// one more term.  ReLU comes last, and for all results of such a tile here (after the rounding to bf16, which changes no sign).
// The lanes look through 32 kept blocks, then decode 32 weights at a time, and then all take the noted ones among them, two by two, until every
// sum is a NaN, which nothing changes.  What it costs are a few round trips to L2.
// (Part of the kernel and at one place of it: as a function that is called it reads the launch's parameters through memory, three times the
// repair's time, and the calls cost products without such values 0.4 us.)
__device__ __forceinline__ void repair_row(const GatherParams &p, Notes notes, int row, int64_t col0) {
    const Geometry &g = p.g;
    const int lane = threadIdx.x & 31, vpr = g.bk / g.m * g.n, vpb = (int)g.vals_per_block();
    const int rt = row / g.bm, local = row - rt * g.bm, valid = (int)min((int64_t)kCols, p.ncols - col0) - lane;      // this lane's columns: 0, 32, 64, 96 below it
    const uint16_t *x0 = p.x + col0 + lane;
    auto value = [](const uint16_t *at) { return __uint_as_float((uint32_t)*at << 16); };
    auto odd = [](float v) { return !(fabsf(v) < __int_as_float(0x7f800000)); };
    float extra[4] = {0.f, 0.f, 0.f, 0.f};
    bool settled = false;
    for (int s0 = 0; s0 < g.kkeep && !settled; s0 += 32) {
        const int col_of_lane = s0 + lane < g.kkeep ? p.blk_col[(int64_t)rt * g.kkeep + s0 + lane] : 0;
        uint32_t slots = __ballot_sync(0xFFFFFFFFu, s0 + lane < g.kkeep && (notes.blocks >> (col_of_lane & 31) & 1u));
        for (; slots && !settled; slots &= slots - 1) {
            const int in32 = __ffs(slots) - 1;
            const int64_t blk = (int64_t)rt * g.kkeep + s0 + in32;
            const int krow0 = __shfl_sync(0xFFFFFFFFu, col_of_lane, in32) * g.bk;
            const uint32_t *iw = p.idx + blk * (vpb * g.idx_bits / 32);
            for (int v0 = 0; v0 < vpr && !settled; v0 += 32) {
                const int v = v0 + lane;
                bool hit = v < vpr;
                uint32_t entry = 0;                          // weight and row of the block
                if (hit) {
                    const int at = local * vpr + v, bit = at * g.idx_bits;
                    uint32_t f = iw[bit >> 5] >> (bit & 31);
                    if ((bit & 31) + g.idx_bits > 32) f |= iw[(bit >> 5) + 1] << (32 - (bit & 31));
                    const int kin = v / g.n * g.m + (int)(f & ((1u << g.idx_bits) - 1u));
                    entry = (uint32_t)p.vals[blk * vpb + at] << 16 | (uint32_t)kin;
                    hit = (notes.rows >> (kin & 31) & 1u) && krow0 + kin < g.k;
                }
                uint32_t hits = __ballot_sync(0xFFFFFFFFu, hit);
                while (hits && !settled) {
                    float w[2], xv[2][4];
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const uint32_t e = __shfl_sync(0xFFFFFFFFu, entry, hits ? __ffs(hits) - 1 : 0);
                        const uint16_t *xr = x0 + (int64_t)(krow0 + (int)(e & 0xFFFFu)) * p.ldx;
                        w[u] = __uint_as_float(e & 0xFFFF0000u);
#pragma unroll
                        for (int c = 0; c < 4; ++c) xv[u][c] = hits && 32 * c < valid ? value(xr + 32 * c) : 0.f;
                        hits &= hits - 1;
                    }
                    bool nan = true;
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
#pragma unroll
                        for (int u = 0; u < 2; ++u)
                            if (odd(xv[u][c])) extra[c] = fmaf(w[u], xv[u][c], extra[c]);
                        nan = nan && (32 * c >= valid || extra[c] != extra[c]);
                    }
                    settled = __all_sync(0xFFFFFFFFu, nan);
                }
            }
        }
    }
    uint16_t *y = p.y + (int64_t)row * p.ldy + col0 + lane;
    float was[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) was[c] = 32 * c < valid && (odd(extra[c]) || p.relu) ? value(y + 32 * c) : 0.f;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float v = !odd(extra[c]) ? was[c] : odd(was[c]) ? was[c] + extra[c] : extra[c];
        if (p.relu) v = fmaxf(v, 0.f);
        if (32 * c < valid && (odd(extra[c]) || p.relu)) y[32 * c] = __bfloat16_as_ushort(__float2bfloat16_rn(v));
    }
}

// Y = act(sum + bias) as the kernel on the CUDA cores rounds it: without a bias nothing is added, and a NaN becomes 0 only under ReLU.
// (`noted`: the tile goes through repair_row, which applies ReLU)
template <int N>
__device__ __forceinline__ void finish(const GatherParams &p, float (&v)[N], float bias, bool noted) {
    if (p.bias) {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] += bias;
    }
    if (p.relu && !noted) {
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = fmaxf(v[i], 0.f);
    }
}

// 1 or -1 in the place of a bf16 value that is not finite, two at a time; whether there was one
__device__ __forceinline__ bool finite_only(uint32_t &w) {
    const bool lo = (w & 0x7F80u) == 0x7F80u, hi = (w & 0x7F800000u) == 0x7F800000u;
    if (lo) w = (w & 0xFFFF8000u) | 0x3F80u;
    if (hi) w = (w & 0x8000FFFFu) | 0x3F800000u;
    return lo | hi;
}

// An X warp's rows of a block, from where they arrived to the operand tile.  The result is not 0 if there was a value that is not finite in
// the lane's columns.  kClean: with such values replaced, and the result says in which of the rows 0, 1, 2 and so on they were (modulo 4).
template <bool kWide, bool kClean>
__device__ __forceinline__ uint32_t move_rows(uint32_t src, uint32_t dst, int rows, uint32_t at, uint32_t box_bytes) {
    uint32_t probe = 0, which = 0;
#pragma unroll 1
    for (int r = 0; r < rows; r += 4) {
        const uint32_t s4 = src + (uint32_t)r * kRawPitch, d4 = dst + (uint32_t)r * 1024u;
        if constexpr (kWide) {
            uint2 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = lds64(s4 + u * kRawPitch);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if constexpr (kClean) which |= (uint32_t)(finite_only(v[u].x) | finite_only(v[u].y)) << u;
                else probe = finite_probe(v[u].y, finite_probe(v[u].x, probe));
                sts64(d4 + 1024u * u, v[u].x, v[u].y);
            }
        } else {
            uint32_t v[4][2];
#pragma unroll
            for (int u = 0; u < 4; ++u) { v[u][0] = lds32(s4 + u * kRawPitch); v[u][1] = lds32(s4 + u * kRawPitch + 128u); }
            if (at & 2u) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    v[u][0] = __funnelshift_r(v[u][0], lds32(s4 + u * kRawPitch + 4u), 16);
                    v[u][1] = __funnelshift_r(v[u][1], lds32(s4 + u * kRawPitch + 132u), 16);
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if constexpr (kClean) which |= (uint32_t)(finite_only(v[u][0]) | finite_only(v[u][1])) << u;
                else probe = finite_probe(v[u][1], finite_probe(v[u][0], probe));
                sts32(d4 + 1024u * u, v[u][0]);
                sts32(d4 + 1024u * u + box_bytes, v[u][1]);
            }
        }
    }
    return kClean ? which : probe & 0x7FFF7FFFu;
}
template <bool kWide>
__device__ __noinline__ uint32_t clean_rows(uint32_t src, uint32_t dst, int rows, uint32_t at, uint32_t box_bytes) {
    return move_rows<kWide, true>(src, dst, rows, at, box_bytes);
}

// A row of results, packed two columns a word: word u of the row in `v`, the one after it in `next`; `valid` columns of it
// exist.  4-byte stores: in a row that starts between two words a lane takes the pair one column further on, and the first
// and the last column go alone.  (Whole rows of whole words, the common case, are one predicated store: the branches of the
// other cases cost more than the store.)
__device__ __forceinline__ void store_words(uint16_t *dst, int u, int valid, uint32_t v, uint32_t next) {
    const int odd = (int)(reinterpret_cast<uintptr_t>(dst) >> 1) & 1, c = 2 * u + odd;
    const uint32_t pair = __funnelshift_r(v, next, 16 * odd);
    if (c + 1 < valid) *reinterpret_cast<uint32_t *>(dst + c) = pair;
    if (odd | (valid & 1)) {                                 // (the same for the whole warp)
        if (c + 1 == valid) dst[c] = (uint16_t)pair;
        if (odd && u == 0 && valid > 0) dst[0] = (uint16_t)v;
    }
}

// 16 rows x 64 columns of results from the warp's staging tile, eight rows read before the first is stored.
__device__ __forceinline__ void store_rows(const GatherParams &p, uint32_t stg, int lane, int y0, int64_t x0) {
    const int rows = min(16, p.g.rows - y0), valid = (int)min((int64_t)64, p.ncols - x0);
    uint16_t *dst = p.y + (int64_t)y0 * p.ldy + x0;
#pragma unroll 1
    for (int r0 = 0; r0 < rows; r0 += 8) {
        uint32_t v[8], next[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const uint32_t src = stg + (uint32_t)(r0 + r) * kStagePitch + 4u * lane;
            v[r] = lds32(src);
            next[r] = lds32(src + 4);                        // (the row's padding behind column 63)
        }
#pragma unroll
        for (int r = 0; r < 8; ++r, dst += p.ldy) store_words(dst, lane, r0 + r < rows ? valid : 0, v[r], next[r]);
    }
}

// ----------------------------------------------------------------------------------- kernel
//
// kWide: every row of X starts at a multiple of 8 bytes, so its 256 bytes are 32 8-byte reads; else 4-byte reads, shifted by half
// a word where the row starts between two words.
// Shared memory: num_stages x [weight tile | metadata | two boxes of X] | raw blocks | 8 staging tiles | barriers
template <bool kSparse, bool kWide>
__global__ void __launch_bounds__(kThreads, 1)
spmm_gather_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ RowMaps map_x, const __grid_constant__ GatherParams p) {
    constexpr int kTmemCols = 512;                           // two accumulators and the metadata buffers
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t ring = smem_u32(smem_raw);
    if (ring & 1023u) {                                      // swizzled operand tiles need it
        wait_for_prerequisites();
        if (threadIdx.x == 0) atomicCAS(p.status, 0, (int)CRISP_CUDA_ERROR);
        return;
    }
    const uint32_t raw = ring + p.num_stages * p.stage_bytes, staging = raw + kRawBytes;
    const uint32_t ctrl = staging + kEpiWarps * kStageTile;
    uint8_t *ctrl_gen = smem_raw + (ctrl - ring);
    const uint32_t bar_full = ctrl, bar_empty = ctrl + 64, bar_tfull = ctrl + 128, bar_tempty = ctrl + 144;
    volatile uint32_t *tmem_base_slot = reinterpret_cast<volatile uint32_t *>(ctrl_gen + 160);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(ctrl_gen + 164);
    volatile Notes *notes = reinterpret_cast<volatile Notes *>(ctrl_gen + 192);
    volatile uint32_t *tile_bits = reinterpret_cast<volatile uint32_t *>(ctrl_gen + kTileBitsAt);          // [kTileBits / 32]
    const uint32_t bar_raw = ctrl + 256;                     // [X warp][4]: its rows of a block have arrived

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 1) {
        tmem_alloc(smem_u32(const_cast<uint32_t *>(tmem_base_slot)), kTmemCols);
        tmem_relinquish();
    }
    if (threadIdx.x == 0) {
        prefetch_tensormap(&map_a);
        for (uint32_t s = 0; s < p.num_stages; ++s) { mbar_init(bar_full + 8 * s, 1 + kGroupWarps); mbar_init(bar_empty + 8 * s, 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(bar_tfull + 8 * a, 1); mbar_init(bar_tempty + 8 * a, kEpiWarps); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2) {
        notes->blocks = notes->rows = 0;
        tile_bits[lane] = tile_bits[32 + lane] = 0;
    }
    if (warp >= kFirstX && lane == 0) {
        for (int i = 0; i < 4; ++i) mbar_init(bar_raw + 32u * (uint32_t)(warp - kFirstX) + 8u * i, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        prefetch_tensormap(&map_x.m[(warp - kFirstX) % kGroupWarps]);
    }
    wait_for_prerequisites();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_base_slot;
    const int rank = p.split > 1 ? (int)cluster_rank() : 0;
    const int first_tile = blockIdx.x >> p.split_log2, tile_step = gridDim.x >> p.split_log2;

    if (warp == 0) {
        // ------------------------------------------------ weight tiles
        if (lane == 0) {
            const int entry_rows = (int)(p.entry_bytes >> 8);
            uint32_t stage = 0, ph = 0;
            int fill = 0;
            bool ok = true;
            for (int t = first_tile; t < p.num_tiles && ok && !*abort_flag; t += tile_step) {
                const int st = t % p.nst;
                const int count = walk_share(p, st, rank);
                int arow = (st * p.wcap + rank) * entry_rows;
                for (int e = 0; e < count; ++e, arow += p.split * entry_rows) {
                    if (!mbar_wait(bar_empty + 8 * stage, ph ^ 1u, abort_flag, p.wait_limit)) { ok = false; break; }
                    mbar_expect_tx(bar_full + 8 * stage, p.entry_bytes);
                    if (fill++ != p.skip_fill) tma_load_2d(ring + stage * p.stage_bytes, &map_a, 0, arow, bar_full + 8 * stage);
                    if (++stage == p.num_stages) { stage = 0; ph ^= 1u; }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (lane == 0) {
            const MmaArgs a{ring, bar_full, bar_empty, bar_tfull, bar_tempty, tmem_base, abort_flag, rank};
            switch (kSparse ? p.g.bk / 32 : p.g.bk / 16) {
                case 1: mma_loop<kSparse, 1>(p, a); break;
                case 2: mma_loop<kSparse, 2>(p, a); break;
                case 3: mma_loop<kSparse, 3>(p, a); break;
                case 4: mma_loop<kSparse, 4>(p, a); break;
                case 6: mma_loop<kSparse, 6>(p, a); break;
                default: mma_loop<kSparse, 8>(p, a); break;
            }
        }
    } else if (warp >= kFirstX) {
        // ------------------------------------------------ X: rows res, res + 8, ... of every other block
        // Every other one of all the blocks this CTA multiplies, whatever tile they belong to: a group that skipped more than num_stages
        // blocks between two of its own would find the parity of an older release of its stage.
        const int gi = (warp - kFirstX) / kGroupWarps, res = (warp - kFirstX) % kGroupWarps;
        const CUtensorMap *map = &map_x.m[res];
        const int rows = p.g.bk / 8;                         // of a block, for this warp
        const uint32_t slot_bytes = raw_slot_bytes(p.g.bk), slot_step = 8 * slot_bytes;
        const uint32_t my_raw = raw + (uint32_t)(gi * p.ahead * 8 + res) * slot_bytes;
        const uint32_t my_bar = bar_raw + 32u * (uint32_t)(warp - kFirstX);
        const uint32_t at = ((uint32_t)(reinterpret_cast<uintptr_t>(p.x) + (uintptr_t)((int64_t)res * p.ldx * 2))) & 15u;     // where the rows start
        const uint32_t box_bytes = (uint32_t)(kBoxN * p.g.bk * 2);
        // operand tile: [box][row][128 bytes], 16-byte chunk c of row r at c ^ (r & 7), and r & 7 = res
        const uint32_t lane_src = kWide ? at + 8u * lane : (at & 12u) + 4u * lane;
        const uint32_t lane_dst = (uint32_t)res * 128u + p.entry_bytes +
                                  (kWide ? (uint32_t)(lane >> 4) * box_bytes + ((((uint32_t)lane >> 1 & 7u) ^ (uint32_t)res) << 4) + ((uint32_t)lane & 1u) * 8u
                                         : ((((uint32_t)lane >> 2) ^ (uint32_t)res) << 4) + ((uint32_t)lane & 3u) * 4u);
        uint32_t stage = (uint32_t)gi, ph = 0, slot = 0, slot_ph = 0;
        int tile_no = 0, first = gi;                         // the group's first block of the tile
        bool ok = true;
#pragma unroll 1
        for (int t = first_tile; t < p.num_tiles && ok; t += tile_step, ++tile_no) {
            const int ct = t / p.nst, st = t - ct * p.nst;
            const int32_t *cols = p.walk_col + (int64_t)st * p.wcap + rank;
            int window = 0, col_of_lane = 0;                 // block columns of entries window .. window + 31 of this rank
            auto load_window = [&](int from) {
                window = from;
                const int e = (from + lane) << p.split_log2;
                col_of_lane = rank + e < p.wcap ? cols[e] : 0;
            };
            load_window(0);
            const int count = walk_share(p, st, rank), mine = (count - first + 1) >> 1;   // blocks first, first + 2, ...
            uint32_t to = slot;                              // slot to ask for next; one block is moved, the one `ahead` on asked for
#pragma unroll 1
            for (int i = 0; i < mine + p.ahead; ++i) {
                if (i >= p.ahead) {
                    // (the lanes wait on their own and give up together: those that went on alone would wait in a warp operation
                    // without a bound for lanes that are in the teardown)
                    const bool have = mbar_wait(my_bar + 8 * slot, slot_ph, abort_flag, p.wait_limit) &&
                                      mbar_wait(bar_empty + 8 * stage, ph ^ 1u, abort_flag, p.wait_limit);
                    if (!__all_sync(0xFFFFFFFFu, have)) { ok = false; break; }
                    const uint32_t src = my_raw + slot * slot_step + lane_src, dst = ring + stage * p.stage_bytes + lane_dst;
                    if (__builtin_expect(move_rows<kWide, false>(src, dst, rows, at, box_bytes) != 0u, 0)) {
                        // (said before the stage is handed over: the epilogue reads it behind the accumulator.  The warp's rows are res,
                        // res + 8 and so on: bit 8 u + res for the u-th of four)
                        const uint32_t which = clean_rows<kWide>(src, dst, rows, at, box_bytes);
                        const int col = cols[(first + 2 * (i - p.ahead)) << p.split_log2];
                        atomicOr(const_cast<uint32_t *>(&notes->blocks), 1u << (col & 31));
                        atomicOr(const_cast<uint32_t *>(&notes->rows), ((which & 1u) | (which & 2u) << 7 | (which & 4u) << 14 | (which & 8u) << 21) << res);
                        atomicOr(const_cast<uint32_t *>(tile_bits) + (tile_no % kTileBits >> 5), 1u << (tile_no & 31));
                    }
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_full + 8 * stage);
                    stage += 2;                              // (past the other group's block)
                    if (stage >= p.num_stages) { stage -= p.num_stages; ph ^= 1u; }
                    if (++slot == (uint32_t)p.ahead) { slot = 0; slot_ph ^= 1u; }
                }
                if (i < mine) {
                    const int e = first + 2 * i;
                    if (e >= window + 32) load_window(e);
                    const int col = __shfl_sync(0xFFFFFFFFu, col_of_lane, e - window);
                    if (lane == 0) {
                        // (row res of the block is row col * bk / 8 of the residue's matrix; a residue that X has no row of is all beyond it)
                        mbar_expect_tx(my_bar + 8 * to, (uint32_t)rows * kRawPitch);
                        tma_load_2d(my_raw + to * slot_step, map, ct * kCols, res < p.g.k ? col * rows : 1, my_bar + 8 * to);
                    }
                    if (++to == (uint32_t)p.ahead) to = 0;
                }
            }
            first ^= count & 1;
        }
        if (warp == kFirstX) launch_dependents();            // (this CTA has asked for its last tile)
    } else if (p.split == 1) {
        // ------------------------------------------------ epilogue of whole tiles: 32 rows x 64 columns a warp
        const int q = warp & 3, half = (warp - 2) >> 2;
        const uint32_t stg = staging + (uint32_t)(warp - 2) * kStageTile;
        uint32_t acc = 0, acc_ph = 0;
        int tile_no = 0;
        for (int t = first_tile; t < p.num_tiles; t += tile_step, ++tile_no) {
            const int st = t % p.nst, ct = t / p.nst;
            int go = 0;
            if (lane == 0) go = !*abort_flag && mbar_wait(bar_tfull + 8 * acc, acc_ph, abort_flag, p.wait_limit);
            go = __shfl_sync(0xFFFFFFFFu, go, 0);
            if (!go) break;
            tc_fence_after();
            const int y0 = st * kTileM + 32 * q;
            const int64_t x0 = (int64_t)ct * kCols + 64 * half;
            const bool noted = tile_bits[tile_no % kTileBits >> 5] >> (tile_no & 31) & 1u;
            uint32_t out[32];                                // 64 columns of the lane's row, packed
            const float bias = p.bias && y0 + lane < p.g.rows ? p.bias[y0 + lane] : 0.f;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                uint32_t bits[32];
                float v[32];
                tmem_ld32(tmem_base + acc * kCols + ((uint32_t)(32 * q) << 16) + 64 * half + 32 * c, bits);
                tmem_ld_wait();
#pragma unroll
                for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(bits[i]);
                finish(p, v, bias, noted);
#pragma unroll
                for (int i = 0; i < 16; ++i) out[16 * c + i] = pack_bf16(v[2 * i], v[2 * i + 1]);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_tempty + 8 * acc);
            if (y0 < p.g.rows && x0 < p.ncols) {
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {                // lanes 0..15, then 16..31
                    if (y0 + 16 * h >= p.g.rows) break;
                    __syncwarp();
                    if ((lane >> 4) == h) {
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            sts128(stg + (uint32_t)(lane & 15) * kStagePitch + 16u * i, out[4 * i], out[4 * i + 1], out[4 * i + 2], out[4 * i + 3]);
                    }
                    __syncwarp();
                    store_rows(p, stg, lane, y0 + 16 * h, x0);
                }
            }
            if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
        }
    }
    Notes all = {0u, 0u};                                    // of a cluster
    if (p.split > 1) {
        // ------------------------------------------------ a split tile: one tile a cluster
        // A rank leaves its sums in its own shared memory ([row][128 columns], where the X warps' rings were: they are done when
        // the accumulator is), and then adds up 128 / split rows of all ranks.
        const int ct = first_tile / p.nst, st = first_tile - ct * p.nst;
        const int64_t x0 = (int64_t)ct * kCols;
        const int valid = (int)min((int64_t)kCols, p.ncols - x0);
        if (warp >= 2 && warp < kFirstX) {
            const int q = warp & 3, half = (warp - 2) >> 2;
            const bool any = walk_share(p, st, rank) > 0;    // (a walk may be shorter than the cluster)
            int go = 0;
            if (lane == 0) go = !*abort_flag && (!any || mbar_wait(bar_tfull, 0, abort_flag, p.wait_limit));
            go = __shfl_sync(0xFFFFFFFFu, go, 0);
            tc_fence_after();
            const uint32_t mine = raw + (uint32_t)(32 * q + lane) * kSumPitch;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const int col = 64 * half + 32 * c;
                if (col >= valid || st * kTileM + 32 * q >= p.g.rows) continue;
                uint32_t v[32];
                if (go && any) {
                    tmem_ld32(tmem_base + ((uint32_t)(32 * q) << 16) + col, v);
                    tmem_ld_wait();
                } else {
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] = 0;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) sts128(mine + 4u * (uint32_t)col + 16u * i, v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            }
            tc_fence_before();
        }
        __syncwarp();
        cluster_arrive();
        cluster_wait();
        const int per_rank = kTileM >> p.split_log2;
        const uint32_t note = peer_address(smem_u32(const_cast<Notes *>(notes)), (uint32_t)(lane < p.split ? lane : rank));
        const uint32_t noted_blocks = lds32_peer(note), noted_rows = lds32_peer(note + 4);
        all = {__reduce_or_sync(0xFFFFFFFFu, noted_blocks), __reduce_or_sync(0xFFFFFFFFu, noted_rows)};
        const int row0 = st * kTileM + rank * per_rank;
        constexpr int kWarps = kThreads / 32;
        for (int r = warp; r < per_rank && row0 + r < p.g.rows; r += kWarps) {
            const int row = row0 + r;
            const uint32_t at = raw + (uint32_t)(rank * per_rank + r) * kSumPitch + 16u * lane;
            float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
            for (int s0 = 0; s0 < p.split; s0 += 4) {    // four loads from the others at a time
                float4 part[4];
#pragma unroll
                for (int s = 0; s < 4; ++s)
                    part[s] = s0 + s < p.split && 4 * lane < valid ? lds128_peer(peer_address(at, (uint32_t)(s0 + s))) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int s = 0; s < 4; ++s) { sum.x += part[s].x; sum.y += part[s].y; sum.z += part[s].z; sum.w += part[s].w; }
            }
            const float bias = p.bias ? p.bias[row] : 0.f;
            float v[4] = {sum.x, sum.y, sum.z, sum.w};
            finish(p, v, bias, all.blocks != 0u);
            const uint32_t lo = pack_bf16(v[0], v[1]), hi = pack_bf16(v[2], v[3]);
            const uint32_t next = __shfl_down_sync(0xFFFFFFFFu, lo, 1);
            uint16_t *dst = p.y + (int64_t)row * p.ldy + x0;
            store_words(dst, 2 * lane, valid, lo, hi);
            store_words(dst, 2 * lane + 1, valid, hi, next);
        }
        __syncwarp();
        cluster_arrive();                                    // no rank's shared memory goes before all have read it
        cluster_wait();
    }
    // ------------------------------------------------ teardown (every wait above is bounded)
    tc_fence_before();
    __syncthreads();
    // (The unlikely branches here and in the X warps are marked as such, and what the repair starts from is worked out anew: left in line, or with
    // its values kept in registers from the start of the kernel, it costs every product 0.3 us.)
    if (p.split == 1) { all.blocks = notes->blocks; all.rows = notes->rows; }
    if (__builtin_expect(all.blocks != 0u && !*abort_flag, 0)) {         // (the same for the whole CTA; a cluster's CTAs have one tile, and their share of its rows)
        constexpr int kWarps = kThreads / 32;
        uint32_t cta, tid, stages = p.num_stages;
        asm volatile("mov.u32 %0, %%ctaid.x;\n\tmov.u32 %1, %%tid.x;" : "=r"(cta), "=r"(tid));
        asm volatile("" : "+r"(stages));
        const uint32_t *bits = reinterpret_cast<const uint32_t *>(smem_raw + stages * p.stage_bytes + kRawBytes + kEpiWarps * kStageTile + kTileBitsAt);
        const int nrows = kTileM >> p.split_log2, my_warp = (int)tid >> 5, row_in_tile = p.split > 1 ? (int)cluster_rank() * nrows : 0;
        int no = 0, turn = 0;                                // the warps take turns over the rows of all such tiles; the next one's
        for (int t = (int)cta >> p.split_log2; t < p.num_tiles; t += (int)gridDim.x >> p.split_log2, ++no) {
            if (p.split == 1 && !(bits[no % kTileBits >> 5] >> (no & 31) & 1u)) continue;
            const int row0 = t % p.nst * kTileM + row_in_tile, count = max(0, min(nrows, p.g.rows - row0));
            for (int r = my_warp >= turn ? my_warp - turn : my_warp - turn + kWarps; r < count; r += kWarps)
                repair_row(p, all, row0 + r, (int64_t)(t / p.nst) * kCols);
            turn = (turn + count) % kWarps;
        }
    }
    if (__builtin_expect(*abort_flag != 0, 0)) {
        if (threadIdx.x == 0) atomicCAS(p.status, 0, (int)CRISP_TIMEOUT);
        const unsigned long long t0 = clock64();             // let copies that may still be in flight land
        while ((unsigned long long)(clock64() - t0) < 2000000ull) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(*tmem_base_slot, kTmemCols);
    }
}

typedef void (*GatherKernel)(const CUtensorMap, const RowMaps, const GatherParams);

GatherKernel pick(bool sparse, bool wide) {
    if (sparse) return wide ? spmm_gather_kernel<true, true> : spmm_gather_kernel<true, false>;
    return wide ? spmm_gather_kernel<false, true> : spmm_gather_kernel<false, false>;
}

}  // namespace

// What products through this kernel keep in the handle: the tensor map of the execution image, which is the handle's own, and the
// maps of the X that the last one read (encoding them takes a few microseconds).
struct GatherPlan {
    CUtensorMap image;
    const void *x;
    int64_t ldx, ncols;
    RowMaps rows;
};
void gather_plan_destroy(GatherPlan *plan) { delete plan; }

// Which products come here.  A CTA of the kernel in spmm_direct.cu takes some 3 us for every 128 kept activation rows or 64 weights of a row, and
// again for every wave of its CTAs; a launch of this one 7 to 8 us and little for each further block.  Measured on both sides of the
// lines (us, that kernel and this one).  Kept rows: 256 7.8 and 8.8 (33 x 1114 x 980), 480 14.8 and 8.0 (160 x 960 x 49), 704 32.3 and 9.1.
// Weights of a row: 96 6.2 and 7.4 (128 x 256 x 98), 7.0 and 7.8 (600 x 128 x 147); 128 9.6 and 8.2 (300 x 200 x 245), 18.1 and 8.3
// (423 x 281 x 539).  Results, and multiply-adds: 6.9 and 7.9 (200 x 588, 64 weights a row), 7.0 and 7.9 (39 x 6076, 32); 12.6 and 7.7
// (400 x 490, 96), 11.6 and 9.1 (810 x 343, 32), 19.5 and 7.3 (93 x 12348); many results of fewer than eight weights are stores alone, 4.3 and 6.9 (49 x 7644, 4),
// 10.4 and 7.4 (191 x 2891, 8).
constexpr int64_t kMinKept = 320, kMinWeights = 128, kMinResults = 1 << 18, kMinTerms = 8, kMinMacs = 10000000;
bool gather_supported(const crisp_handle_s *h, int64_t ncols, int y_dtype) {
    if (y_dtype != 0 || (h->exec_kind != CRISP_PATH_DENSE && h->exec_kind != CRISP_PATH_SPARSE) || h->g.kkeep == 0) return false;
    if (!tensor_maps_available() || ncols >= (1ll << 31)) return false;
    const int64_t kept = (int64_t)h->g.kkeep * h->g.bk, weights = kept * h->g.n / h->g.m, results = (int64_t)h->g.rows * ncols;
    if (kept < kMinKept && weights < kMinWeights && (results < kMinResults || weights < kMinTerms) && results * weights < kMinMacs) return false;
    const TcImageLayout L = tc_image_layout(h->g, h->exec_kind);
    const int64_t tiles = (int64_t)L.nst * ((ncols + kCols - 1) / kCols);
    return tiles <= 0x7FFFFFFF && (uint64_t)L.stack * L.nst * L.wcap * L.entry_bytes / 256 < (1ull << 31);
}

cudaError_t launch_spmm_gather(crisp_handle_s *h, const uint16_t *d_x, int64_t ldx, int64_t ncols, void *d_y, int64_t ldy,
                               cudaStream_t st) {
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    const uint64_t moment = encodes.now();
    const Geometry &g = h->g;
    const bool sparse = h->exec_kind == CRISP_PATH_SPARSE;
    const TcImageLayout L = tc_image_layout(g, h->exec_kind);
    CUtensorMap image;
    RowMaps rows;
    {
        std::lock_guard<std::mutex> hold(h->plan_lock);
        if (!h->gather) {
            e = ensure_context(device);
            if (e != cudaSuccess) return e;
            GatherPlan *fresh = new (std::nothrow) GatherPlan;
            if (!fresh) return cudaErrorMemoryAllocation;
            if (!make_map_image(&fresh->image, h->d_exec + L.image_off, (uint64_t)L.stack * L.nst * L.wcap * L.entry_bytes, L.entry_bytes)) {
                delete fresh;
                return cudaErrorNotSupported;
            }
            fresh->x = nullptr;
            h->gather = fresh;
        }
        GatherPlan &plan = *h->gather;
        if (plan.x != d_x || plan.ldx != ldx || plan.ncols != ncols) {
            e = ensure_context(device);
            if (e != cudaSuccess) return e;
            plan.x = nullptr;                                // not valid until all are made
            for (int r = 0; r < 8; ++r) {
                // from the 16-byte boundary in front of row r; a residue without rows gets the first row's matrix (and is read beyond its end)
                const uintptr_t row = reinterpret_cast<uintptr_t>(d_x) + (uintptr_t)(r < g.k ? (int64_t)r * ldx * 2 : 0), at = row & 15u;
                const int64_t n = r < g.k ? (g.k - r + 7) / 8 : 1;
                if (!make_map_rows(&plan.rows.m[r], reinterpret_cast<const void *>(row - at), (uint64_t)(ncols + (int64_t)at / 2), (uint64_t)n,
                                   (uint64_t)ldx * 16, kRawCols, (uint32_t)g.bk / 8))
                    return cudaErrorNotSupported;            // (the caller has another kernel)
            }
            plan.x = d_x; plan.ldx = ldx; plan.ncols = ncols;
        }
        image = plan.image;
        rows = plan.rows;
    }
    const int sms = sm_count_of(device);
    GatherParams p = {};
    p.walk_col = reinterpret_cast<const int32_t *>(h->d_exec + L.walk_col_off);
    p.walk_len = reinterpret_cast<const int32_t *>(h->d_exec + L.walk_len_off);
    p.blk_col = h->d_blk_col; p.vals = h->d_vals; p.idx = h->d_idx;
    p.x = d_x; p.ldx = ldx; p.ncols = ncols;
    p.y = reinterpret_cast<uint16_t *>(d_y); p.ldy = ldy;
    p.bias = h->epilogue.bias; p.relu = h->epilogue.relu;
    p.status = h->d_status; p.g = g;
    p.nst = L.nst; p.wcap = L.wcap;
    p.num_tiles = (int)(L.nst * ((ncols + kCols - 1) / kCols));
    p.a_bytes = L.a_bytes; p.entry_bytes = L.entry_bytes;
    p.stage_bytes = L.entry_bytes + (uint32_t)(kCols * g.bk * 2);
    p.wait_limit = h->wait_limit_cycles ? h->wait_limit_cycles : kWaitLimitCycles;
    p.skip_fill = h->debug_skip_stage;
    p.ahead = g.bk >= 96 ? 1 : 128 / g.bk;
    p.split = 1;
    for (int s = kMaxSplit; s >= 2; s >>= 1)
        if (p.num_tiles * s <= sms * 7 / 8 && L.wcap >= 2 * s) { p.split = s; break; }
    while ((1 << p.split_log2) < p.split) ++p.split_log2;
    const uint32_t fixed = kRawBytes + kEpiWarps * kStageTile + 1024;
    uint32_t stages = (kSmemBudget + 1024 - fixed) / p.stage_bytes;
    if (stages > 8) stages = 8;
    if (stages < 2) return cudaErrorNotSupported;
    p.num_stages = stages;
    const size_t smem = fixed + (size_t)stages * p.stage_bytes;
    const bool wide = ((reinterpret_cast<uintptr_t>(d_x) | (uintptr_t)(ldx * 2)) & 7) == 0;
    const GatherKernel kern = pick(sparse, wide);
    static std::atomic<bool> configured[4][64];
    const int which = (sparse ? 2 : 0) + (wide ? 1 : 0);
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    if (!configured[which][device].load(std::memory_order_relaxed)) {
        // the most there is, once: the limit belongs to the function, not to a call
        e = cudaFuncSetAttribute(reinterpret_cast<const void *>(kern), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBudget + 1024);
        if (e != cudaSuccess) return e;
        configured[which][device].store(true, std::memory_order_relaxed);
    }
    const int grid = p.split > 1 ? p.num_tiles * p.split : (p.num_tiles < sms ? p.num_tiles : sms);
    e = launch_clusters(kern, (unsigned)grid, (unsigned)kThreads, smem, st, (unsigned)p.split, image, rows, p);
    if (e == cudaSuccess) note_launch(h, crisp_launch_info_t{CRISP_PATH_DIRECT, kCols, 2, 1, kEpiWarps, (int)stages, grid, 0, 1}, 0, st, moment);
    return e;
}

}  // namespace crisp
