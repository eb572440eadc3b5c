// Global rank selection across layers (Algorithm 1 of the paper, between the block scores and the
// pruning itself; Sec. III-C "Pruning Algorithm"):
//   K-R1  per row of every block-score grid: its scores in increasing order, the o-th smallest added
//         to the layer's rank-column sum c_o (128-bit: sums can pass 2^64);
//   K-R2  global order of all c_o of all layers by their real value c * 2^e (e = the layer's score
//         scale), ties to the lower layer, then the lower rank position; a rank position is pruned
//         while the weight of everything before it in that order is still below the target;
//   K-R3  kkeep = nblk - pruned rank positions, per layer.
// The order is not materialised: for every candidate one warp adds up the weight of the candidates that
// precede it (all pairs, tiled through shared memory).  The lists are small (one entry per rank position per
// layer: hundreds to a few thousand for the networks of Sec. IV), so the quadratic pass costs
// microseconds, is exact, and has no data-dependent control flow.
#include <climits>
#include <cmath>
#include <memory>
#include <new>

#include "crisp_internal.h"

namespace crisp {
namespace {

constexpr int kRankThreads = 256;
constexpr int kRankMaxBlocks = 4096;                 // k-blocks per row tile (one shared-memory row)

struct RankLayer {                                   // device copy of one crisp_rank_layer_t
    const unsigned long long *scores;
    const uint32_t *max_key;
    long long block_elems;
    int nrt, nblk, candidates, entry_off;
    int row_off, pad;                                // first row of the layer among the rows of all layers
};

// One candidate rank position.  Its value c * 2^e is stored normalised, so that the global order is a
// plain lexicographic comparison: `top` = position of the leading bit of the real value (bit length of
// c plus e; INT_MIN for c = 0) and the 128-bit c shifted left until its leading bit is bit 127.  Two
// non-zero values with the same `top` compare like their left-aligned digits; nothing is rounded.
struct RankEntry {
    unsigned long long mhi, mlo;
    unsigned long long weight;                       // weights removed by pruning this rank position
    int top, layer, o, pad;
};

// Exponent of a positive finite float given by its bits (ilogb), denormals included; 0 for zero.
__device__ __forceinline__ int float_bits_exponent(uint32_t key) {
    if (!key) return 0;
    const int e = (int)(key >> 23);
    return e ? e - 127 : (31 - __clz(key)) - 149;
}

__device__ __forceinline__ RankEntry make_entry(unsigned long long lo, unsigned long long hi, int e, int layer, int o,
                                                unsigned long long weight) {
    RankEntry out;
    out.weight = weight; out.layer = layer; out.o = o; out.pad = 0;
    if ((lo | hi) == 0) { out.top = INT_MIN; out.mhi = out.mlo = 0; return out; }
    const int bits = hi ? 128 - __clzll(hi) : 64 - __clzll(lo);
    const int sh = 128 - bits;                       // 0..127
    if (sh >= 64) { out.mhi = lo << (sh - 64); out.mlo = 0; }
    else if (sh) { out.mhi = (hi << sh) | (lo >> (64 - sh)); out.mlo = lo << sh; }
    else { out.mhi = hi; out.mlo = lo; }
    out.top = bits + e;
    return out;
}

// a strictly before b in the global order: value, then layer, then rank position (branch-free, so that
// the loads of consecutive comparisons overlap)
__device__ __forceinline__ bool entry_before(const RankEntry &a, const RankEntry &b) {
    const bool by_pos = (a.layer < b.layer) | ((a.layer == b.layer) & (a.o < b.o));
    const bool by_lo = (a.mlo < b.mlo) | ((a.mlo == b.mlo) & by_pos);
    const bool by_hi = (a.mhi < b.mhi) | ((a.mhi == b.mhi) & by_lo);
    return (a.top < b.top) | ((a.top == b.top) & by_hi);
}

// Increasing bitonic sort of `padded` (a power of two) values in shared memory by `nthreads` threads that
// call it together; `sync` separates the exchange steps (the warp or the whole CTA).
template <typename Sync>
__device__ __forceinline__ void bitonic_sort(unsigned long long *v, int padded, int tid, int nthreads, Sync sync) {
    for (int k = 2; k <= padded; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = tid; i < padded; i += nthreads) {
                const int partner = i ^ j;
                if (partner > i) {
                    const unsigned long long a = v[i], b = v[partner];
                    if ((a > b) == ((i & k) == 0)) { v[i] = b; v[partner] = a; }
                }
            }
            sync();
        }
}

constexpr int kCountRowMax = 512;                    // rows up to this length are ranked by counting, longer ones sorted

// K-R1.  One CTA per row of a block-score grid: the row's scores in increasing order, each added to the rank-column sum of
// its position.  A sum can pass 2^64, so the low and the high half of the scores are summed apart, by 64-bit atomics
// (integers: any order gives the same sum).  Rows of up to 512 blocks are ranked by counting the scores that come before
// (ties by position, which changes nothing in the sums): no exchange steps, one barrier.  All rows of all layers are CTAs
// of one launch: 5.5 us for the 13 layers of VGG-16, 21 us when one CTA per layer went through the layer's rows.
__global__ void __launch_bounds__(kRankThreads)
rank_columns_kernel(const RankLayer *__restrict__ layers, int n_layers, ulonglong2 *__restrict__ sums) {
    __shared__ unsigned long long s_row[kRankMaxBlocks];
    int lo = 0, hi = n_layers - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (layers[mid].row_off <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
    }
    const RankLayer L = layers[lo];
    const unsigned long long *row = L.scores + (long long)((int)blockIdx.x - L.row_off) * L.nblk;
    auto add = [&](int o, unsigned long long v) {
        if (o >= L.candidates) return;
        unsigned long long *c = reinterpret_cast<unsigned long long *>(sums + L.entry_off + o);
        atomicAdd(c, v & 0xFFFFFFFFull);
        atomicAdd(c + 1, v >> 32);
    };
    if (L.nblk <= kCountRowMax) {
        for (int i = threadIdx.x; i < L.nblk; i += kRankThreads) s_row[i] = row[i];
        __syncthreads();
        for (int i = threadIdx.x; i < L.nblk; i += kRankThreads) {
            const unsigned long long mine = s_row[i];
            int rank = 0;
#pragma unroll 4
            for (int j = 0; j < L.nblk; ++j) {
                const unsigned long long o = s_row[j];
                rank += (o < mine) | ((o == mine) & (j < i));
            }
            add(rank, mine);
        }
        return;
    }
    int padded = 1;
    while (padded < L.nblk) padded <<= 1;
    for (int i = threadIdx.x; i < padded; i += kRankThreads) s_row[i] = i < L.nblk ? row[i] : ~0ull;
    __syncthreads();
    bitonic_sort(s_row, padded, threadIdx.x, kRankThreads, [] { __syncthreads(); });
    for (int o = threadIdx.x; o < L.candidates; o += kRankThreads) add(o, s_row[o]);
}

// K-R1 of layers that a CTA holds in shared memory, with the candidates made from it: a thread a score, whose rank is its place in the row, then
// a thread a column.  No sums in global memory, so nothing to clear, and the table travels as a kernel parameter: a copy, a memset and two
// kernels less in front of the selection.  Bound by latency (the longest layer's row, some 10 cycles a score of it, and the launch).
// Measured (13 layers of VGG-16, us): 4.8 where copy, memset and the two kernels below took 0.9 + 1.5 + 4.1 + 3.0 and the gaps between them, some 8.
// The line: a score is compared with its row by one thread, so a layer's 2^19 comparisons are some 500 a thread, 5 us; beyond, and for more layers than the
// parameter holds, rows are CTAs of their own (4096 x 4096 in 32 x 32 blocks is 2^21).
constexpr int kRankLayers = 64, kRankScores = 2560, kRankLayerThreads = 1024;
constexpr long long kRankCompares = 1 << 19;         // of a layer: each score with the others of its row
struct RankTable { RankLayer layer[kRankLayers]; };
__global__ void __launch_bounds__(kRankLayerThreads)
rank_layer_kernel(const __grid_constant__ RankTable table, RankEntry *entries, int32_t *kkeep) {
    __shared__ unsigned long long s_score[kRankScores], s_sorted[kRankScores];
    wait_for_prerequisites();
    const RankLayer &L = table.layer[blockIdx.x];
    const int n = L.nrt * L.nblk;
    for (int i = threadIdx.x; i < n; i += kRankLayerThreads) s_score[i] = L.scores[i];
    if (threadIdx.x == 0) kkeep[blockIdx.x] = L.nblk;        // the selection takes the pruned positions off
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kRankLayerThreads) {
        const int at = i % L.nblk;
        const unsigned long long *row = s_score + (i - at), mine = s_score[i];
        int rank = 0;
#pragma unroll 4
        for (int j = 0; j < L.nblk; ++j) {
            const unsigned long long o = row[j];
            rank += (o < mine) | ((o == mine) & (j < at));
        }
        s_sorted[i - at + rank] = mine;
    }
    __syncthreads();
    const int e = float_bits_exponent(*L.max_key);
    for (int o = threadIdx.x; o < L.candidates; o += kRankLayerThreads) {
        unsigned long long lo = 0ull, hi = 0ull;
        for (int r = 0; r < L.nrt; ++r) {
            const unsigned long long v = s_sorted[r * L.nblk + o];
            lo += v;
            hi += lo < v;
        }
        entries[L.entry_off + o] = make_entry(lo, hi, e, (int)blockIdx.x, o, (unsigned long long)L.nrt * (unsigned long long)L.block_elems);
    }
}
bool rank_layer_fits(const RankLayer &L) {
    return (long long)L.nrt * L.nblk <= kRankScores && (long long)L.nrt * L.nblk * L.nblk <= kRankCompares;
}

// The candidates in the form they are compared in.
__global__ void __launch_bounds__(kRankThreads)
rank_entries_kernel(const RankLayer *__restrict__ layers, int n_layers, int n, const ulonglong2 *__restrict__ sums,
                    RankEntry *__restrict__ entries, int32_t *__restrict__ kkeep) {
    const int i = blockIdx.x * kRankThreads + threadIdx.x;
    if (i < n_layers) kkeep[i] = layers[i].nblk;             // K-R3 starts here: the selection takes the pruned positions off
    if (i >= n) return;
    int lo = 0, hi = n_layers - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (layers[mid].entry_off <= i) lo = mid; else hi = mid - 1;
    }
    const RankLayer L = layers[lo];
    const ulonglong2 c = sums[i];
    const unsigned long long low = c.x + (c.y << 32), high = (c.y >> 32) + (low < c.x);
    entries[i] = make_entry(low, high, float_bits_exponent(*L.max_key), lo, i - L.entry_off,
                            (unsigned long long)L.nrt * (unsigned long long)L.block_elems);
}

// K-R2.  One warp per candidate i: the lanes share out the other candidates (tiled through shared memory),
// each adds up the weight of those that precede i in the global order, and a shuffle reduction gives the
// weight pruned before i.
__global__ void __launch_bounds__(kRankThreads)
global_select_kernel(const RankEntry *entries, int n, unsigned long long target, int32_t *kkeep) {
    __shared__ RankEntry s_tile[kRankThreads];
    wait_for_prerequisites();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int i = blockIdx.x * (kRankThreads / 32) + warp;
    RankEntry mine;
    mine.top = 0; mine.mhi = mine.mlo = 0; mine.layer = mine.o = 0;
    if (i < n) mine = entries[i];
    unsigned long long before = 0;
    for (int base = 0; base < n; base += kRankThreads) {
        if (base + (int)threadIdx.x < n) s_tile[threadIdx.x] = entries[base + threadIdx.x];
        __syncthreads();
        const int cnt = min(kRankThreads, n - base);
#pragma unroll 4
        for (int j = lane; j < cnt; j += 32) {
            const RankEntry other = s_tile[j];
            before += entry_before(other, mine) ? other.weight : 0ull;
        }
        __syncthreads();
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) before += __shfl_xor_sync(0xFFFFFFFFu, before, d);
    if (i < n && lane == 0 && before < target) atomicSub(&kkeep[mine.layer], 1);
}

struct RankLayout {
    size_t table_off, sums_off, entries_off, total;
    long long n_entries, n_rows;
};

crisp_status_t rank_layout(int32_t n_layers, const crisp_rank_layer_t *layers, RankLayout *out) {
    if (n_layers <= 0 || !layers) return CRISP_INVALID_ARG;
    long long n = 0, rows = 0;
    for (int l = 0; l < n_layers; ++l) {
        const crisp_rank_layer_t &L = layers[l];
        if (L.nrt <= 0 || L.nblk <= 0 || L.block_elems <= 0) return CRISP_BAD_SHAPE;
        if (L.min_keep < 0 || L.min_keep > L.nblk) return CRISP_INVALID_ARG;
        if (L.nblk > kRankMaxBlocks) return CRISP_UNSUPPORTED;
        n += L.nblk - L.min_keep;
        rows += L.nrt;
    }
    if (n > 0x7FFFFFFF || rows > 0x7FFFFFFF) return CRISP_UNSUPPORTED;
    out->n_rows = rows;
    out->n_entries = n;
    out->table_off = 0;
    out->sums_off = align_up((size_t)n_layers * sizeof(RankLayer));
    out->entries_off = out->sums_off + align_up((size_t)(n > 0 ? n : 1) * sizeof(ulonglong2));
    out->total = out->entries_off + align_up((size_t)(n > 0 ? n : 1) * sizeof(RankEntry));
    return CRISP_OK;
}

}  // namespace
}  // namespace crisp

using crisp::RankEntry;
using crisp::RankLayer;
using crisp::RankLayout;

extern "C" {

CRISP_API crisp_status_t crisp_global_rank_sizes(int32_t n_layers, const crisp_rank_layer_t *layers,
                                                 size_t *workspace_bytes) {
    if (!workspace_bytes) return CRISP_INVALID_ARG;
    RankLayout lay;
    crisp_status_t s = crisp::rank_layout(n_layers, layers, &lay);
    if (s != CRISP_OK) return s;
    *workspace_bytes = lay.total;
    return CRISP_OK;
}

CRISP_API crisp_status_t crisp_global_rank(int32_t n_layers, const crisp_rank_layer_t *layers, double prune_fraction,
                                           void *d_workspace, int32_t *d_kkeep, void *stream) {
    RankLayout lay;
    crisp_status_t s = crisp::rank_layout(n_layers, layers, &lay);
    if (s != CRISP_OK) return s;
    if (!d_workspace || !d_kkeep || reinterpret_cast<uintptr_t>(d_workspace) % crisp::kAlign) return CRISP_INVALID_ARG;
    if (!(prune_fraction >= 0.0 && prune_fraction <= 1.0)) return CRISP_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    // A table that does not fit a kernel parameter is staged from a temporary host array, so the call cannot be part of a stream capture
    // (the graph would keep a pointer to memory that is gone when it is replayed); smaller ones neither, so that no size decides it.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) return CRISP_CUDA_ERROR;
    if (cap != cudaStreamCaptureStatusNone) return CRISP_UNSUPPORTED;
    std::unique_ptr<RankLayer[]> table(new (std::nothrow) RankLayer[(size_t)n_layers]);
    if (!table) return CRISP_CUDA_ERROR;
    double total = 0.0;
    int off = 0, row_off = 0;
    for (int l = 0; l < n_layers; ++l) {
        const crisp_rank_layer_t &L = layers[l];
        if (!L.d_scores || !L.d_max_key) return CRISP_INVALID_ARG;
        table[l].scores = L.d_scores;
        table[l].max_key = L.d_max_key;
        table[l].block_elems = L.block_elems;
        table[l].nrt = L.nrt; table[l].nblk = L.nblk;
        table[l].candidates = L.nblk - L.min_keep;
        table[l].entry_off = off;
        table[l].row_off = row_off; table[l].pad = 0;
        off += table[l].candidates;
        row_off += L.nrt;
        total += (double)L.nrt * (double)L.nblk * (double)L.block_elems;
    }
    const unsigned long long target = (unsigned long long)floor(prune_fraction * total + 0.5);
    uint8_t *ws = reinterpret_cast<uint8_t *>(d_workspace);
    RankLayer *d_table = reinterpret_cast<RankLayer *>(ws + lay.table_off);
    ulonglong2 *d_sums = reinterpret_cast<ulonglong2 *>(ws + lay.sums_off);
    RankEntry *d_entries = reinterpret_cast<RankEntry *>(ws + lay.entries_off);
    const int n = (int)lay.n_entries;
    bool fits = n_layers <= crisp::kRankLayers;
    for (int l = 0; l < n_layers && fits; ++l) fits = crisp::rank_layer_fits(table[l]);
    if (fits) {
        crisp::RankTable param;
        for (int l = 0; l < n_layers; ++l) param.layer[l] = table[l];
        if (crisp::launch_chained(crisp::rank_layer_kernel, (unsigned)n_layers, crisp::kRankLayerThreads, 0, st, param, d_entries, d_kkeep) != cudaSuccess)
            return CRISP_CUDA_ERROR;
    } else {
        // the table is read from pageable host memory: the call returns once it has been staged
        if (cudaMemcpyAsync(d_table, table.get(), (size_t)n_layers * sizeof(RankLayer), cudaMemcpyHostToDevice, st) != cudaSuccess)
            return CRISP_CUDA_ERROR;
        if (n > 0) {
            if (cudaMemsetAsync(d_sums, 0, (size_t)n * sizeof(ulonglong2), st) != cudaSuccess) return CRISP_CUDA_ERROR;
            crisp::rank_columns_kernel<<<(unsigned)lay.n_rows, crisp::kRankThreads, 0, st>>>(d_table, n_layers, d_sums);
        }
        const int most = n > n_layers ? n : n_layers;
        crisp::rank_entries_kernel<<<(most + crisp::kRankThreads - 1) / crisp::kRankThreads, crisp::kRankThreads, 0, st>>>(
            d_table, n_layers, n, d_sums, d_entries, d_kkeep);
    }
    if (n > 0 && crisp::launch_chained(crisp::global_select_kernel, (unsigned)((n + crisp::kRankThreads / 32 - 1) / (crisp::kRankThreads / 32)), crisp::kRankThreads,
                                       0, st, (const RankEntry *)d_entries, n, target, d_kkeep) != cudaSuccess)
        return CRISP_CUDA_ERROR;
    return cudaGetLastError() == cudaSuccess ? CRISP_OK : CRISP_CUDA_ERROR;
}

CRISP_API crisp_status_t crisp_mask_scores(const crisp_layer_desc_t *desc, const void *d_workspace,
                                           const unsigned long long **d_scores, const uint32_t **d_max_key) {
    if (!desc || !d_workspace || !d_scores || !d_max_key) return CRISP_INVALID_ARG;
    size_t mask_bytes = 0, ws_bytes = 0;
    crisp_status_t s = crisp_mask_sizes(desc, &mask_bytes, &ws_bytes);
    if (s != CRISP_OK) return s;
    const uint8_t *ws = reinterpret_cast<const uint8_t *>(d_workspace);
    *d_max_key = reinterpret_cast<const uint32_t *>(ws);
    *d_scores = reinterpret_cast<const unsigned long long *>(ws + crisp::kAlign);
    return CRISP_OK;
}

}  // extern "C"
