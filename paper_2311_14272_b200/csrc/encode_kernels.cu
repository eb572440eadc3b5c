// Canonical compressed format of Sec. III-A: kept-block column list (Blocked-ELLPACK) plus,
// per kept value, its bf16 payload and a log2(M)-bit zero-based offset inside its M-vector.
#include "crisp_internal.h"

namespace crisp {

namespace {

// One CTA per entry of the walk list of a 128-row CTA tile of the tensor-core kernel: it writes the canonical blocks
// (values, offsets) of the tile's row tiles that keep the entry's column and, from the same registers, the entry of the
// execution image: the weight tile and the 2:4 metadata of all 128 rows, with zeros (and valid padding metadata) for row
// tiles that do not keep it.  The walk list of a CTA tile is the ascending union of its row tiles' lists: with 128-row
// blocks the list itself, else every CTA marks the union in a bitmap and takes the column at its own position.
//
// A thread takes eight consecutive elements of a row: one 16-byte load and one byte of the mask.  Everything a 4-group
// needs follows from its four mask bits and is looked up in a 16-entry table: byte-permute selectors that move the kept
// values to the front, offset fields, the slot pair of the 2:4 image and its metadata nibble.  Values go straight to
// global memory (consecutive lanes write consecutive bytes), the tile and the offset fields through shared memory;
// every metadata byte belongs to one thread, so there are no atomics on it.  What bounds the kernel is the chain of
// dependent round trips of a CTA (block list, weights, stores), hidden by the five CTAs an SM holds (48 registers, for which
// most forms spill 8 to 48 bytes a thread; with 40 registers they spill more and take 20 us where this takes 14).  A thread keeps its chunk column and goes down the rows: with the row and column of
// every chunk computed anew, and the image chosen at run time, the same work took 22 us.
// Measured: 4096 x 4096, 2:4, keep 0.5, 128 x 64 blocks 14.0 us (36 MB moved); the 13 layers of VGG-16 with 64 x 64 blocks in
// one launch 15.9 us (18 under ncu with a cold L2), where a canonical pass and an image pass over it per layer took 62 + 165 us.
// Shared-memory planes of the tile are padded (2064 or 2080 instead of 2048 bytes), which spreads the eight lanes of a row
// over the banks.
// Image layouts: see the tensor-core SpMM.  Stacked thin layers: copy q of the image holds the rows shifted by
// q * 128 / stack; the copies are written from one staged tile.
constexpr int kTileRows = 128, kMetaTileBytes = 2048;

// What a 4-group needs, by its four mask bits:
//   x  byte-permute selectors that move the kept values to the front in ascending order: 1st and 2nd | 3rd and 4th << 16
//   y  byte-permute selector of the 2:4 slot pair | metadata nibble << 16 | kept count << 24
//   z  2-bit positions of the kept values, ascending | 3-bit positions << 16
//   w  0xFFFF in the slots that carry a value
__device__ __forceinline__ uint4 nibble_entry(uint32_t nib) {
    uint32_t front = 0u, f2 = 0u, f3 = 0u;
    int cnt = 0;
#pragma unroll
    for (int p = 0; p < 4; ++p)
        if ((nib >> p) & 1u) {
            front |= (uint32_t)((2 * p) | ((2 * p + 1) << 4)) << (8 * cnt);
            f2 |= (uint32_t)p << (2 * cnt);
            f3 |= (uint32_t)p << (3 * cnt);
            ++cnt;
        }
    int a = 0, b = 1, va = 0, vb = 0;                        // 2:4 slots: ascending positions, an empty slot padded
    if (nib) {
        const int first = __ffs(nib) - 1;
        const uint32_t rest = nib & (nib - 1);
        if (rest) { a = first; va = 1; b = __ffs(rest) - 1; vb = 1; }
        else if (first == 3) { a = 0; b = 3; vb = 1; }
        else { a = first; va = 1; b = 3; }
    }
    return make_uint4(front,
                      (uint32_t)(2 * a) | ((uint32_t)(2 * a + 1) << 4) | ((uint32_t)(2 * b) << 8) | ((uint32_t)(2 * b + 1) << 12) |
                          ((uint32_t)(a | (b << 2)) << 16) | ((uint32_t)cnt << 24),
                      f2 | (f3 << 16), (va ? 0x0000FFFFu : 0u) | (vb ? 0xFFFF0000u : 0u));
}
// 0xFFFF in the halves whose bit is set
__device__ __forceinline__ uint32_t half_mask(uint32_t two_bits) {
    return ((two_bits & 1u) ? 0x0000FFFFu : 0u) | ((two_bits & 2u) ? 0xFFFF0000u : 0u);
}

// IMAGE: the image the layers of the launch have (CRISP_PATH_DENSE also for layers without one).
template <int M, int N, int IMAGE, int CAP>
__global__ void __launch_bounds__(256, 5)
encode_kernel(const __grid_constant__ Batch<EncodeLayer, CAP> batch) {
    constexpr int V = 8 / M * N, kIdxBits = M == 4 ? 2 : 3, kFieldBits = V * kIdxBits;
    constexpr int kUnroll = 4;
    constexpr bool kSparse = IMAGE == CRISP_PATH_SPARSE;
    extern __shared__ uint4 s_raw4[];
    __shared__ uint4 s_lut[16];
    __shared__ uint32_t s_map[kMaxBlockWords];               // kept columns of the tile (the union)
    __shared__ int s_slot[4];                                // where row tile i keeps this column, or -1
    chain_kernels();
    const int l = batch.find(blockIdx.x);
    const EncodeLayer &L = batch.layer[l];
    const Geometry &g = L.g;
    const int cta = (int)(blockIdx.x - batch.first[l]);
    const int r = kTileRows / g.bm;
    const int per_tile = min(min(r, g.nrt) * g.kkeep, g.nblk);            // most entries of a walk list
    const int st = cta / per_tile, entry = cta - st * per_tile;
    const int first_rt = st * r, n_rt = min(r, g.nrt - first_rt);
    if (cta == 0 && L.header != nullptr && threadIdx.x < 64) L.header[threadIdx.x] = 0u;     // the handle's status block
    const bool lists = L.walk_col != nullptr;
    int jb;
    if (r == 1) {                                            // the walk list is the row tile's kept list
        jb = L.mask_blk_col[(int64_t)st * g.kkeep + entry];
        if (threadIdx.x < 4) s_slot[threadIdx.x] = threadIdx.x == 0 ? entry : -1;
        if (threadIdx.x >= 32 && threadIdx.x < 48) s_lut[threadIdx.x - 32] = nibble_entry(threadIdx.x - 32);
        if (lists && entry == 0 && threadIdx.x == 0) L.walk_len[st] = g.kkeep;
        __syncthreads();
    } else {
        const int map_words = (g.nblk + 31) / 32, listed = n_rt * g.kkeep;
        const int c = threadIdx.x < listed ? L.mask_blk_col[(int64_t)first_rt * g.kkeep + threadIdx.x] : 0;
        for (int i = threadIdx.x; i < map_words; i += blockDim.x) s_map[i] = 0u;
        if (threadIdx.x < 4) s_slot[threadIdx.x] = -1;
        if (threadIdx.x >= 32 && threadIdx.x < 48) s_lut[threadIdx.x - 32] = nibble_entry(threadIdx.x - 32);
        __syncthreads();
        if (threadIdx.x < listed) atomicOr(&s_map[c >> 5], 1u << (c & 31));
        for (int i = threadIdx.x + blockDim.x; i < listed; i += blockDim.x) {
            const int d = L.mask_blk_col[(int64_t)first_rt * g.kkeep + i];
            atomicOr(&s_map[d >> 5], 1u << (d & 31));
        }
        __syncthreads();
        // the column with `entry` kept columns of the union below it
        int word = 0, below = 0, cnt = 0;
        for (; word < map_words; ++word, below += cnt) {
            cnt = __popc(s_map[word]);
            if (below + cnt > entry) break;
        }
        if (lists && entry == 0 && threadIdx.x == 0) {
            int n = 0;
            for (int i = 0; i < map_words; ++i) n += __popc(s_map[i]);
            L.walk_len[st] = n;
        }
        if (word == map_words) return;                       // a shorter list
        uint32_t left = s_map[word];
        for (int i = below; i < entry; ++i) left &= left - 1;
        jb = word * 32 + __ffs(left) - 1;
        if (threadIdx.x < listed && c == jb) { const int q = threadIdx.x / g.kkeep; s_slot[q] = threadIdx.x - q * g.kkeep; }
        for (int i = threadIdx.x + blockDim.x; i < listed; i += blockDim.x)
            if (L.mask_blk_col[(int64_t)first_rt * g.kkeep + i] == jb) { const int q = i / g.kkeep; s_slot[q] = i - q * g.kkeep; }
        __syncthreads();
    }
    if (lists && threadIdx.x == 0) L.walk_col[(int64_t)st * L.wcap + entry] = jb;
    if (threadIdx.x < n_rt && s_slot[threadIdx.x] >= 0)
        L.blk_col[(int64_t)(first_rt + threadIdx.x) * g.kkeep + s_slot[threadIdx.x]] = jb;

    const int c8n = g.bk / 8;                                // a chunk: eight elements of a row
    const bool image = kSparse || L.kind == CRISP_PATH_DENSE;
    // staged tile: planes of 8 columns (one per 16-byte chunk of a row) with 128 rows of 16 bytes
    constexpr uint32_t kPlane = kSparse ? 2080u : 2064u;
    const int planes = kSparse ? c8n / 2 : c8n;
    const uint32_t meta_at = (uint32_t)planes * kPlane, addend_bytes = meta_at + (kSparse ? kMetaTileBytes : 0);
    const int addends = kSparse && N > 2 ? 2 : 1;
    uint8_t *tile = reinterpret_cast<uint8_t *>(s_raw4);
    uint32_t *s_field = reinterpret_cast<uint32_t *>(tile + (image ? addends * addend_bytes : 0u));    // [128 * c8n]
    if (kSparse && g.bk < 128) {                             // metadata words beyond block_k / 32 per row are zero
        for (int i = threadIdx.x; i < addends * kMetaTileBytes / 16; i += blockDim.x) {
            const int a = i / (kMetaTileBytes / 16);
            reinterpret_cast<uint4 *>(tile + a * addend_bytes + meta_at)[i - a * (kMetaTileBytes / 16)] = make_uint4(0u, 0u, 0u, 0u);
        }
        __syncthreads();
    }
    const int groups = g.bk / M, vpb = g.bm * groups * N, bm_log2 = 31 - __clz(g.bm);
    // a thread keeps its chunk column and goes down the rows, so that all addresses advance by constants
    const int step = blockDim.x / c8n, c8 = threadIdx.x % c8n, row_first = threadIdx.x / c8n;
    const int64_t col = (int64_t)jb * g.bk + 8 * c8;
    const bool wide = L.vec_ok && col + 8 <= g.k;
    const int64_t grow = (int64_t)st * kTileRows;
    const uint8_t *bits_col = reinterpret_cast<const uint8_t *>(L.nm_bits + grow * g.wpr) + (col >> 3);
    const uint16_t *w_col = L.w + grow * L.ld + col;
    uint8_t *const tile_col = tile + (kSparse ? (c8 >> 1) * kPlane + (c8 & 1) * 8 : c8 * kPlane);
    const uint32_t meta_col = meta_at + (8 * ((c8 >> 1) & 1) * 4 + (c8 >> 2)) * 4 + (c8 & 1);
    for (int row0 = row_first < step ? row_first : kTileRows; row0 < kTileRows; row0 += kUnroll * step) {
        uint4 wv[kUnroll];
        uint32_t bits[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int row = row0 + u * step;
            wv[u] = make_uint4(0u, 0u, 0u, 0u);
            bits[u] = 0u;
            if (row < kTileRows && s_slot[row >> bm_log2] >= 0) {
                bits[u] = bits_col[(int64_t)row * g.wpr * 4];
                if (grow + row < g.rows) {
                    const uint16_t *p = w_col + row * L.ld;
                    if (wide) {
                        wv[u] = *reinterpret_cast<const uint4 *>(p);
                    } else {
                        uint32_t e[8];
#pragma unroll
                        for (int t = 0; t < 8; ++t) e[t] = col + t < g.k ? (uint32_t)p[t] : 0u;
                        wv[u] = make_uint4(e[0] | (e[1] << 16), e[2] | (e[3] << 16), e[4] | (e[5] << 16), e[6] | (e[7] << 16));
                    }
                }
            }
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
            const int row = row0 + u * step;
            if (row >= kTileRows) break;
            const uint32_t n0 = bits[u] & 15u, n1 = bits[u] >> 4;
            const uint4 t0 = s_lut[n0], t1 = s_lut[n1];
            const int sub = row >> bm_log2, slot = s_slot[sub];
            if (slot >= 0) {
                // canonical: V values and V offset fields, in ascending position
                unsigned long long lo = (unsigned long long)__byte_perm(wv[u].x, wv[u].y, t0.x & 0xFFFFu) |
                                        ((unsigned long long)__byte_perm(wv[u].x, wv[u].y, t0.x >> 16) << 32);
                const unsigned long long q = (unsigned long long)__byte_perm(wv[u].z, wv[u].w, t1.x & 0xFFFFu) |
                                             ((unsigned long long)__byte_perm(wv[u].z, wv[u].w, t1.x >> 16) << 32);
                const int n_lo = M == 4 ? N : (int)(t0.y >> 24);                        // values of the first 4-group
                unsigned long long hi = q;
                if (n_lo != 4) {
                    const int sh = 16 * (n_lo & 3);
                    lo = (lo & ((1ull << sh) - 1ull)) | (q << sh);
                    hi = q >> 1 >> (63 - sh);
                }
                uint16_t *vout = L.vals + (int64_t)((first_rt + sub) * g.kkeep + slot) * vpb + ((row & (g.bm - 1)) * c8n + c8) * V;
                if constexpr (V == 8) {
                    *reinterpret_cast<uint4 *>(vout) = make_uint4((uint32_t)lo, (uint32_t)(lo >> 32), (uint32_t)hi, (uint32_t)(hi >> 32));
                } else if constexpr (V == 4) {
                    *reinterpret_cast<uint2 *>(vout) = make_uint2((uint32_t)lo, (uint32_t)(lo >> 32));
                } else if constexpr (V % 2 == 0) {
#pragma unroll
                    for (int j = 0; j < V; j += 2)
                        *reinterpret_cast<uint32_t *>(vout + j) = (uint32_t)((j < 4 ? lo : hi) >> (16 * (j & 3)));
                } else {
#pragma unroll
                    for (int j = 0; j < V; ++j) vout[j] = (uint16_t)((j < 4 ? lo : hi) >> (16 * (j & 3)));
                }
                uint32_t field;
                if constexpr (M == 4) field = (t0.z & 0xFFu) | ((t1.z & 0xFFu) << (2 * N));
                else                                         // bit 2 of every field of the second 4-group: + 4 each
                    field = (t0.z >> 16) | (((t1.z >> 16) | (0x924u & ((1u << (3 * (t1.y >> 24))) - 1u))) << (3 * n_lo));
                s_field[row * c8n + c8] = field;
            }
            if constexpr (!kSparse) {
                if (image)
                    *reinterpret_cast<uint4 *>(tile_col + row * 16) =
                        make_uint4(wv[u].x & half_mask(n0), wv[u].y & half_mask(n0 >> 2), wv[u].z & half_mask(n1), wv[u].w & half_mask(n1 >> 2));
            } else {
                const uint32_t meta_row = ((row & 7) + 16 * (row >> 4)) * 16 + 2 * ((row >> 3) & 1);
                auto slots = [&](int a, const uint4 &e0, const uint4 &e1) {
                    const uint32_t p0 = __byte_perm(wv[u].x, wv[u].y, e0.y & 0xFFFFu) & e0.w;
                    const uint32_t p1 = __byte_perm(wv[u].z, wv[u].w, e1.y & 0xFFFFu) & e1.w;
                    *reinterpret_cast<uint2 *>(tile_col + a * addend_bytes + row * 16) = make_uint2(p0, p1);
                    tile[a * addend_bytes + meta_col + meta_row] = (uint8_t)(((e0.y >> 16) & 15u) | (((e1.y >> 16) & 15u) << 4));
                };
                if constexpr (N <= 2) slots(0, t0, t1);
                else {                                       // the first two values of a 4-group, then the rest
                    const uint32_t r0 = n0 & (n0 - 1), r1 = n1 & (n1 - 1);
                    const uint32_t s0 = r0 & (r0 - 1), s1 = r1 & (r1 - 1);
                    slots(0, s_lut[n0 ^ s0], s_lut[n1 ^ s1]);
                    slots(1, s_lut[s0], s_lut[s1]);
                }
            }
        }
    }
    __syncthreads();
    // offsets: word w of a block's bit stream holds the fields of chunks from 32 w / kFieldBits on
    const int words = vpb * kIdxBits / 32, block_chunks = g.bm * c8n;
    for (int sub = 0; sub < n_rt; ++sub) {
        if (s_slot[sub] < 0) continue;
        uint32_t *iout = L.idx + ((int64_t)(first_rt + sub) * g.kkeep + s_slot[sub]) * words;
        const uint32_t *f = s_field + sub * block_chunks;
        for (int w = threadIdx.x; w < words; w += blockDim.x) {
            int c = 32 * w / kFieldBits, at = c * kFieldBits - 32 * w;
            uint32_t v = 0u;
#pragma unroll
            for (int j = 0; j < (31 + kFieldBits - 1) / kFieldBits + 1; ++j, ++c, at += kFieldBits)
                if (at < 32 && c < block_chunks) v |= at >= 0 ? f[c] << at : f[c] >> -at;
            iout[w] = v;
        }
    }
    if (!image) return;
    const int window = kTileRows / L.stack;                  // rows a copy of a stacked image carries
    for (int q = 0; q < L.stack; ++q) {
        const int shift = q * window;
        for (int a = 0; a < addends; ++a) {
            const uint8_t *ta = tile + a * addend_bytes;
            uint4 *out = reinterpret_cast<uint4 *>(L.image + ((int64_t)(q * L.nst + st) * L.wcap + entry) * L.entry_bytes +
                                                   (int64_t)a * (L.a_bytes + kMetaTileBytes));
            for (int i = threadIdx.x; i < planes * kTileRows; i += blockDim.x) {
                const int src = (i & (kTileRows - 1)) - shift;
                out[i] = src >= 0 && src < window ? *reinterpret_cast<const uint4 *>(ta + (i >> 7) * kPlane + src * 16) : make_uint4(0u, 0u, 0u, 0u);
            }
            if constexpr (kSparse) {
                const uint32_t pad = 0x44444444u;
                for (int i = threadIdx.x; i < kMetaTileBytes / 16; i += blockDim.x) {
                    const int src = i - shift;
                    out[planes * kTileRows + i] = src >= 0 && src < window
                        ? *reinterpret_cast<const uint4 *>(ta + meta_at + src * 16)
                        : make_uint4(pad, g.bk > 32 ? pad : 0u, g.bk > 64 ? pad : 0u, g.bk > 96 ? pad : 0u);
                }
            }
        }
    }
}

// Dense weights from the canonical format, pruned positions as zero, in one pass over the output (which is what has to
// be written: 2 bytes an element).  A CTA takes 32 rows x 256 elements, a warp four of the rows, a lane eight consecutive
// elements of each: one 16-byte store, 512 consecutive bytes per row and warp.  The values of a lane's eight elements are
// V = 8 N / M consecutive ones of their block and their offsets V consecutive fields, so a lane reads both with a load or
// two and shifts every value to its place in registers.  Which slot of the row tile holds a block column is looked up once
// per CTA.  Measured (4096 x 4096, 2:4, keep 0.5; 33 MB out, 19 MB in): 9.8 us, against 25 us + 6 us for a memset
// and a kernel that scattered 2-byte values one by one with three integer divisions each.  (A fill of as much takes
// 10.8: writing is most of it.)  Several slabs of 32 rows a CTA, the next one's loads ahead, gained nothing.
// With one or two values a group a byte permute puts a pair of values into a word of the result, and what it does follows from the group's offset
// fields: a table of selectors in shared memory, 2 bytes for a word of two elements.  (Placing value by value with 64-bit shifts, as from three values a group on, took 160
// instructions a lane and row, two thirds of the issue slots, and 11.3 us.  That form is kept there as it was.)
constexpr int kDecodeRows = 32, kDecodeCols = 256;
// Selectors of the words of a group of M whose fields are `code`: value j (bytes 2 j, 2 j + 1) where field j says, zero (bytes 4..) elsewhere.
template <int M, int N>
__device__ __forceinline__ uint2 place_selectors(uint32_t code) {
    constexpr int kBits = M == 4 ? 2 : 3;
    uint32_t sel[4] = {0x4444u, 0x4444u, 0x4444u, 0x4444u};
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const int at = (int)(code >> (kBits * j)) & (M - 1);
        const uint32_t mask = 0xFFu << (8 * (at & 1)), take = (uint32_t)(2 * j | (2 * j + 1) << 4) << (8 * (at & 1));
#pragma unroll
        for (int w = 0; w < M / 2; ++w)
            if (at >> 1 == w) sel[w] = (sel[w] & ~mask) | take;
    }
    return make_uint2(sel[0] | sel[1] << 16, sel[2] | sel[3] << 16);
}

template <int M, int N>
__global__ void __launch_bounds__(256)
decode_kernel(Geometry g, const int32_t *blk_col, const uint16_t *vals, const uint32_t *idx, uint16_t *w, int64_t ld,
              bool vec_ok, int chunks) {
    constexpr int V = 8 / M * N, kBits = M == 4 ? 2 : 3, kRows = kDecodeRows / 8;
    constexpr bool kTable = N <= 2;
    constexpr int kCodes = 1 << (N * kBits);
    __shared__ int s_slot[kDecodeCols / 32];
    __shared__ uint2 s_place[kTable ? kCodes : 1];
    if (kTable && threadIdx.x < kCodes) s_place[threadIdx.x] = place_selectors<M, N>(threadIdx.x);
    chain_kernels();
    const int rg = blockIdx.x / chunks, chunk = blockIdx.x - rg * chunks;
    const int row0 = rg * kDecodeRows, rt = row0 / g.bm;
    const int jb0 = chunk * kDecodeCols / g.bk;
    if (threadIdx.x < kDecodeCols / 32) s_slot[threadIdx.x] = -1;
    __syncthreads();
    for (int i = threadIdx.x; i < g.kkeep; i += blockDim.x) {
        const int d = blk_col[(int64_t)rt * g.kkeep + i] - jb0;
        if (d >= 0 && d < kDecodeCols / 32) s_slot[d] = i;          // (block columns beyond the chunk do no harm)
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int k0 = chunk * kDecodeCols + lane * 8;
    if (k0 >= g.k) return;
    const int jb = k0 / g.bk, slot = s_slot[jb - jb0];
    const int first = row0 + warp * kRows;
    if constexpr (kTable) {
        uint32_t v[kRows][(V + 1) / 2], f[kRows];                // values two a word, offset fields
        if (slot >= 0) {
            const int vpb = (int)g.vals_per_block(), vpr = g.groups() * N;
            const int64_t blk = (int64_t)rt * g.kkeep + slot;
            const int o0 = (first - rt * g.bm) * vpr + (k0 - jb * g.bk) / M * N;             // (rows of padding are stored too)
            const uint16_t *vin = vals + blk * vpb + o0;
            const uint32_t *iin = idx + blk * (vpb * kBits / 32);
#pragma unroll
            for (int i = 0; i < kRows; ++i, vin += vpr) {
                if constexpr (V == 4) {
                    const uint2 t = *reinterpret_cast<const uint2 *>(vin);
                    v[i][0] = t.x; v[i][1] = t.y;
                } else if constexpr (V == 2) {
                    v[i][0] = *reinterpret_cast<const uint32_t *>(vin);
                } else {
                    v[i][0] = *vin;
                }
                const int bit = (o0 + i * vpr) * kBits;
                uint32_t t = iin[bit >> 5] >> (bit & 31);
                if (32 % (V * kBits) != 0 && (bit & 31) + V * kBits > 32) t |= iin[(bit >> 5) + 1] << (32 - (bit & 31));
                f[i] = t;
            }
        }
        uint16_t *dst = w + (int64_t)first * ld + k0;
#pragma unroll
        for (int i = 0; i < kRows; ++i, dst += ld) {
            if (first + i >= g.rows) break;
            uint4 out = make_uint4(0u, 0u, 0u, 0u);              // the row's eight elements
            if (slot >= 0) {
                if constexpr (M == 4) {
                    const uint32_t e0 = s_place[f[i] & (kCodes - 1)].x, e1 = s_place[(f[i] >> (N * kBits)) & (kCodes - 1)].x;
                    const uint32_t w0 = v[i][0], w1 = N == 1 ? v[i][0] >> 16 : v[i][N - 1];
                    out = make_uint4(__byte_perm(w0, 0u, e0 & 0xFFFFu), __byte_perm(w0, 0u, e0 >> 16), __byte_perm(w1, 0u, e1 & 0xFFFFu), __byte_perm(w1, 0u, e1 >> 16));
                } else {
                    const uint2 e = s_place[f[i] & (kCodes - 1)];
                    const uint32_t w0 = v[i][0];
                    out = make_uint4(__byte_perm(w0, 0u, e.x & 0xFFFFu), __byte_perm(w0, 0u, e.x >> 16), __byte_perm(w0, 0u, e.y & 0xFFFFu), __byte_perm(w0, 0u, e.y >> 16));
                }
            }
            if (vec_ok && k0 + 8 <= g.k) {
                *reinterpret_cast<uint4 *>(dst) = out;
            } else {
                const uint32_t word[4] = {out.x, out.y, out.z, out.w};
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (k0 + j < g.k) dst[j] = (uint16_t)(word[j >> 1] >> (16 * (j & 1)));
            }
        }
    } else {
        uint16_t v[kRows][V];
        uint32_t f[kRows];
        if (slot >= 0) {
            const int vpb = (int)g.vals_per_block(), groups = g.groups();
            const int64_t blk = (int64_t)rt * g.kkeep + slot;
            const uint16_t *vin = vals + blk * vpb;
            const uint32_t *iin = idx + blk * (vpb * kBits / 32);
#pragma unroll
            for (int i = 0; i < kRows; ++i) {
                const int o = ((first + i - rt * g.bm) * groups + (k0 - jb * g.bk) / M) * N;     // (rows of padding are stored too)
                if constexpr (V == 8) {
                    const uint4 t = *reinterpret_cast<const uint4 *>(vin + o);
                    v[i][0] = (uint16_t)t.x; v[i][1] = (uint16_t)(t.x >> 16); v[i][2] = (uint16_t)t.y; v[i][3] = (uint16_t)(t.y >> 16);
                    v[i][4] = (uint16_t)t.z; v[i][5] = (uint16_t)(t.z >> 16); v[i][6] = (uint16_t)t.w; v[i][7] = (uint16_t)(t.w >> 16);
                } else if constexpr (V == 4) {
                    const uint2 t = *reinterpret_cast<const uint2 *>(vin + o);
                    v[i][0] = (uint16_t)t.x; v[i][1] = (uint16_t)(t.x >> 16); v[i][2] = (uint16_t)t.y; v[i][3] = (uint16_t)(t.y >> 16);
                } else if constexpr (V % 2 == 0) {
#pragma unroll
                    for (int j = 0; j < V; j += 2) {
                        const uint32_t t = *reinterpret_cast<const uint32_t *>(vin + o + j);
                        v[i][j] = (uint16_t)t; v[i][j + 1] = (uint16_t)(t >> 16);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < V; ++j) v[i][j] = vin[o + j];
                }
                const int bit = o * kBits;
                uint32_t t = iin[bit >> 5] >> (bit & 31);
                if (32 % (V * kBits) != 0 && (bit & 31) + V * kBits > 32) t |= iin[(bit >> 5) + 1] << (32 - (bit & 31));
                f[i] = t;
            }
        }
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
            const int row = first + i;
            if (row >= g.rows) break;
            unsigned long long half[2] = {0ull, 0ull};                   // elements 0..3 and 4..7
            if (slot >= 0) {
#pragma unroll
                for (int j = 0; j < V; ++j) {
                    const uint32_t t = (f[i] >> (j * kBits)) & ((1u << kBits) - 1u);
                    const unsigned long long at = (unsigned long long)v[i][j] << (16 * (t & 3u));
                    if constexpr (M == 4) half[j / N] |= at;
                    else { half[0] |= t < 4u ? at : 0ull; half[1] |= t < 4u ? 0ull : at; }
                }
            }
            uint16_t *dst = w + (int64_t)row * ld + k0;
            if (vec_ok && k0 + 8 <= g.k) {
                *reinterpret_cast<uint4 *>(dst) = make_uint4((uint32_t)half[0], (uint32_t)(half[0] >> 32), (uint32_t)half[1], (uint32_t)(half[1] >> 32));
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (k0 + j < g.k) dst[j] = (uint16_t)(half[j >> 2] >> (16 * (j & 3)));
            }
        }
    }
}

}  // namespace

namespace {

size_t encode_smem(const EncodeLayer &L) {
    const size_t c8n = (size_t)L.g.bk / 8, fields = kTileRows * c8n * 4;
    switch (L.kind) {
        case CRISP_PATH_DENSE: return c8n * 2064 + fields;
        case CRISP_PATH_SPARSE: return c8n / 2 * 2080 + kMetaTileBytes + fields;
        case CRISP_PATH_SPARSE2: return 2 * (c8n / 2 * 2080 + kMetaTileBytes) + fields;
        default: return fields;
    }
}

template <int M, int N, int IMAGE, int CAP>
cudaError_t run_encode_image(const Batch<EncodeLayer, CAP> &b, cudaStream_t st) {
    size_t smem = 0;
    for (int i = 0; i < b.n; ++i) smem = encode_smem(b.layer[i]) > smem ? encode_smem(b.layer[i]) : smem;
    if (smem > 40 * 1024) {          // (the kernel's own arrays take some of the default 48 KB)
        cudaError_t e = cudaFuncSetAttribute(encode_kernel<M, N, IMAGE, CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    if (b.first[b.n] == 0) return cudaSuccess;
    if (b.first[b.n] > 0x7FFFFFFFll) return cudaErrorInvalidValue;
    return launch_chained(encode_kernel<M, N, IMAGE, CAP>, (unsigned)b.first[b.n], 256, smem, st, b);
}
template <int M, int N, int CAP>
cudaError_t run_encode(const Batch<EncodeLayer, CAP> &b, cudaStream_t st) {
    // (one addend for n <= 2, two beyond: the kind follows from n, or is dense or none for all layers)
    if (b.layer[0].kind == CRISP_PATH_SPARSE || b.layer[0].kind == CRISP_PATH_SPARSE2)
        return run_encode_image<M, N, CRISP_PATH_SPARSE, CAP>(b, st);
    return run_encode_image<M, N, CRISP_PATH_DENSE, CAP>(b, st);
}

template <int CAP>
cudaError_t run_encode_any(const Batch<EncodeLayer, CAP> &b, cudaStream_t st) {
    const int n = b.layer[0].g.n;
    if (b.layer[0].g.m == 4) {
        switch (n) {
            case 1: return run_encode<4, 1, CAP>(b, st);
            case 2: return run_encode<4, 2, CAP>(b, st);
            case 3: return run_encode<4, 3, CAP>(b, st);
            case 4: return run_encode<4, 4, CAP>(b, st);
        }
    } else {
        switch (n) {
            case 1: return run_encode<8, 1, CAP>(b, st);
            case 2: return run_encode<8, 2, CAP>(b, st);
            case 3: return run_encode<8, 3, CAP>(b, st);
            case 4: return run_encode<8, 4, CAP>(b, st);
            case 5: return run_encode<8, 5, CAP>(b, st);
            case 6: return run_encode<8, 6, CAP>(b, st);
            case 7: return run_encode<8, 7, CAP>(b, st);
            case 8: return run_encode<8, 8, CAP>(b, st);
        }
    }
    return cudaErrorInvalidValue;
}

template <int CAP>
cudaError_t encode_batch(const EncodeLayer *layers, int n, cudaStream_t st) {
    Batch<EncodeLayer, CAP> b;
    b.n = 0;
    b.first[0] = 0;
    for (int i = 0; i < n; ++i) {
        const Geometry &g = layers[i].g;
        if (g.nrt * g.kkeep == 0) continue;                  // nothing kept: nothing to write
        EncodeLayer &L = b.layer[b.n];
        L = layers[i];
        // the 16-byte loads of eight elements need every row to start 16-byte aligned (block columns are multiples of 32)
        L.vec_ok = reinterpret_cast<uintptr_t>(L.w) % 16 == 0 && L.ld % 8 == 0;
        const int64_t tiles = (g.mp() + kTileRows - 1) / kTileRows;
        const int r = kTileRows / g.bm;
        const int64_t entries = (int64_t)(r < g.nrt ? r : g.nrt) * g.kkeep;
        b.first[b.n + 1] = b.first[b.n] + tiles * (entries < g.nblk ? entries : g.nblk);
        ++b.n;
    }
    return b.n ? run_encode_any<CAP>(b, st) : cudaSuccess;
}

}  // namespace

EncodeCount encodes;

namespace {

// If the stream is being captured: the encode counts as one that may happen at any time, from here on until the graph and all that is made from it (it holds a
// reference to the object for each, and until launches under way have finished) are gone.
void count_graph(cudaStream_t st) {
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    cudaGraph_t graph = nullptr;
    const cudaError_t asked = cudaStreamGetCaptureInfo(st, &capture, nullptr, &graph);
    if (asked == cudaSuccess && capture != cudaStreamCaptureStatusActive) return;      // (one that has failed makes no graph)
    encodes.graph_made();
    cudaUserObject_t object;
    if (asked != cudaSuccess || !graph ||
        cudaUserObjectCreate(&object, &encodes, [](void *count) { static_cast<EncodeCount *>(count)->graph_gone(); }, 1u, (unsigned)cudaUserObjectNoDestructorSync) != cudaSuccess)
        return;                                              // (it counts for good)
    if (cudaGraphRetainUserObject(graph, object, 1u, (unsigned)cudaGraphUserObjectMove) != cudaSuccess) {
        encodes.graph_made();                                // (for the reference that is given up)
        cudaUserObjectRelease(object, 1u);
    }
}

}  // namespace

cudaError_t launch_encode(const EncodeLayer *layers, int n, cudaStream_t st) {
    count_graph(st);
    encodes.begin();
    cudaError_t e = cudaSuccess;
    if (n == 1) e = encode_batch<1>(layers, 1, st);
    else
        for (int at = 0; at < n && e == cudaSuccess; at += kBatchLayers)
            e = encode_batch<kBatchLayers>(layers + at, n - at < kBatchLayers ? n - at : kBatchLayers, st);
    encodes.end();
    return e;
}

cudaError_t launch_decode(const Geometry &g, const int32_t *d_blk_col, const uint16_t *d_vals,
                          const uint32_t *d_idx, uint16_t *d_w, int64_t ld, cudaStream_t st) {
    const int chunks = (g.k + kDecodeCols - 1) / kDecodeCols;
    const int64_t ctas = (int64_t)((g.rows + kDecodeRows - 1) / kDecodeRows) * chunks;
    if (ctas > 0x7FFFFFFFll) return cudaErrorInvalidValue;
    const bool vec_ok = reinterpret_cast<uintptr_t>(d_w) % 16 == 0 && ld % 8 == 0;
#define CRISP_DECODE(MV, NV)                                                                                        \
    case NV: return launch_chained(decode_kernel<MV, NV>, (unsigned)ctas, 256, 0, st, g, d_blk_col, d_vals, d_idx, d_w, ld, vec_ok, chunks)
    if (g.m == 4) {
        switch (g.n) { CRISP_DECODE(4, 1); CRISP_DECODE(4, 2); CRISP_DECODE(4, 3); CRISP_DECODE(4, 4); default: return cudaErrorInvalidValue; }
    } else {
        switch (g.n) {
            CRISP_DECODE(8, 1); CRISP_DECODE(8, 2); CRISP_DECODE(8, 3); CRISP_DECODE(8, 4);
            CRISP_DECODE(8, 5); CRISP_DECODE(8, 6); CRISP_DECODE(8, 7); CRISP_DECODE(8, 8);
            default: return cudaErrorInvalidValue;
        }
    }
#undef CRISP_DECODE
}

}  // namespace crisp
