// Convolution with NHWC results in which the filter taps share one load of the activation.
//
// The gather of spmm_tc.cu loads the pixels of a column tile once for every kept block, so a 3x3 filter brings most of them
// several times, from lines of L2 that no other SM reads: that rate is what bounded it (3x3, 64 channels, 224 x 224 x 16, 4 of
// 9 taps kept: 417 MB at 6.6 TB/s).  Here a tile brings, for each slab of 64 channels that any of its blocks keeps, the pixel box with
// its border once, and every tap multiplies the same tile at a shifted start.  That works without moving data because the
// operand tile is a run of pixels of 128 bytes each, swizzled by address bits 7..9: a tap (i, j) begins (i * tb * pw + j) pixels
// further on, and the groups of eight pixels that the MMA takes (one image row of the 8-pixel-wide tile each) are pw pixels
// apart, pw = 8 + kernel width - 1.  Images of one tile are interleaved by rows ([y][image][x]), so the groups of a tile are
// evenly spaced for any number of images.
// What bounds it: for one slab and few taps HBM (64 -> 64 channels, 224 x 224 x 16, 4 taps: 241 MB in 36.3 us when replayed from a graph, 56.3 with the
// gather; 46.6 and 63.7 on buffers that L2 does not hold); for long walks shared memory, which takes 288 cycles to feed the two
// sparse MMAs of an entry (144 each, measured) and some 150 to take in its weight tile and its share of the activation, of 440 in all.
// A tile is 224 pixels (28 rows of 8, or 14 rows of two images, 7 of four): the image sizes that are multiples of 7 come out even, and two
// accumulators fit beside the metadata of the sparse image, so that a tile's results leave under the next one's MMAs; 256 pixels
// where that makes fewer waves of tiles, 128 or 64 where few tiles would leave SMs without one.
// The walk is taken slab by slab (the list is put in that order when a CTA starts); the weight tiles come through a ring of
// their own, or stay when there is one CTA tile of rows and the ring holds its whole walk.
// Results: a warp takes 32 channels x 32 pixels from tensor memory in the layout of the transposing matrix store (stmatrix),
// which writes them channel-fastest without a conflict (64-byte swizzle), and a bulk tensor store brings them out.
#include <cuda.h>
#include <cuda_bf16.h>

#include <atomic>
#include <new>

#include "crisp_internal.h"
#include "tc_common.cuh"

namespace crisp {

using namespace tc;

namespace {

constexpr int kEpiWarps = 16, kThreads = 32 * (3 + kEpiWarps);      // weights, MMA issuer, epilogue, activations
constexpr uint32_t kStgTile = 2048;                                 // 32 pixels x 32 channels
// Walk entries per stage of the weight ring: a stage costs the MMA issuer a wait and a commit, some 120 of the 500 cycles that an
// entry took with one of each (the tensor core needs about 320).
constexpr int kGroup = 2;
constexpr uint32_t kMaxStages = 4;
constexpr uint32_t kListBytes = 8192;
constexpr int kMaxRowTiles = 32;

struct HaloParams {
    const int32_t *walk_col, *walk_len;
    const float *bias;
    int32_t *status;
    int relu, rows;
    int nst, wcap, num_tiles;
    int cpt, kw, pad;                    // slabs of 64 channels; filter width; zero padding
    int th, tb, tb_log2, pw;             // tile: 8 x th pixels of tb images; pixels of a row with its border
    int tiles_x, tiles_y;                // per image
    int wo, ho, batch;
    uint32_t a_bytes, entry_bytes, x_bytes, x_stage, x_stages, w_stages;       // (a stage of weights: kGroup entries)
    int resident;
    int early;                           // weight tiles and walks may be read before the kernel in front has finished (settled.h)
    uint16_t *y;
    int64_t ldy;
    // From this channel on (a multiple of 32) results are stored pixel by pixel: all where TMA cannot address the pixels (pitch or base not a
    // multiple of 16 bytes), the last 32 or fewer where their number is not a multiple of 8: TMA clips at 16 bytes, and what lies
    // behind the last channel is the caller's.
    int plain_from;
    unsigned long long wait_limit;
    int skip_fill;                       // test hook: this load of the activation is left out (-1 = none)
};

struct Tile { int x, y, b; };
__device__ __forceinline__ Tile tile_at(const HaloParams &p, int ct) {
    const int per_image = p.tiles_x * p.tiles_y, bb = ct / per_image, r = ct - bb * per_image, by = r / p.tiles_x;
    return Tile{(r - by * p.tiles_x) * 8, by * p.th, bb * p.tb};
}

// 16 rows of tensor memory x 32 columns: of every 8 columns a thread gets columns 2 (t % 4), + 1 of rows t / 4 and t / 4 + 8
__device__ __forceinline__ void tmem_ld_16x32(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr) : "memory");
}
// four 8x8 matrices of 16-bit elements, transposed: lane l gives the address of row l % 8 of matrix l / 8
__device__ __forceinline__ void store_matrices(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// ----------------------------------------------------------------------------------- kernel
//
// Shared memory: x_stages x [pixel box with border] | w_stages x 2 x [weight tile | metadata] | 16 staging tiles | barriers | walks
// kPlain: some channels are stored pixel by pixel (HaloParams::plain_from)
template <int kN, bool kSparse, bool kPlain>
__global__ void __launch_bounds__(kThreads, 1)
spmm_halo_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_y,
                 const __grid_constant__ CUtensorMap map_a, const __grid_constant__ HaloParams p) {
    constexpr int kMetaCols = kSparse ? 4 * kGroup * (int)kMaxStages : 0;                // metadata of a ring full of entries
    constexpr int kAcc = 2 * kN + kMetaCols <= 512 ? 2 : 1;
    constexpr int kChunks = kN / 32;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    if (base & 1023u) {                                      // swizzled operand tiles need it
        wait_for_prerequisites();
        if (threadIdx.x == 0) atomicCAS(p.status, 0, (int)CRISP_CUDA_ERROR);
        return;
    }
    const uint32_t w_ring = base + p.x_stages * p.x_stage, staging = w_ring + p.w_stages * kGroup * p.entry_bytes;
    const uint32_t ctrl = staging + kEpiWarps * kStgTile;
    uint8_t *ctrl_gen = smem_raw + (ctrl - base);              // (512 bytes, then the walks)
    const uint32_t x_full = ctrl, x_empty = ctrl + 64, w_full = ctrl + 128, w_empty = ctrl + 192, t_full = ctrl + 256, t_empty = ctrl + 272;
    volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(ctrl_gen + 288);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(ctrl_gen + 292);
    // a walk in the order of slabs: x = entry | first of its slab << 30 | last << 31, y = slab << 16 | start of the tap
    int2 *s_walk = reinterpret_cast<int2 *>(ctrl_gen + 512);
    int32_t *s_len = reinterpret_cast<int32_t *>(ctrl_gen + 320);                      // [kMaxRowTiles] lengths of the walks
    int32_t *s_cols = reinterpret_cast<int32_t *>(smem_raw + (staging - base));        // (the staging tiles are not in use yet)

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp == 1) {
        tmem_alloc(smem_u32(const_cast<uint32_t *>(tmem_slot)), 512);
        tmem_relinquish();
    }
    if (threadIdx.x == 0) {
        prefetch_tensormap(&map_a);
        prefetch_tensormap(&map_x);
        if (!kPlain || p.plain_from > 0) prefetch_tensormap(&map_y);
        for (uint32_t s = 0; s < p.x_stages; ++s) { mbar_init(x_full + 8 * s, 1); mbar_init(x_empty + 8 * s, 1); }
        for (uint32_t s = 0; s < p.w_stages; ++s) { mbar_init(w_full + 8 * s, 1); mbar_init(w_empty + 8 * s, 1); }
        for (int a = 0; a < kAcc; ++a) { mbar_init(t_full + 8 * a, 1); mbar_init(t_empty + 8 * a, kEpiWarps); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // (where the weights have not just been encoded, the walks and the first weight tiles come while the kernel in front finishes)
    if (!p.early) wait_for_prerequisites();
    for (int i = threadIdx.x; i < p.nst * p.wcap; i += kThreads) {
        const int jb = __ldcg(p.walk_col + i), tap = jb / p.cpt, ti = tap / p.kw;
        s_cols[i] = (jb - tap * p.cpt) << 16 | ((ti * p.tb * p.pw + tap - ti * p.kw) * 8);       // slab | start of the tap
    }
    if ((int)threadIdx.x < p.nst) s_len[threadIdx.x] = min(__ldcg(p.walk_len + threadIdx.x), p.wcap);
    __syncthreads();
    for (int i = threadIdx.x; i < p.nst * p.wcap; i += kThreads) {
        const int st = i / p.wcap, e = i - st * p.wcap, len = s_len[st];
        if (e >= len) continue;
        const int32_t *cols = s_cols + st * p.wcap;
        const int mine = cols[e], slab = mine >> 16;
        int at = 0, before = 0, after = 0;
#pragma unroll 4
        for (int o = 0; o < len; ++o) {
            const int s = cols[o] >> 16;
            at += s < slab;
            before += s == slab && o < e;
            after += s == slab && o > e;
        }
        s_walk[st * p.wcap + at + before] = make_int2(e | (before == 0 ? 1 << 30 : 0) | (after == 0 ? (int)(1u << 31) : 0), mine);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    if (p.early && warp != 0) wait_for_prerequisites();      // the activation, the bias and the results' place

    if (warp == 0) {
        // ------------------------------------------------ weight tiles
        if (lane == 0) {
            const int entry_rows = (int)(p.entry_bytes >> 8);
            uint32_t stage = 0, ph = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < p.num_tiles && ok && !*abort_flag; t += gridDim.x) {
                const int st = t % p.nst, len = s_len[st];
                for (int i = 0; i < len; i += kGroup) {
                    if (!mbar_wait_early(w_empty + 8 * stage, ph ^ 1u, abort_flag, p.wait_limit)) { ok = false; break; }
                    const int n = min(kGroup, len - i);
                    mbar_expect_tx(w_full + 8 * stage, (uint32_t)n * p.entry_bytes);
                    for (int g = 0; g < n; ++g)
                        tma_load_2d(w_ring + (stage * kGroup + g) * p.entry_bytes, &map_a, 0,
                                    (st * p.wcap + (s_walk[st * p.wcap + i + g].x & 0xFFFFFF)) * entry_rows, w_full + 8 * stage);
                    if (++stage == p.w_stages) { stage = 0; ph ^= 1u; }
                }
                if (p.resident) break;                       // (the only walk there is: its tiles stay)
            }
        }
        wait_for_prerequisites();                            // (there may have been nothing to wait for)
    } else if (warp == 2 + kEpiWarps) {
        // ------------------------------------------------ activations: a box with its border per slab
        if (lane == 0) {
            uint32_t stage = 0, ph = 0;
            int fill = 0;
            bool ok = true;
            for (int t = blockIdx.x; t < p.num_tiles && ok && !*abort_flag; t += gridDim.x) {
                const int ct = t / p.nst, st = t - ct * p.nst, len = s_len[st];
                const Tile org = tile_at(p, ct);
                for (int i = 0; i < len; ++i) {
                    const int2 w = s_walk[st * p.wcap + i];
                    if (!(w.x >> 30 & 1)) continue;
                    if (!mbar_wait(x_empty + 8 * stage, ph ^ 1u, abort_flag, p.wait_limit)) { ok = false; break; }
                    mbar_expect_tx(x_full + 8 * stage, p.x_bytes);
                    if (fill++ != p.skip_fill)
                        tma_load_4d(base + stage * p.x_stage, &map_x, (w.y >> 16) * 64, org.x - p.pad, org.b, org.y - p.pad, x_full + 8 * stage);
                    if (++stage == p.x_stages) { stage = 0; ph ^= 1u; }
                }
            }
        }
        __syncwarp();
        launch_dependents();                                 // (this CTA has asked for its last tile)
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (lane == 0) {
            constexpr uint32_t idesc = make_idesc(kN, kSparse) & ~(1u << 16);          // X K-major: a pixel's channels are consecutive
            constexpr uint32_t b_step = kSparse ? 4u : 2u;                             // 32 or 16 channels
            constexpr int kMmas = kSparse ? 2 : 4;
            const uint64_t a_desc0 = make_smem_desc(w_ring, 2048, 128, kLayoutNone);
            const uint64_t m_desc0 = make_smem_desc(w_ring + p.a_bytes, 128, 128, kLayoutNone);
            const uint64_t b_desc0 = make_smem_desc(base, 16, (uint32_t)p.pw * 128u, kLayoutSw128);
            const uint32_t w_step = p.entry_bytes >> 4, x_step = p.x_stage >> 4, meta_base = tmem_base + kAcc * kN;
            uint32_t xs = 0, xph = 0, ws = 0, wph = 0, acc = 0, acc_ph = 0;
            bool ok = true;
            // One walk entry whose weight tile lies in slot `at` of the ring.
            auto entry = [&](const int2 &w, uint32_t at, uint32_t d_tmem, uint32_t accum, bool metadata) -> bool {
                if ((w.x >> 30 & 1) && !mbar_wait(x_full + 8 * xs, xph, abort_flag, p.wait_limit)) return false;
                tc_fence_after();
                const uint64_t ad = a_desc0 + at * w_step, bd = b_desc0 + (xs * x_step + (uint32_t)(w.y & 0xFFFF));
                if constexpr (kSparse) {
                    const uint32_t meta = meta_base + 4 * at;
                    if (metadata) tmem_copy_128x128b(meta, m_desc0 + at * w_step);
#pragma unroll
                    for (int j = 0; j < kMmas; ++j)
                        mma_sparse(d_tmem, ad + j * 256, bd + j * b_step, idesc | (uint32_t)(j & 1), accum | (uint32_t)j, meta + (j & ~1));
                } else {
#pragma unroll
                    for (int j = 0; j < kMmas; ++j) mma_dense(d_tmem, ad + j * 256, bd + j * b_step, idesc, accum | (uint32_t)j);
                }
                if (w.x < 0) {                               // the slab's last tap
                    mma_commit(x_empty + 8 * xs);
                    if (++xs == p.x_stages) { xs = 0; xph ^= 1u; }
                }
                return true;
            };
            if (p.resident) {
                // The only walk there is: its tiles are in the ring for good, and their metadata in tensor memory.
                const int len = s_len[0];
                for (int i = 0; i < len && ok; i += kGroup) ok = mbar_wait(w_full + 8 * (i / kGroup), 0, abort_flag, p.wait_limit);
                tc_fence_after();
                if (kSparse && ok)
                    for (int i = 0; i < len; ++i) tmem_copy_128x128b(meta_base + 4 * i, m_desc0 + i * w_step);
                for (int t = blockIdx.x; t < p.num_tiles && ok && !*abort_flag; t += gridDim.x) {
                    if (!mbar_wait(t_empty + 8 * acc, acc_ph ^ 1u, abort_flag, p.wait_limit)) break;
                    tc_fence_after();
                    const uint32_t d_tmem = tmem_base + acc * kN;
                    for (int i = 0; i < len && ok; i += 4) {
                        int2 w[4];
#pragma unroll
                        for (int g = 0; g < 4; ++g) w[g] = s_walk[min(i + g, len - 1)];
#pragma unroll
                        for (int g = 0; g < 4; ++g)
                            if (i + g < len && ok) ok = entry(w[g], (uint32_t)(i + g), d_tmem, (uint32_t)(i + g), false);
                    }
                    if (!ok) break;
                    mma_commit(t_full + 8 * acc);
                    if (++acc == kAcc) { acc = 0; acc_ph ^= 1u; }
                }
            } else {
                for (int t = blockIdx.x; t < p.num_tiles && ok && !*abort_flag; t += gridDim.x) {
                    const int st = t % p.nst, len = s_len[st];
                    const int2 *walk = s_walk + st * p.wcap;
                    if (!mbar_wait(t_empty + 8 * acc, acc_ph ^ 1u, abort_flag, p.wait_limit)) break;
                    tc_fence_after();
                    const uint32_t d_tmem = tmem_base + acc * kN;
                    for (int i = 0; i < len && ok; i += 2 * kGroup) {
                        int2 w[2 * kGroup];
#pragma unroll
                        for (int g = 0; g < 2 * kGroup; ++g) w[g] = walk[min(i + g, len - 1)];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {        // two stages of weights
                            if (i + h * kGroup >= len || !ok) break;
                            if (!mbar_wait(w_full + 8 * ws, wph, abort_flag, p.wait_limit)) { ok = false; break; }
#pragma unroll
                            for (int g = 0; g < kGroup; ++g)
                                if (i + h * kGroup + g < len && ok)
                                    ok = entry(w[h * kGroup + g], ws * kGroup + g, d_tmem, (uint32_t)(i + h * kGroup + g), true);
                            mma_commit(w_empty + 8 * ws);
                            if (++ws == p.w_stages) { ws = 0; wph ^= 1u; }
                        }
                    }
                    if (!ok) break;
                    mma_commit(t_full + 8 * acc);
                    if (++acc == kAcc) { acc = 0; acc_ph ^= 1u; }
                }
            }
        }
    } else {
        // ------------------------------------------------ epilogue: every fourth chunk of 32 pixels for 32 channels
        constexpr int kParts = kEpiWarps / 4;
        const int q = warp & 3, part = (warp - 2) >> 2;
        const uint32_t tile = staging + (uint32_t)(warp - 2) * kStgTile;
        // lane l writes pixel l % 8 of a group, channels 8 (l / 8) ..: 16-byte chunk c of pixel row r lies at c ^ (r / 2 % 4)
        const uint32_t my_row = (uint32_t)((lane & 7) * 64 + (((lane >> 3) ^ ((lane >> 1) & 3)) << 4));
        uint32_t acc = 0, acc_ph = 0;
        const float floor_v = p.relu ? 0.f : __int_as_float(0x7FFFFFFF);     // max(v, NaN) is v, whatever v is: a NaN stays
        const bool fuse = p.bias != nullptr || p.relu != 0;
        for (int t = blockIdx.x; t < p.num_tiles; t += gridDim.x) {
            const int ct = t / p.nst, st = t - ct * p.nst;
            const Tile org = tile_at(p, ct);
            const int ch0 = st * kTileM + 32 * q;
            float bias[4];                                   // of channels l / 4, + 8, + 16, + 24
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int ch = ch0 + (lane >> 2) + 8 * i;
                bias[i] = p.bias && ch < p.rows ? p.bias[ch] : 0.f;
            }
            int go = 0;
            if (lane == 0) go = !*abort_flag && mbar_wait(t_full + 8 * acc, acc_ph, abort_flag, p.wait_limit);
            go = __shfl_sync(0xFFFFFFFFu, go, 0);
            if (!go) break;
            tc_fence_after();
            // a chunk: channels 0..15 and 16..31 of 32 pixels
            auto load = [&](int c, uint32_t (&lo)[16], uint32_t (&hi)[16]) {
                const uint32_t taddr = tmem_base + acc * kN + 32 * c + ((uint32_t)(32 * q) << 16);
                tmem_ld_16x32(taddr, lo);
                tmem_ld_16x32(taddr + (16u << 16), hi);
            };
            auto store = [&](int c, uint32_t (&lo)[16], uint32_t (&hi)[16]) {
                if (fuse) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        lo[i] = __float_as_uint(fmaxf(__uint_as_float(lo[i]) + bias[i >> 1 & 1], floor_v));
                        hi[i] = __float_as_uint(fmaxf(__uint_as_float(hi[i]) + bias[2 + (i >> 1 & 1)], floor_v));
                    }
                }
                if (lane == 0) bulk_wait_read<0>();      // the store that last used the staging tile has read it
                __syncwarp();
#pragma unroll
                for (int g = 0; g < 4; ++g) {            // groups of 8 pixels
                    auto pack = [](uint32_t a, uint32_t b) { return pack_bf16(__uint_as_float(a), __uint_as_float(b)); };
                    store_matrices(tile + (uint32_t)(512 * g) + my_row, pack(lo[4 * g], lo[4 * g + 1]), pack(lo[4 * g + 2], lo[4 * g + 3]),
                                   pack(hi[4 * g], hi[4 * g + 1]), pack(hi[4 * g + 2], hi[4 * g + 3]));
                }
                if (kPlain && ch0 >= p.plain_from) {     // pixel by pixel, the lanes on consecutive channels
                    __syncwarp();
                    const bool ch_ok = ch0 + lane < p.rows;
#pragma unroll 8
                    for (int px = 0; px < 32; ++px) {
                        const int g = 4 * c + (px >> 3), y = org.y + (g >> p.tb_log2), b = org.b + (g & (p.tb - 1)), x = org.x + (px & 7);
                        uint16_t v;
                        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(tile + (uint32_t)(64 * px + (((lane >> 3) ^ (px >> 1 & 3)) << 4) + 2 * (lane & 7))) : "memory");
                        if (ch_ok && y < p.ho && b < p.batch && x < p.wo) p.y[(((int64_t)b * p.ho + y) * p.wo + x) * p.ldy + ch0 + lane] = v;
                    }
                } else {
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) {
                        const int y = org.y + (4 * c >> p.tb_log2);
                        if (y < p.ho) tma_store_4d(&map_y, tile, ch0, org.x, org.b, y);
                        bulk_commit();
                    }
                }
            };
            if constexpr (kAcc == 1) {
                // One accumulator: the warp takes all of its share before the next tile's MMAs may begin, and stores it under them (three
                // convolutions of 56 x 56, 256 pixels a tile: 61.7 -> 58.5 us).
                constexpr int kMine = kChunks / kParts;
                uint32_t lo[kMine][16], hi[kMine][16];
                if (ch0 < p.rows) {
#pragma unroll
                    for (int i = 0; i < kMine; ++i) load(part + kParts * i, lo[i], hi[i]);
                    tmem_ld_wait();
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(t_empty);
                if (ch0 < p.rows) {
#pragma unroll
                    for (int i = 0; i < kMine; ++i) store(part + kParts * i, lo[i], hi[i]);
                }
                acc_ph ^= 1u;
                continue;
            }
            if (ch0 < p.rows) {
                for (int c = part; c < kChunks; c += kParts) {
                    uint32_t lo[16], hi[16];
                    load(c, lo, hi);
                    tmem_ld_wait();
                    store(c, lo, hi);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(t_empty + 8 * acc);
            if (++acc == kAcc) { acc = 0; acc_ph ^= 1u; }
        }
        if (lane == 0) bulk_wait_read<0>();
    }
    // ------------------------------------------------ teardown (every wait above is bounded)
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        if (threadIdx.x == 0) atomicCAS(p.status, 0, (int)CRISP_TIMEOUT);
        const unsigned long long t0 = clock64();             // let copies that may still be in flight land
        while ((unsigned long long)(clock64() - t0) < 2000000ull) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, 512);
    }
}

typedef void (*HaloKernel)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const HaloParams);

}  // namespace

// What a launch takes.
struct HaloLaunch {
    CUtensorMap mx, my, ma;
    HaloParams p;
    HaloKernel kern;
    int which, grid;
    size_t smem;
    crisp_launch_info_t info;
    int64_t resident_bytes;
};
// Launch plan: tensor maps and tile shape for one set of operands; or that convolutions of this shape stay with the other kernel,
// so that this is not worked out at every call.
struct HaloPlan {
    const void *x, *y;
    int64_t ldy;
    ConvGeom conv;
    int device;
    bool plain;                          // results pixel by pixel (plain_from), which the choice of a tile depends on
    bool refused;
    HaloLaunch launch;
};
void halo_plan_destroy(HaloPlan *plan) { delete plan; }

namespace {

bool make_map_nhwc(CUtensorMap *map, const void *base, uint64_t c, uint64_t pitch, uint64_t w, uint64_t h, uint64_t b, uint32_t box_c,
                   uint32_t box_w, uint32_t box_b, uint32_t box_h) {
    // [channel, x, image, y]: images of a tile are interleaved by rows
    const uint64_t dims[4] = {c, w, b, h}, strides[3] = {pitch * 2, h * w * pitch * 2, w * pitch * 2};
    const uint32_t box[4] = {box_c, box_w, box_b, box_h};
    return make_map_4d(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box);
}

enum class Choice { kTaken, kRefused, kNoMaps };

// From which channel on results are stored pixel by pixel (see HaloParams).
int plain_channels(int rows, const void *d_y, int64_t ldy) {
    return ldy % 8 != 0 || reinterpret_cast<uintptr_t>(d_y) % 16 != 0 ? 0 : rows % 8 != 0 ? rows / 32 * 32 : rows;
}

// Whether convolutions of this shape go through the kernel above, and the plan of this one if so.
Choice plan_halo(const crisp_handle_s *h, const uint16_t *d_x, void *d_y, int64_t ldy, const ConvGeom &cv, int device,
               HaloLaunch *plan) {
    const Geometry &g = h->g;
    if (h->exec_kind != CRISP_PATH_SPARSE && h->exec_kind != CRISP_PATH_DENSE) return Choice::kRefused;
    const bool sparse = h->exec_kind == CRISP_PATH_SPARSE;
    const TcImageLayout L = tc_image_layout(g, h->exec_kind);
    const int sms = sm_count_of(device);
    HaloParams p = {};
    p.plain_from = plain_channels(g.rows, d_y, ldy);
    const bool plain = p.plain_from < g.rows;
    // Cycles of a launch in its longest CTA, by what was measured.  An entry of the walk takes as long as shared memory needs to feed its
    // MMAs and take in its weight tile, at least the 330 that issuing it takes; a box of the activation a cycle for each pixel of 128
    // bytes; a tile 300 more, and where its accumulator has to be drained before the next one begins 800, or 1800 with results that are stored pixel by
    // pixel, which takes longer than the next tile's MMAs; the gather in spmm_tc.cu 700 for an entry of 256 pixels, 500 for one of 128.
    // Both sides of the lines it draws (us, 3x3, replayed from a graph): 56 x 56 x 16 images, 256 -> 256 channels, 19 entries: 224 pixels in 4
    // waves of tiles 25.9, 256 in 3 waves 24.1, the gather in 3 waves 26.7; 3:4 dense tiles 30.4, 28.0, 29.7; 56 x 56 x 4, 384 -> 384,
    // 11 entries: 224 in 2 waves 12.1, 256 in one 9.2, gather 9.9; 14 x 14 x 32, 256 -> 256: 128 pixels 8.8, gather 10.2; 7 x 7 x 8, 512 -> 512:
    // 64 pixels 15.0, gather 17.1; 1x1, 64 -> 64, 112 x 112 x 16: 11.8 and 14.1; 512 -> 512, 7 x 7 x 3: 6.4 and 6.3.  (The 800: 224 and 256 pixels, 128 -> 128, 224 x 224 x 3
    // 30.5 and 26.8, x 4 38.1 and 34.9, which 1800 left with 224; 256 -> 112, 1x1, 224 x 224 x 2 10.2 and 11.7, 64 -> 509, 1x1 50.3 and 56.1, which 300 would take to 256.  The 1800: 224 and 256 pixels, 224 x 224, all channels
    // pixel by pixel, 128 -> 477 53.3 and 58.1, 256 -> 408 52.8 and 58.2, 256 -> 171, 1x1 29.5 and 28.8; the last ones only, 128 -> 477 53.6 and 57.4, 64 -> 243 29.0 and 27.9; 0.97 of
    // the time with 224 in the mean of 50 random shapes that the 800 would take to 256, 0.88 to 1.15.)
    const int cpt = cv.channels / g.bk, boxes = L.wcap < cpt ? L.wcap : cpt;
    auto waves = [&](int64_t tiles) { return (tiles * L.nst + sms - 1) / sms; };
    int n = 0;
    int64_t best = 0, tiles = 0;
    for (int cand : {224, 256, 128, 64})
        for (int tb = 1; tb <= 4; tb <<= 1) {
            const int th = cand / 8 / tb, pw = 8 + cv.kw - 1, ph = th + cv.kh - 1;
            if (pw > 256 || ph > 256 || (int64_t)pw * ph * tb * 128 > 56 * 1024 || (ph * tb * pw) * 8 > 0xFFFF) continue;
            const int64_t count = (int64_t)((cv.wo + 7) / 8) * ((cv.ho + th - 1) / th) * ((cv.batch + tb - 1) / tb);
            const int fill = cand + (sparse ? 144 : 256), entry = fill > 330 ? fill : 330;
            const int64_t cost = waves(count) * (L.wcap * entry + boxes * pw * ph * tb + (cand == 256 && sparse ? plain ? 1800 : 800 : 300)) + 2500;
            if (n && cost >= best) continue;
            best = cost; n = cand; tiles = count * L.nst;
            p.th = th; p.tb = tb; p.pw = pw;
        }
    if (!n) return Choice::kRefused;
    int bw, bh, bb;
    const int64_t gather = conv_box(256, 64, cv, &bw, &bh, &bb) / 256;
    const bool narrow = 2 * gather * L.nst < sms;            // (the gather's tiles are half as wide then)
    if (best >= (narrow ? waves(2 * gather) * (L.wcap * 500 + 500) : waves(gather) * (L.wcap * 700 + (sparse ? 2000 : 500))) + 2500) return Choice::kRefused;
    // Where an entry's cost decides, the estimates above are too low: with every SM at work an entry of 128, 224 and 256 pixels takes some
    // 410, 560 and 520 cycles (dense tiles what was estimated), and what a tile costs besides is 1500 less than in the gather.  (us, gather
    // and this kernel, 2 waves of tiles there and 3 here: 512 -> 448 channels, 55 x 57 x 5, 72 entries 51.2 and 59.7; 256 -> 256, 112 x 112 x 3, 24 entries 21.0
    // and 23.4; one and two: 128 -> 128, 28 x 28 x 40, 18 entries 11.4 and 13.4.  On the other side: 4 and 5 waves, 256 -> 256, 12 entries and more 1.08
    // times faster here in the median, 3 and 4 waves of dense tiles, 256 -> 448, 28 x 28 x 30, 36 entries 51.2 and 48.5; as many waves on both sides 1.2
    // times.)  Walks of up to four blocks in one wave of 128-pixel tiles gain nothing that the set-up does not cost, where the gather's tiles are as
    // narrow: 64 -> 448, 1x1, 28 x 28 x 4 5.0 and 5.4; 128 -> 320, 28 x 28 x 6, 256-pixel tiles there, 6.4 and 5.6.
    // (Channels that are no multiple of 8 leave the gather element by element, 1.2 to 1.6 times slower on all of these.)
    if (g.rows % 8 == 0 && narrow) {
        const int64_t pixels = (int64_t)cv.batch * cv.ho * cv.wo;
        if (n == 128 && L.wcap <= 4 && L.nst * ((pixels + 191) / 192) < sms / 2) return Choice::kRefused;
    } else if (g.rows % 8 == 0) {
        const int entry = n <= 128 ? 410 : !sparse ? n + 256 : n == 224 ? 560 : 520;
        if ((tiles + sms - 1) / sms * (L.wcap * entry + 1000) > waves(gather) * (L.wcap * 700 + 2500)) return Choice::kRefused;
    }
    // One CTA tile of rows and a walk of up to eight blocks: from three tiles a CTA on.  (us, gather and this kernel, 64 -> 64 channels: 9 images
    // of 112 x 112 10.5 and 8.8, 3.4 tiles a CTA; 6 images 9.2 and 8.5; 3 images 6.8 each; one image of 56 x 56 5.5 and 5.9.  Below the line stays the gather with
    // resident weight tiles, whose form its tests and crisp_last_resident_bytes' callers look for.)
    if (L.nst == 1 && L.wcap <= 8 && tiles < 3 * (int64_t)sms) return Choice::kRefused;
    if (tiles > 0x7FFFFFFF) return Choice::kRefused;
    if ((int64_t)L.nst * L.wcap * 8 > kListBytes || L.nst > kMaxRowTiles) return Choice::kRefused;
    p.tb_log2 = p.tb == 4 ? 2 : p.tb - 1;
    p.tiles_x = (cv.wo + 7) / 8; p.tiles_y = (cv.ho + p.th - 1) / p.th;
    p.num_tiles = (int)tiles;
    p.walk_col = reinterpret_cast<const int32_t *>(h->d_exec + L.walk_col_off);
    p.walk_len = reinterpret_cast<const int32_t *>(h->d_exec + L.walk_len_off);
    p.status = h->d_status; p.rows = g.rows;
    p.nst = L.nst; p.wcap = L.wcap;
    p.cpt = cv.channels / g.bk; p.kw = cv.kw; p.pad = cv.pad;
    p.wo = cv.wo; p.ho = cv.ho; p.batch = cv.batch;
    p.a_bytes = L.a_bytes; p.entry_bytes = L.entry_bytes;
    const int ph = p.th + cv.kh - 1;
    p.x_bytes = (uint32_t)(p.pw * ph * p.tb * 128);
    p.x_stage = (uint32_t)align_up(p.x_bytes, 1024);
    // up to three boxes in flight beside the one in use where the weight tiles leave the room
    const uint32_t fixed = kEpiWarps * kStgTile + 512 + kListBytes, budget = kSmemBudget + 1024, w_stage = kGroup * p.entry_bytes;
    const uint32_t want_w = 3 * w_stage;
    p.x_stages = fixed + want_w + 2 * p.x_stage > budget ? 2u : (budget - fixed - want_w) / p.x_stage;
    if (p.x_stages > 4) p.x_stages = 4;
    p.w_stages = (budget - fixed - p.x_stages * p.x_stage) / w_stage;
    if (p.w_stages > kMaxStages) p.w_stages = kMaxStages;
    if (p.w_stages < 2) return Choice::kRefused;
    p.resident = L.nst == 1 && (uint32_t)L.wcap <= p.w_stages * kGroup;
    p.y = reinterpret_cast<uint16_t *>(d_y); p.ldy = ldy;
    plan->smem = fixed + (size_t)p.x_stages * p.x_stage + (size_t)p.w_stages * w_stage;
    plan->grid = (int)(tiles < sms ? tiles : sms);
    if (!make_map_image(&plan->ma, h->d_exec + L.image_off, (uint64_t)L.stack * L.nst * L.wcap * L.entry_bytes, L.entry_bytes) ||
        !make_map_nhwc(&plan->mx, d_x, cv.channels, cv.channels, cv.width, cv.height, cv.batch, 64, p.pw, p.tb, ph) ||
        (p.plain_from > 0 && !make_map_nhwc(&plan->my, d_y, g.rows, ldy, cv.wo, cv.ho, cv.batch, 32, 8, p.tb, 4 / p.tb)))
        return Choice::kNoMaps;
    plan->p = p;
    plan->which = (n == 256 ? 12 : n == 224 ? 8 : n == 128 ? 4 : 0) + (sparse ? 2 : 0) + (plain ? 1 : 0);
#define CRISP_HALO_KERNELS(N) spmm_halo_kernel<N, false, false>, spmm_halo_kernel<N, false, true>, spmm_halo_kernel<N, true, false>, spmm_halo_kernel<N, true, true>
    static const HaloKernel kernels[16] = {CRISP_HALO_KERNELS(64), CRISP_HALO_KERNELS(128), CRISP_HALO_KERNELS(224), CRISP_HALO_KERNELS(256)};
#undef CRISP_HALO_KERNELS
    plan->kern = kernels[plan->which];
    plan->resident_bytes = p.resident ? (int64_t)L.wcap * p.entry_bytes : 0;
    plan->info = crisp_launch_info_t{h->exec_kind, n, n == 256 && sparse ? 1 : 2, 1, kEpiWarps, (int)p.x_stages, plan->grid, 1, 1};
    return Choice::kTaken;
}

}  // namespace

// A convolution through the kernel above if it is one of those (*done), with a plan that is kept while the operands and the
// shape are those of the previous call.
cudaError_t launch_spmm_halo(crisp_handle_s *h, const uint16_t *d_x, void *d_y, int64_t ldy, int y_dtype, const ConvGeom &cv, int device,
                             cudaStream_t st, bool *done) {
    *done = false;
    if (y_dtype != 0 || !cv.nhwc_out || h->nt_override > 0 || h->group_override > 0) return cudaSuccess;
    const uint64_t moment = encodes.now();
    HaloLaunch launch;
    {
        std::lock_guard<std::mutex> hold(h->plan_lock);
        HaloPlan *plan = h->halo;
        const bool plain = plain_channels(h->g.rows, d_y, ldy) < h->g.rows;
        const bool same = plan && plan->device == device && plan->plain == plain && same_conv(plan->conv, cv);
        if (same && plan->refused) return cudaSuccess;
        if (!same || plan->x != d_x || plan->y != d_y || plan->ldy != ldy) {
            const cudaError_t e = ensure_context(device);    // (a plan encodes tensor maps)
            if (e != cudaSuccess) return e;
            HaloPlan fresh = {};
            const Choice choice = plan_halo(h, d_x, d_y, ldy, cv, device, &fresh.launch);
            if (choice == Choice::kNoMaps) return cudaSuccess;
            fresh.x = d_x; fresh.y = d_y; fresh.ldy = ldy; fresh.conv = cv; fresh.device = device; fresh.plain = plain;
            fresh.refused = choice == Choice::kRefused;
            if (!plan) {
                plan = new (std::nothrow) HaloPlan;
                if (!plan) return cudaErrorMemoryAllocation;
                h->halo = plan;
            }
            *plan = fresh;
            if (fresh.refused) return cudaSuccess;
        }
        launch = plan->launch;
        launch.p.early = h->settled.holds(st, moment);
    }
    *done = true;
    static std::atomic<bool> configured[16][64];
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    if (!configured[launch.which][device].load(std::memory_order_relaxed)) {
        // the most there is, once: the limit belongs to the function, not to a call
        const cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(launch.kern), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)kSmemBudget + 1024);
        if (e != cudaSuccess) return e;
        configured[launch.which][device].store(true, std::memory_order_relaxed);
    }
    HaloParams &p = launch.p;
    p.bias = h->epilogue.bias; p.relu = h->epilogue.relu;
    p.wait_limit = h->wait_limit_cycles ? h->wait_limit_cycles : kWaitLimitCycles;
    p.skip_fill = h->debug_skip_stage;
    const cudaError_t e = launch_product(encodes, p, moment, [&] {
        return launch_chained(launch.kern, (unsigned)launch.grid, (unsigned)kThreads, launch.smem, st, launch.mx, launch.my, launch.ma, p);
    });
    if (e == cudaSuccess) note_launch(h, launch.info, launch.resident_bytes, st, moment);
    return e;
}

}  // namespace crisp
