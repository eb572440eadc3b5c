// Direct SpMM on the canonical format (CUDA cores).  It follows the three steps of Sec. III-E
// literally: stage the activation rows of kept blocks (step 1), pick for each stored weight the
// activation its offset names (step 2), multiply-accumulate in fp32 (step 3).  It accepts every
// shape and alignment and serves the layouts TMA cannot address (row pitches that are not multiples of 16 bytes) where
// spmm_gather.cu does not: small products, fp32 results, and calls that ask for this path.
//
// Large products are bound by instruction issue: a stored weight costs a warp one look-up of its activation row
// and the multiply-adds of the columns its lanes own, so everything else is taken out of that loop.  A weight and the
// shared-memory offset of its activation row are decoded once per (row, value) by the lanes of the warp that owns the
// row and kept as one 32-bit word {row offset : weight}; the loop reads four of these words with one broadcast load.
// Small ones are bound by latency: all memory traffic is asynchronous copies several stages ahead, and a row of X is
// copied as the aligned 16-byte words that hold it, whatever its alignment (the distance to the first wanted element
// is part of the weight's row offset), so that nothing passes through registers.
// Sums run over blocks, groups and values in ascending order, one fused multiply-add each: results do not
// depend on the tile chosen.
// Measured (the kernel before staged scalar 2-byte loads and decoded an offset at every use): 256 x 2304 x 6076, 1:4,
// keep 0.25: 508 -> 51 us (38 M warp instructions, 76 % of the issue slots of busy SMs); 160 x 960 x 49, 2:8, keep 0.5:
// 147 -> 16.4 us, a chain of four stages on 20 CTAs.  One warp per row that gathers its activations from L2 without
// staging took 13-22 us on the second and 65 us on the first; staging through registers with two buffers 70 us.
// The next kernel's launch overlaps the end of this one: products in a row, us, without and with it, 216 x 106 x 245 6.2 and 4.0, 64 x 64 x 6076 fp32
// 14.4 and 11.4, 3554 x 199 x 3332 fp32 178 and 175.
#include <cuda_bf16.h>

#include "crisp_internal.h"

namespace crisp {

namespace {

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 16 bytes (`bytes` of them from global memory, the rest zero) / 4 bytes into shared memory, asynchronously
__device__ __forceinline__ void copy16(uint32_t dst, uintptr_t src, uint32_t bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void copy4(uint32_t dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void commit_copies() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void wait_copies() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ uint4 lds128(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds16(uint32_t a) {
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
    return v;
}
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

// How kept blocks are cut into parts of 32 or 64 activation rows, and the divisions of the kernel as multiplications:
// div_small(i, small_inverse(d)) = i / d for the values here (parts of a row tile over 1..3, values of a row over 1..8).
struct DirectSplit {
    int part_log2, ppb, vpp;                     // log2(activation rows of a part), parts per block, weights per row and part
    uint32_t inv_ppb, inv_vpp, inv_n;
};
constexpr uint32_t small_inverse(uint32_t d) { return ((1u << 21) + d - 1) / d; }
__device__ __forceinline__ int div_small(int i, uint32_t inv) { return (int)(((uint64_t)(uint32_t)i * inv) >> 21); }

// Tile of one CTA: kWarps * RW rows of one row tile x 32 * CPL columns; warp w owns RW rows.  A stage holds kStageRows
// activation rows (one or more parts); kStages of them are in flight.
template <int RW, int CPL>
struct DirectTile {
    static constexpr int kWarps = 8, kThreads = 32 * kWarps;
    static constexpr int kTileN = 32 * CPL, kRows = kWarps * RW;
    static constexpr int kStageRows = CPL == 4 ? 64 : 128;
    static constexpr int kStages = CPL == 4 ? 3 : 4;
    static constexpr int kPitch = kTileN * 2 + 16;           // a row of X: the aligned 16-byte words that hold kTileN elements
    // Dynamic shared memory at most: a stage holds kStageRows rows of X and, for each of the kRows rows, up to kStageRows weights
    // of 2 bytes with offsets of 3 bits (n = m = 8); the weight words and the block list come after the stages.
    static constexpr int kMostSmem = kStages * kStageRows * (kPitch + kRows * 2 + kRows * 3 / 8) + kRows * kStageRows * 4 + 4 * kMaxBlocksPerRowTile;
    static_assert(kMostSmem <= 227 * 1024, "shared memory of a CTA");
};

// ALIGN: bytes every row of X is aligned to (2, 4 or 8), which fixes the columns a lane owns: consecutive ones as far as
// one shared-memory load can bring them.
template <int RW, int CPL, int ALIGN, typename OutT>
__global__ void __launch_bounds__(DirectTile<RW, CPL>::kThreads, 3)
spmm_direct_kernel(Geometry g, const int32_t *blk_col, const uint16_t *vals, const uint32_t *idx, const uint16_t *x, int64_t ldx,
                   int64_t ncols, OutT *y, int64_t ldy, Epilogue epi, DirectSplit sp) {
    using T = DirectTile<RW, CPL>;
    constexpr int kThreads = T::kThreads, kTileN = T::kTileN, kRows = T::kRows, kStageRows = T::kStageRows, kPitch = T::kPitch;
    constexpr int kRun = ALIGN / 2 < CPL ? ALIGN / 2 : CPL;  // consecutive columns of a lane
    extern __shared__ __align__(16) uint8_t s_raw[];
    const int group = kStageRows >> sp.part_log2;            // parts per stage
    const int vpp = sp.vpp, vpr = vpp * sp.ppb;              // stored weights per row and part, per row and block (4 divides both)
    // a stage: [kStageRows][kPitch] X | [group][kRows * vpp] weights | [group][kRows * vpp * idx_bits / 8] offsets
    const int val_bytes = kRows * vpp * 2, idx_bytes = kRows * vpp * g.idx_bits / 8;
    const int stage_bytes = kStageRows * kPitch + group * (val_bytes + idx_bytes);
    const uint32_t s_x = smem_addr(s_raw);
    const uint32_t s_words = s_x + T::kStages * stage_bytes;                                 // [kRows][group * vpp] weight words
    const int32_t *s_col = reinterpret_cast<const int32_t *>(s_raw + T::kStages * stage_bytes + kRows * group * vpp * 4);   // [kkeep]

    wait_for_prerequisites();                                // (behind it nothing is read through the read-only path)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int slabs = g.bm / kRows;                          // CTAs that share a row tile
    const int64_t ct = blockIdx.x / (g.nrt * slabs);         // row slabs fastest: they share X
    const int rs = (int)(blockIdx.x - ct * (g.nrt * slabs));
    const int rt = rs / slabs, slab_row = (rs - rt * slabs) * kRows;
    const int64_t c0 = ct * kTileN;
    if ((int64_t)rt * g.bm + slab_row >= g.rows) return;     // only padding rows
    const uintptr_t x_begin = reinterpret_cast<uintptr_t>(x);
    const uintptr_t x_end = reinterpret_cast<uintptr_t>(x + (int64_t)(g.k - 1) * ldx + ncols);
    const int vpb = (int)g.vals_per_block();
    const int idx_words = vpb * g.idx_bits / 32;
    const uint32_t field = (1u << g.idx_bits) - 1u;
    const int parts = g.kkeep * sp.ppb, stages = (parts + group - 1) / group;
    for (int i = threadIdx.x; i < g.kkeep; i += kThreads) const_cast<int32_t *>(s_col)[i] = blk_col[(int64_t)rt * g.kkeep + i];
    __syncthreads();

    // step 1: the activation rows of a stage's parts and the slab's weights and offsets
    auto issue_stage = [&](int st) {
        if (st < stages) {
            const int part0 = st * group, cnt = min(group, parts - part0);
            const uint32_t buf = s_x + (uint32_t)(st % T::kStages) * (uint32_t)stage_bytes;
            constexpr int kWords = kPitch / 16;
            for (int i = threadIdx.x; i < (cnt << sp.part_log2) * kWords; i += kThreads) {
                const int kr = i / kWords, j = i - kr * kWords;
                const int part = part0 + (kr >> sp.part_log2);
                const int slot = div_small(part, sp.inv_ppb);
                const int krow = s_col[slot] * g.bk + ((part - slot * sp.ppb) << sp.part_log2) + (kr & ((1 << sp.part_log2) - 1));
                const uint32_t dst = buf + (uint32_t)(kr * kPitch + 16 * j);
                const uintptr_t p = (reinterpret_cast<uintptr_t>(x + (int64_t)krow * ldx + c0) & ~(uintptr_t)15) + 16 * j;
                if (krow < g.k && p < x_begin) {             // the first word of X starts before it: element by element
#pragma unroll
                    for (int t = 0; t < 8; ++t)
                        reinterpret_cast<uint16_t *>(s_raw)[(dst - s_x) / 2 + t] =
                            p + 2 * t >= x_begin && p + 2 * t < x_end ? reinterpret_cast<const uint16_t *>(p)[t] : (uint16_t)0;
                } else {                                     // zero beyond the matrix (the address is not used then)
                    const uint32_t bytes = krow >= g.k || p >= x_end ? 0u : (p + 16 <= x_end ? 16u : (uint32_t)(x_end - p));
                    copy16(dst, bytes ? p : reinterpret_cast<uintptr_t>(vals), bytes);
                }
            }
            const uint32_t vdst = buf + kStageRows * kPitch, idst = vdst + (uint32_t)(group * val_bytes);
            for (int b = 0; b < cnt; ++b) {
                const int slot = div_small(part0 + b, sp.inv_ppb), sub = part0 + b - slot * sp.ppb;
                const int64_t blk = (int64_t)rt * g.kkeep + slot;
                if (sp.ppb == 1) {                           // the slab's rows are consecutive in memory
                    const uint16_t *vsrc = vals + blk * vpb + slab_row * vpr;
                    for (int i = threadIdx.x; i < val_bytes / 16; i += kThreads)
                        copy16(vdst + b * val_bytes + 16 * i, reinterpret_cast<uintptr_t>(vsrc + 8 * i), 16u);
                } else {                                     // a part of each row: vpp * 2 bytes (a multiple of 8) every vpr * 2
                    const int wpr = vpp / 2;
                    for (int i = threadIdx.x; i < kRows * wpr; i += kThreads) {
                        const int r = i / wpr, c = i - r * wpr;
                        copy4(vdst + b * val_bytes + 4 * i, vals + blk * vpb + (slab_row + r) * vpr + sub * vpp + 2 * c);
                    }
                }
            }
            // offsets stay a bit stream: the whole slab of the block, also where the stage holds a part of it
            if (sp.ppb == 1) {
                for (int b = 0; b < cnt; ++b) {
                    const int64_t blk = (int64_t)rt * g.kkeep + part0 + b;
                    const uint32_t *isrc = idx + blk * idx_words + slab_row * vpr * g.idx_bits / 32;
                    for (int i = threadIdx.x; i < idx_bytes / 4; i += kThreads) copy4(idst + b * idx_bytes + 4 * i, isrc + i);
                }
            }
        }
        commit_copies();
    };
#pragma unroll
    for (int s = 0; s < T::kStages - 1; ++s) issue_stage(s);

    float acc[RW][CPL];
#pragma unroll
    for (int r = 0; r < RW; ++r)
#pragma unroll
        for (int c = 0; c < CPL; ++c) acc[r][c] = 0.f;
    const uint32_t x_low = (uint32_t)x_begin + (uint32_t)c0 * 2u, ldx2 = (uint32_t)ldx * 2u;
    const uint32_t my_words = s_words + (uint32_t)(warp * RW * group * vpp) * 4u;
    for (int st = 0; st < stages; ++st) {
        wait_copies<T::kStages - 2>();
        __syncthreads();                                     // this stage has landed, the previous one has been read
        issue_stage(st + T::kStages - 1);
        const int part0 = st * group, cnt = min(group, parts - part0);
        const uint32_t buf = s_x + (uint32_t)(st % T::kStages) * (uint32_t)stage_bytes;
        const uint32_t vsrc = buf + kStageRows * kPitch, isrc = vsrc + (uint32_t)(group * val_bytes);
        // step 2: the warp's own rows, each stored weight with the place of the activation it multiplies
        for (int b = 0; b < cnt; ++b) {
            const int slot = div_small(part0 + b, sp.inv_ppb), sub = part0 + b - slot * sp.ppb;
            const uint32_t krow0 = (uint32_t)(s_col[slot] * g.bk + (sub << sp.part_log2));
            const uint32_t *ib = idx + ((int64_t)rt * g.kkeep + slot) * idx_words;
            for (int i = lane; i < RW * vpp; i += 32) {
                const int r = div_small(i, sp.inv_vpp), v = i - r * vpp;
                const uint32_t w = lds16(vsrc + b * val_bytes + (uint32_t)(warp * RW * vpp + i) * 2u);
                uint32_t t;
                if (sp.ppb == 1) {
                    const int bit = (warp * RW * vpp + i) * g.idx_bits;
                    const uint32_t a = isrc + b * idx_bytes + (uint32_t)(bit >> 5) * 4u;
                    t = lds32(a) >> (bit & 31);
                    if ((bit & 31) + g.idx_bits > 32) t |= lds32(a + 4) << (32 - (bit & 31));
                } else {
                    const int bit = ((slab_row + warp * RW + r) * vpr + sub * vpp + v) * g.idx_bits;
                    t = ib[bit >> 5] >> (bit & 31);
                    if ((bit & 31) + g.idx_bits > 32) t |= ib[(bit >> 5) + 1] << (32 - (bit & 31));
                }
                const uint32_t kin = (uint32_t)(div_small(v, sp.inv_n) * g.m) + (t & field);       // activation row in the part
                const uint32_t off = ((uint32_t)(b << sp.part_log2) + kin) * (uint32_t)kPitch + ((x_low + (krow0 + kin) * ldx2) & 15u);
                asm volatile("st.shared.u32 [%0], %1;" ::"r"(my_words + (uint32_t)((r * cnt + b) * vpp + v) * 4u), "r"((off << 16) | w) : "memory");
            }
        }
        __syncwarp();
        // step 3
        const uint32_t xl = buf + lane * kRun * 2;
#pragma unroll
        for (int r = 0; r < RW; ++r) {
            const uint32_t wr = my_words + (uint32_t)(r * cnt * vpp) * 4u;
#pragma unroll 2
            for (int v4 = 0; v4 < cnt * vpp; v4 += 4) {
                const uint4 e4 = lds128(wr + (uint32_t)v4 * 4u);
                const uint32_t e[4] = {e4.x, e4.y, e4.z, e4.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float wv = __uint_as_float(e[u] << 16);
                    const uint32_t src = xl + (e[u] >> 16);
                    if constexpr (kRun == 4) {
                        const uint2 p = lds64(src);
                        acc[r][0] = fmaf(wv, __uint_as_float(p.x << 16), acc[r][0]);
                        acc[r][1] = fmaf(wv, __uint_as_float(p.x & 0xFFFF0000u), acc[r][1]);
                        acc[r][2] = fmaf(wv, __uint_as_float(p.y << 16), acc[r][2]);
                        acc[r][3] = fmaf(wv, __uint_as_float(p.y & 0xFFFF0000u), acc[r][3]);
                    } else if constexpr (kRun == 2) {
#pragma unroll
                        for (int c = 0; c < CPL; c += 2) {
                            const uint32_t p = lds32(src + c * 64);
                            acc[r][c] = fmaf(wv, __uint_as_float(p << 16), acc[r][c]);
                            acc[r][c + 1] = fmaf(wv, __uint_as_float(p & 0xFFFF0000u), acc[r][c + 1]);
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < CPL; ++c) acc[r][c] = fmaf(wv, __uint_as_float(lds16(src + c * 64) << 16), acc[r][c]);
                    }
                }
            }
        }
        __syncwarp();                                        // the warp's weight words may be overwritten
    }
    wait_copies<0>();
    // The next kernel may begin now.  Asked for at the start, its CTAs wait beside this one's on some SMs and leave others empty: 47 x 1048 x 196
    // fp32 37.5 us in a row instead of 29.7 (32.5 without overlap), 1783 x 107 x 7 14.9 instead of 12.2 (14.4).
    launch_dependents();

#pragma unroll
    for (int r = 0; r < RW; ++r) {
        const int64_t row = (int64_t)rt * g.bm + slab_row + warp * RW + r;
        if (row >= g.rows) break;
        const float bias = epi.bias ? epi.bias[row] : 0.f;
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
            float v = acc[r][c];
            if (epi.bias) v += bias;
            if (epi.relu) v = fmaxf(v, 0.f);
            acc[r][c] = v;
        }
#pragma unroll
        for (int c = 0; c < CPL; c += kRun) {
            const int64_t col = c0 + lane * kRun + 32 * c;
            OutT *dst = y + row * ldy + col;
            const bool whole = reinterpret_cast<uintptr_t>(dst) % (kRun * sizeof(OutT)) == 0 && col + kRun <= ncols;
            if constexpr (sizeof(OutT) == 2) {
                uint32_t p[kRun];
#pragma unroll
                for (int t = 0; t < kRun; ++t) p[t] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(acc[r][c + t]));
                if (kRun == 4 && whole) *reinterpret_cast<uint2 *>(dst) = make_uint2(p[0] | (p[kRun / 4] << 16), p[kRun / 2] | (p[kRun - 1] << 16));
                else if (kRun == 2 && whole) *reinterpret_cast<uint32_t *>(dst) = p[0] | (p[kRun - 1] << 16);
                else {
#pragma unroll
                    for (int t = 0; t < kRun; ++t)
                        if (col + t < ncols) dst[t] = (OutT)p[t];
                }
            } else {
                if (kRun == 4 && whole) *reinterpret_cast<float4 *>(dst) = make_float4(acc[r][c], acc[r][c + kRun / 4], acc[r][c + kRun / 2], acc[r][c + kRun - 1]);
                else if (kRun == 2 && whole) *reinterpret_cast<float2 *>(dst) = make_float2(acc[r][c], acc[r][c + kRun - 1]);
                else {
#pragma unroll
                    for (int t = 0; t < kRun; ++t)
                        if (col + t < ncols) dst[t] = acc[r][c + t];
                }
            }
        }
    }
}

template <int RW, int CPL, typename OutT>
cudaError_t launch_form(const Geometry &g, const int32_t *bc, const uint16_t *vals, const uint32_t *idx, const uint16_t *x,
                        int64_t ldx, int64_t ncols, OutT *y, int64_t ldy, const Epilogue &epi, cudaStream_t st) {
    using T = DirectTile<RW, CPL>;
    DirectSplit sp;
    sp.part_log2 = g.bk % 64 == 0 ? 6 : 5;
    sp.ppb = g.bk >> sp.part_log2;
    sp.vpp = (1 << sp.part_log2) / g.m * g.n;
    sp.inv_ppb = small_inverse(sp.ppb); sp.inv_vpp = small_inverse(sp.vpp); sp.inv_n = small_inverse(g.n);
    const int group = T::kStageRows >> sp.part_log2;
    const size_t stage = T::kStageRows * T::kPitch + (size_t)group * (T::kRows * sp.vpp * 2 + T::kRows * sp.vpp * g.idx_bits / 8);
    const size_t smem = T::kStages * stage + (size_t)T::kRows * group * sp.vpp * 4 + (size_t)g.kkeep * 4;
    const int64_t ctas = ((ncols + T::kTileN - 1) / T::kTileN) * g.nrt * (g.bm / T::kRows);
    if (ctas > 0x7FFFFFFFll) return cudaErrorInvalidValue;
    const uintptr_t al = reinterpret_cast<uintptr_t>(x) | (uintptr_t)(ldx * 2);
    auto launch = [&](auto kern) {
        // The limit belongs to the function, so it is the same at every call: set to a call's own size, it would refuse the
        // larger launch of another host thread that set it a moment before.
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, T::kMostSmem);
        if (e != cudaSuccess) return e;
        return launch_chained(kern, (unsigned)ctas, T::kThreads, smem, st, g, bc, vals, idx, x, ldx, ncols, y, ldy, epi, sp);
    };
    if (CPL == 4 && al % 8 == 0) return launch(spmm_direct_kernel<RW, CPL, CPL == 4 ? 8 : 4, OutT>);
    if (al % 4 == 0) return launch(spmm_direct_kernel<RW, CPL, 4, OutT>);
    return launch(spmm_direct_kernel<RW, CPL, 2, OutT>);
}

template <typename OutT>
cudaError_t launch_typed(const Geometry &g, const int32_t *bc, const uint16_t *vals, const uint32_t *idx,
                         const uint16_t *x, int64_t ldx, int64_t ncols, OutT *y, int64_t ldy,
                         const Epilogue &epi, cudaStream_t st) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
        sms = 148;
    // Rows per warp and columns per lane: wide tiles re-use a staged activation for more rows and a decoded weight for
    // more columns, small ones give a small product enough CTAs.  The widest form that leaves every SM two CTAs is
    // taken, or the smallest form (1280 x 320 x 392: 14.0 us with 16 x 128 tiles, 19 with 8 x 64 ones at twice the CTAs).
    auto fits = [&](int rows, int64_t per_sm) {
        return g.bm % rows == 0 && ((ncols + 127) / 128) * g.nrt * (g.bm / rows) >= per_sm * sms;
    };
    if (fits(64, 2)) return launch_form<8, 4, OutT>(g, bc, vals, idx, x, ldx, ncols, y, ldy, epi, st);
    if (fits(32, 2)) return launch_form<4, 4, OutT>(g, bc, vals, idx, x, ldx, ncols, y, ldy, epi, st);
    if (fits(16, 2)) return launch_form<2, 4, OutT>(g, bc, vals, idx, x, ldx, ncols, y, ldy, epi, st);
    return launch_form<1, 2, OutT>(g, bc, vals, idx, x, ldx, ncols, y, ldy, epi, st);
}

}  // namespace

cudaError_t launch_spmm_direct(const Geometry &g, const int32_t *d_blk_col, const uint16_t *d_vals,
                               const uint32_t *d_idx, const uint16_t *d_x, int64_t ldx, int64_t ncols,
                               void *d_y, int64_t ldy, int y_dtype, const Epilogue &epi, cudaStream_t st) {
    if (y_dtype == 0)
        return launch_typed<uint16_t>(g, d_blk_col, d_vals, d_idx, d_x, ldx, ncols,
                                      reinterpret_cast<uint16_t *>(d_y), ldy, epi, st);
    return launch_typed<float>(g, d_blk_col, d_vals, d_idx, d_x, ldx, ncols,
                               reinterpret_cast<float *>(d_y), ldy, epi, st);
}

}  // namespace crisp
