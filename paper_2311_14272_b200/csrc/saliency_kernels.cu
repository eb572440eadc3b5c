// Class-aware saliency score (Sec. III-C "Pruning Metric", Eq. 1): T_w = | (1/H) * sum_i g_i (.) W |, the
// first-order Taylor estimate with the gradient averaged over the H samples of the user's classes.
// The gradients come from the caller's training step, one tensor per sample or mini-batch:
//   crisp_saliency_accumulate  acc += g           (fp32 running sum, once per gradient tensor)
//   crisp_saliency_finish      S = |acc / H * W|   (fp32, the input of crisp_build_mask)
// and, for all layers and samples of a network in one launch, saliency_bits_kernel below.
// Both are element-wise streams and HBM-bound: 16-byte accesses where the rows allow it, one grid-stride
// pass with a grid of a whole number of waves.
#include <cuda_bf16.h>

#include <memory>
#include <new>

#include "crisp_internal.h"
#include "mask_common.cuh"

namespace crisp {
namespace {

constexpr int kSalThreads = 256;

__device__ __forceinline__ float bf16_bits_to_float(uint32_t b) { return __uint_as_float(b << 16); }

// rows of k elements with leading dimensions in elements; kVec: every row start and k are multiples of 4
template <bool kBf16, bool kVec>
__global__ void __launch_bounds__(kSalThreads)
saliency_accumulate_kernel(const void *__restrict__ grad, int64_t ld_g, int rows, int k, float *__restrict__ acc,
                           int64_t ld_a, int first) {
    const int kq = kVec ? k / 4 : k;
    const int64_t total = (int64_t)rows * kq;
    for (int64_t i = (int64_t)blockIdx.x * kSalThreads + threadIdx.x; i < total; i += (int64_t)gridDim.x * kSalThreads) {
        const int r = (int)(i / kq), c = (int)(i - (int64_t)r * kq);
        if constexpr (kVec) {
            float4 g;
            if constexpr (kBf16) {
                const uint2 raw = *reinterpret_cast<const uint2 *>(reinterpret_cast<const uint16_t *>(grad) + r * ld_g + 4 * c);
                g = make_float4(bf16_bits_to_float(raw.x & 0xFFFFu), bf16_bits_to_float(raw.x >> 16),
                                bf16_bits_to_float(raw.y & 0xFFFFu), bf16_bits_to_float(raw.y >> 16));
            } else {
                g = *reinterpret_cast<const float4 *>(reinterpret_cast<const float *>(grad) + r * ld_g + 4 * c);
            }
            float4 *dst = reinterpret_cast<float4 *>(acc + r * ld_a + 4 * c);
            if (first) { *dst = g; continue; }
            float4 a = *dst;
            a.x += g.x; a.y += g.y; a.z += g.z; a.w += g.w;
            *dst = a;
        } else {
            const float g = kBf16 ? bf16_bits_to_float(reinterpret_cast<const uint16_t *>(grad)[r * ld_g + c])
                                  : reinterpret_cast<const float *>(grad)[r * ld_g + c];
            float *dst = acc + r * ld_a + c;
            *dst = first ? g : *dst + g;
        }
    }
}

// |s| as the mask projection reads it (NaN -> 0, Inf -> FLT_MAX), as ordered bits
__device__ __forceinline__ uint32_t canonical_key_bits(float v) {
    return __float_as_uint(fminf(fmaxf(v, 0.f), 3.402823466e+38f));
}

// max_key != nullptr: the layer-wide maximum of the canonical score is left there as well (one atomic per warp),
// which is the first thing the mask projection needs: it then does not have to stream S once more to find it.
template <bool kVec>
__global__ void __launch_bounds__(kSalThreads)
saliency_finish_kernel(const float *__restrict__ acc, int64_t ld_a, const uint16_t *__restrict__ w, int64_t ld_w,
                       int rows, int k, float inv_samples, float *__restrict__ s, int64_t ld_s,
                       uint32_t *__restrict__ max_key) {
    const int kq = kVec ? k / 4 : k;
    const int64_t total = (int64_t)rows * kq;
    uint32_t best = 0u;
    for (int64_t i = (int64_t)blockIdx.x * kSalThreads + threadIdx.x; i < total; i += (int64_t)gridDim.x * kSalThreads) {
        const int r = (int)(i / kq), c = (int)(i - (int64_t)r * kq);
        if constexpr (kVec) {
            const float4 a = *reinterpret_cast<const float4 *>(acc + r * ld_a + 4 * c);
            const uint2 raw = *reinterpret_cast<const uint2 *>(w + r * ld_w + 4 * c);
            float4 o;
            o.x = fabsf(a.x * inv_samples * bf16_bits_to_float(raw.x & 0xFFFFu));
            o.y = fabsf(a.y * inv_samples * bf16_bits_to_float(raw.x >> 16));
            o.z = fabsf(a.z * inv_samples * bf16_bits_to_float(raw.y & 0xFFFFu));
            o.w = fabsf(a.w * inv_samples * bf16_bits_to_float(raw.y >> 16));
            *reinterpret_cast<float4 *>(s + r * ld_s + 4 * c) = o;
            best = max(max(best, canonical_key_bits(o.x)), max(canonical_key_bits(o.y), max(canonical_key_bits(o.z), canonical_key_bits(o.w))));
        } else {
            const float v = fabsf(acc[r * ld_a + c] * inv_samples * bf16_bits_to_float(w[r * ld_w + c]));
            s[r * ld_s + c] = v;
            best = max(best, canonical_key_bits(v));
        }
    }
    if (max_key != nullptr) {
        best = __reduce_max_sync(0xFFFFFFFFu, best);
        if ((threadIdx.x & 31) == 0 && best) atomicMax(max_key, best);
    }
}

// The gradients of all samples to the saliency and on to the group bits and the layer maximum, for all layers of a network
// in one launch:
//     S = |(g_0 + g_1 + ...) * (1 / H) * W|  (fp32, each step rounded, the order of the calls above)
// The sum stays in registers: a sample costs its own bytes once (2 or 4 an element), where one launch per sample adds a
// read and a write of the fp32 accumulator to them; the bits and the maximum come from the values the thread already
// holds instead of from another pass over S, and so do the records that the block scores are made of (bits_and_record's, of 32 x 32 elements: the
// CTA's 16 warps agree on a scale through shared memory).  Work items of 32 rows x 256 elements; a lane owns eight consecutive elements of two
// rows, and a warp 512 consecutive bytes of each row (32 x 32 elements a warp: 64 us on the first below, twice the requests).  Bound by HBM; what a small network waits
// for is latency, so items are CTAs of their own, all layers share the launch and a sample is asked for before the last one is added.
// Measured (us, this kernel and the score kernel; 13 layers of VGG-16, 14.7 M weights, four bf16 samples, 206 MB): 52.2 + 3.4, before the
// records 51.1 + 14.8; 35 layers of MobileNetV2 13.0 + 3.2, 15.0 + 5.8.  Four rows a lane 56.5 and 17.1, two CTAs an SM 53.6 and 15.9
// (the 40 registers of three spill 64 to 112 bytes, all forms).
constexpr int kSalChunk = 256, kSalWords = kSalChunk / 32;                     // k-elements of a work item: 32 lanes x 8
constexpr int kSalLaneRows = 2, kSalItemThreads = kM1Rows / kSalLaneRows * 32;
struct SaliencyLayer {
    Geometry g;
    const uint16_t *w;
    float *s;
    int64_t ld_w, ld_s;
    uint32_t *max_key, *nm_bits;
    unsigned long long *records;
    float inv;
    int grad0, samples, chunks, vec_ok;
};
struct GradRef {
    const void *p;
    int64_t ld;                          // in elements; negative: fp32 with pitch -ld
};
constexpr int kBatchGrads = 640;
struct SaliencyBatch {
    Batch<SaliencyLayer, kBatchLayers> b;
    GradRef grad[kBatchGrads];
};
static_assert(sizeof(SaliencyBatch) < 32000, "kernel parameters");

template <int M, int TOP>
__global__ void __launch_bounds__(kSalItemThreads, 3)
saliency_bits_kernel(const __grid_constant__ SaliencyBatch batch) {
    __shared__ uint8_t s_keep[64];
    __shared__ uint32_t s_top[kSalWords], s_low[kSalWords], s_r[kSalWords];        // of the CTA's 32 x 32 elements in a mask word's columns
    __shared__ int s_d[kSalWords];
    chain_kernels();
    const int l = batch.b.find(blockIdx.x);
    const SaliencyLayer &L = batch.b.layer[l];
    const Geometry &g = L.g;
    if (M == 4 && threadIdx.x < 64) s_keep[threadIdx.x] = (uint8_t)keep_mask_of_outcomes(threadIdx.x, g.n);
    if (threadIdx.x < kSalWords) { s_top[threadIdx.x] = 0u; s_low[threadIdx.x] = 0xFFFFFFFFu; s_r[threadIdx.x] = 0u; s_d[threadIdx.x] = 0; }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t item = blockIdx.x - (uint32_t)batch.b.first[l], rg = item / (uint32_t)L.chunks, chunk = item - rg * (uint32_t)L.chunks;
    const int64_t k0 = (int64_t)chunk * kSalChunk + lane * 8;
    const int64_t row0 = (int64_t)rg * kM1Rows + warp * kSalLaneRows;
    float v[kSalLaneRows][8];
    if (L.vec_ok && row0 + kSalLaneRows <= g.rows && k0 + 8 <= g.k) {
        uint4 wr[kSalLaneRows];
#pragma unroll
        for (int i = 0; i < kSalLaneRows; ++i) wr[i] = *reinterpret_cast<const uint4 *>(L.w + (row0 + i) * L.ld_w + k0);
        // (a bf16 sample is asked for before the one in front of it is added)
        uint4 t[kSalLaneRows];
        auto ask = [&](const GradRef &G, uint4 (&to)[kSalLaneRows]) {
#pragma unroll
            for (int i = 0; i < kSalLaneRows; ++i)
                to[i] = *reinterpret_cast<const uint4 *>(reinterpret_cast<const uint16_t *>(G.p) + (row0 + i) * G.ld + k0);
        };
        GradRef G = batch.grad[L.grad0];
        if (G.ld > 0) ask(G, t);
        for (int h = 0; h < L.samples; ++h) {
            uint4 next[kSalLaneRows];
            GradRef N = G;
            if (h + 1 < L.samples) {
                N = batch.grad[L.grad0 + h + 1];
                if (N.ld > 0) ask(N, next);
            }
            if (G.ld > 0) {
#pragma unroll
                for (int i = 0; i < kSalLaneRows; ++i) {
                    const uint32_t q[4] = {t[i].x, t[i].y, t[i].z, t[i].w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float a = __uint_as_float(q[j] << 16), b = __uint_as_float(q[j] & 0xFFFF0000u);
                        v[i][2 * j] = h ? __fadd_rn(v[i][2 * j], a) : a;
                        v[i][2 * j + 1] = h ? __fadd_rn(v[i][2 * j + 1], b) : b;
                    }
                }
            } else {
#pragma unroll
                for (int i = 0; i < kSalLaneRows; ++i) {
                    const float4 *p = reinterpret_cast<const float4 *>(reinterpret_cast<const float *>(G.p) + (row0 + i) * -G.ld + k0);
                    const float4 a = p[0], b = p[1];
                    const float q[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[i][j] = h ? __fadd_rn(v[i][j], q[j]) : q[j];
                }
            }
            G = N;
#pragma unroll
            for (int i = 0; i < kSalLaneRows; ++i) t[i] = next[i];
        }
#pragma unroll
        for (int i = 0; i < kSalLaneRows; ++i) {
            const uint32_t q[4] = {wr[i].x, wr[i].y, wr[i].z, wr[i].w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                v[i][2 * j] = fabsf(__fmul_rn(__fmul_rn(v[i][2 * j], L.inv), __uint_as_float(q[j] << 16)));
                v[i][2 * j + 1] = fabsf(__fmul_rn(__fmul_rn(v[i][2 * j + 1], L.inv), __uint_as_float(q[j] & 0xFFFF0000u)));
            }
            float4 *dst = reinterpret_cast<float4 *>(L.s + (row0 + i) * L.ld_s + k0);
            dst[0] = make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
            dst[1] = make_float4(v[i][4], v[i][5], v[i][6], v[i][7]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < kSalLaneRows; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int64_t row = row0 + i, k = k0 + j;
                float a = 0.f;
                if (row < g.rows && k < g.k) {
                    for (int h = 0; h < L.samples; ++h) {
                        const GradRef G = batch.grad[L.grad0 + h];
                        const float q = G.ld > 0 ? bf16_bits_to_float(reinterpret_cast<const uint16_t *>(G.p)[row * G.ld + k])
                                                 : reinterpret_cast<const float *>(G.p)[row * -G.ld + k];
                        a = h ? __fadd_rn(a, q) : q;
                    }
                    a = fabsf(__fmul_rn(__fmul_rn(a, L.inv), bf16_bits_to_float(L.w[row * L.ld_w + k])));
                    L.s[row * L.ld_s + k] = a;
                }
                v[i][j] = a;
            }
    }
    __syncthreads();                                         // (the tables)
    uint32_t key[kSalLaneRows][8];
#pragma unroll
    for (int i = 0; i < kSalLaneRows; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) key[i][j] = __float_as_uint(v[i][j]) & 0x7FFFFFFFu;
    auto reload = [&](int i, uint32_t (&q)[8]) {             // (this thread's own stores)
#pragma unroll
        for (int j = 0; j < 8; ++j) q[j] = row0 + i < g.rows && k0 + j < g.k ? canonical_bits(__float_as_uint(L.s[(row0 + i) * L.ld_s + k0 + j])) : 0u;
    };
    float counted[kSalLaneRows][kCounted<M, TOP>];
    uint32_t top;
    const uint32_t bits = select_rows<M, TOP>(key, g.n, g.score_mode != 0, s_keep, reload, counted, top);
    const bool in_kp = k0 < g.kp();
    // a lane's eight bits are byte (k0 / 8) mod 4 of their little-endian mask word: a warp stores 32 consecutive bytes of a row
    if (in_kp)
#pragma unroll
        for (int i = 0; i < kSalLaneRows; ++i) reinterpret_cast<uint8_t *>(L.nm_bits + (row0 + i) * g.wpr)[k0 >> 3] = (uint8_t)(bits >> (8 * i));
    // A record is of four lanes of every warp: their largest first, for the unit that all of them add up in.
    const int q = lane >> 2;
    top = max(top, __shfl_xor_sync(0xFFFFFFFFu, top, 1));
    top = max(top, __shfl_xor_sync(0xFFFFFFFFu, top, 2));
    if ((lane & 3) == 0) atomicMax(&s_top[q], top);
    __syncthreads();
    top = s_top[q];
    LaneSums s = sum_rows<M, TOP>(counted, (int)(top >> 23));
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
        s.low = min(s.low, __shfl_xor_sync(0xFFFFFFFFu, s.low, o));
        s.r += __shfl_xor_sync(0xFFFFFFFFu, s.r, o);
        s.d += __shfl_xor_sync(0xFFFFFFFFu, s.d, o);
    }
    if ((lane & 3) == 0) { atomicMin(&s_low[q], s.low); atomicAdd(&s_r[q], s.r); atomicAdd(&s_d[q], s.d); }
    __syncthreads();
    if (threadIdx.x < kSalWords) {
        const int word = (int)chunk * kSalWords + (int)threadIdx.x;
        const uint32_t t = s_top[threadIdx.x];
        if (word < g.wpr) L.records[(int64_t)rg * g.wpr + word] = make_record((int)(t >> 23), s_low[threadIdx.x], s_r[threadIdx.x], s_d[threadIdx.x]);
        const uint32_t best = __reduce_max_sync((1u << kSalWords) - 1u, t);
        if (threadIdx.x == 0 && best) atomicMax(L.max_key, best);
    }
}

int wave_grid(int64_t work_items) {
    int dev = 0, sm_count = 0;                               // asked for at every call: the current device may change
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sm_count <= 0)
        sm_count = 148;
    const int64_t blocks = (work_items + kSalThreads - 1) / kSalThreads;
    const int64_t cap = (int64_t)sm_count * 8;               // 8 resident CTAs of 256 threads per SM
    return (int)(blocks < cap ? (blocks > 0 ? blocks : 1) : cap);
}

bool vec_ok(const void *p, int64_t ld, int elem_bytes, int k) {
    return k % 4 == 0 && (ld * elem_bytes) % (4 * elem_bytes) == 0 && reinterpret_cast<uintptr_t>(p) % (4 * elem_bytes) == 0;
}

}  // namespace

cudaError_t launch_saliency_bits(const crisp_prune_layer_t *layers, const ScoreLayer *scores, int n, cudaStream_t st) {
    std::unique_ptr<SaliencyBatch> batch(new (std::nothrow) SaliencyBatch);
    if (!batch) return cudaErrorMemoryAllocation;
    Batch<SaliencyLayer, kBatchLayers> &b = batch->b;
    b.n = 0; b.first[0] = 0;
    int grads = 0;
    auto flush = [&]() -> cudaError_t {
        if (b.n == 0) return cudaSuccess;
        if (b.first[b.n] > 0x7FFFFFFFll) return cudaErrorInvalidValue;
        bool all_count = false;                              // (score modes may differ between the layers of a call, n and m may not)
        for (int i = 0; i < b.n; ++i) all_count = all_count || b.layer[i].g.score_mode != 0;
        const int top = top_counted(b.layer[0].g.n, all_count);
        const auto kern = b.layer[0].g.m == 4 ? (top == 0 ? saliency_bits_kernel<4, 0> : top == 1 ? saliency_bits_kernel<4, 1> : saliency_bits_kernel<4, 2>)
                                              : (top == 0 ? saliency_bits_kernel<8, 0> : top == 1 ? saliency_bits_kernel<8, 1> : saliency_bits_kernel<8, 2>);
        const cudaError_t e = launch_chained(kern, (unsigned)b.first[b.n], kSalItemThreads, 0, st, *batch);
        b.n = 0; grads = 0;
        return e;
    };
    for (int l = 0; l < n; ++l) {
        const crisp_prune_layer_t &P = layers[l];
        const ScoreLayer &S = scores[l];
        // more samples than the table holds: their running sum is formed in S first, and S takes the place of the samples
        const bool presum = P.samples > kBatchGrads;
        if (presum)
            for (int h = 0; h < P.samples; ++h)
                if (crisp_saliency_accumulate(P.d_grads[h], P.grad_dtypes[h], P.ld_grads[h], S.g.rows, S.g.k, P.d_saliency, P.ld_s,
                                              h == 0, st) != CRISP_OK)
                    return cudaErrorUnknown;
        const int samples = presum ? 1 : P.samples;
        if (b.n == kBatchLayers || grads + samples > kBatchGrads) {
            cudaError_t e = flush();
            if (e != cudaSuccess) return e;
        }
        SaliencyLayer &L = b.layer[b.n];
        L.g = S.g;
        L.w = P.d_w_bf16; L.ld_w = P.ld_w;
        L.s = P.d_saliency; L.ld_s = P.ld_s;
        L.max_key = S.max_key; L.nm_bits = S.nm_bits; L.records = S.records;
        L.inv = 1.0f / (float)P.samples;
        L.chunks = (int)((S.g.kp() + kSalChunk - 1) / kSalChunk);
        L.grad0 = grads; L.samples = samples;
        auto vec = [](const void *p, int64_t ld, int bytes) { return reinterpret_cast<uintptr_t>(p) % 16 == 0 && ld * bytes % 16 == 0; };
        bool ok = vec(L.w, L.ld_w, 2) && vec(L.s, L.ld_s, 4);
        for (int h = 0; h < samples; ++h) {
            GradRef &G = batch->grad[grads + h];
            G.p = presum ? P.d_saliency : P.d_grads[h];
            const bool f32 = presum || P.grad_dtypes[h] == 1;
            const int64_t ld = presum ? P.ld_s : P.ld_grads[h];
            G.ld = f32 ? -ld : ld;
            ok = ok && vec(G.p, ld, f32 ? 4 : 2);
        }
        L.vec_ok = ok;
        grads += samples;
        b.first[b.n + 1] = b.first[b.n] + (S.g.mp() / kM1Rows) * (int64_t)L.chunks;
        ++b.n;
    }
    return flush();
}

}  // namespace crisp

extern "C" {

CRISP_API crisp_status_t crisp_saliency_accumulate(const void *d_grad, int32_t grad_dtype, int64_t ld_g, int32_t rows,
                                                   int32_t k, float *d_acc, int64_t ld_acc, int32_t first, void *stream) {
    using namespace crisp;
    if (!d_grad || !d_acc || (grad_dtype != 0 && grad_dtype != 1) || (first != 0 && first != 1)) return CRISP_INVALID_ARG;
    if (rows <= 0 || k <= 0 || ld_g < k || ld_acc < k) return CRISP_BAD_SHAPE;
    const int gb = grad_dtype ? 4 : 2;
    if (reinterpret_cast<uintptr_t>(d_grad) % gb || reinterpret_cast<uintptr_t>(d_acc) % 4) return CRISP_INVALID_ARG;
    const bool vec = vec_ok(d_grad, ld_g, gb, k) && vec_ok(d_acc, ld_acc, 4, k);
    const int grid = wave_grid((int64_t)rows * (vec ? k / 4 : k));
    cudaStream_t st = (cudaStream_t)stream;
    if (grad_dtype == 0) {
        if (vec) saliency_accumulate_kernel<true, true><<<grid, kSalThreads, 0, st>>>(d_grad, ld_g, rows, k, d_acc, ld_acc, first);
        else saliency_accumulate_kernel<true, false><<<grid, kSalThreads, 0, st>>>(d_grad, ld_g, rows, k, d_acc, ld_acc, first);
    } else {
        if (vec) saliency_accumulate_kernel<false, true><<<grid, kSalThreads, 0, st>>>(d_grad, ld_g, rows, k, d_acc, ld_acc, first);
        else saliency_accumulate_kernel<false, false><<<grid, kSalThreads, 0, st>>>(d_grad, ld_g, rows, k, d_acc, ld_acc, first);
    }
    return cudaGetLastError() == cudaSuccess ? CRISP_OK : CRISP_CUDA_ERROR;
}

CRISP_API crisp_status_t crisp_saliency_finish(const float *d_acc, int64_t ld_acc, const uint16_t *d_w_bf16, int64_t ld_w,
                                               int32_t rows, int32_t k, int32_t samples, float *d_saliency, int64_t ld_s,
                                               void *stream) {
    return crisp_saliency_finish_max(d_acc, ld_acc, d_w_bf16, ld_w, rows, k, samples, d_saliency, ld_s, nullptr, stream);
}

CRISP_API crisp_status_t crisp_saliency_finish_max(const float *d_acc, int64_t ld_acc, const uint16_t *d_w_bf16,
                                                   int64_t ld_w, int32_t rows, int32_t k, int32_t samples,
                                                   float *d_saliency, int64_t ld_s, void *d_mask_workspace, void *stream) {
    using namespace crisp;
    if (d_mask_workspace && reinterpret_cast<uintptr_t>(d_mask_workspace) % kAlign) return CRISP_INVALID_ARG;
    if (!d_acc || !d_w_bf16 || !d_saliency || samples <= 0) return CRISP_INVALID_ARG;
    if (rows <= 0 || k <= 0 || ld_acc < k || ld_w < k || ld_s < k) return CRISP_BAD_SHAPE;
    if (reinterpret_cast<uintptr_t>(d_acc) % 4 || reinterpret_cast<uintptr_t>(d_w_bf16) % 2 ||
        reinterpret_cast<uintptr_t>(d_saliency) % 4)
        return CRISP_INVALID_ARG;
    const bool vec = vec_ok(d_acc, ld_acc, 4, k) && vec_ok(d_w_bf16, ld_w, 2, k) && vec_ok(d_saliency, ld_s, 4, k);
    const int grid = wave_grid((int64_t)rows * (vec ? k / 4 : k));
    const float inv = 1.0f / (float)samples;
    cudaStream_t st = (cudaStream_t)stream;
    uint32_t *max_key = reinterpret_cast<uint32_t *>(d_mask_workspace);
    if (max_key && cudaMemsetAsync(max_key, 0, kAlign, st) != cudaSuccess) return CRISP_CUDA_ERROR;
    if (vec) saliency_finish_kernel<true><<<grid, kSalThreads, 0, st>>>(d_acc, ld_acc, d_w_bf16, ld_w, rows, k, inv, d_saliency, ld_s, max_key);
    else saliency_finish_kernel<false><<<grid, kSalThreads, 0, st>>>(d_acc, ld_acc, d_w_bf16, ld_w, rows, k, inv, d_saliency, ld_s, max_key);
    return cudaGetLastError() == cudaSuccess ? CRISP_OK : CRISP_CUDA_ERROR;
}

}  // extern "C"
