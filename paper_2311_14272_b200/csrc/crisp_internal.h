// Internal declarations shared by the translation units of libcrisp.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "crisp.h"
#include "settled.h"

namespace crisp {

// Layer epilogue applied to the fp32 accumulator before the store: Y = act(W*X + bias).
struct Epilogue {
    const float *bias;      // device, [rows] fp32, or nullptr
    int relu;               // max(., 0) after the bias
};

// Shape of one layer after padding to whole blocks.
struct Geometry {
    int rows, k, n, m, bm, bk;
    int score_mode;
    int nrt;        // row tiles
    int nblk;       // k-blocks per row tile
    int kkeep;      // kept k-blocks per row tile
    int wpr;        // uint32 words of bit mask per (padded) row = nblk * bk / 32
    int idx_bits;   // log2(m)
    __host__ __device__ int64_t mp() const { return (int64_t)nrt * bm; }
    __host__ __device__ int64_t kp() const { return (int64_t)nblk * bk; }
    __host__ __device__ int groups() const { return bk / m; }
    __host__ __device__ int64_t vals_per_block() const { return (int64_t)bm * groups() * n; }
    __host__ __device__ int64_t nnz() const { return (int64_t)nrt * kkeep * vals_per_block(); }
    __host__ __device__ int64_t idx_words() const { return (nnz() * idx_bits + 31) / 32; }
};

// One launch over several layers: work units (items, CTAs) are numbered through, layer l owning first[l] .. first[l + 1] - 1.
// The table travels as a kernel parameter (no copy, nothing to keep alive).  CAP = 1 is the single-layer call.
constexpr int kBatchLayers = 64;
template <typename L, int CAP>
struct Batch {
    int n;
    int64_t first[CAP + 1];
    L layer[CAP];
#ifdef __CUDACC__
    __device__ __forceinline__ int find(int64_t unit) const {       // the layer that owns `unit`
        if constexpr (CAP == 1) return 0;
        int lo = 0, hi = n - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (first[mid] <= unit) lo = mid; else hi = mid - 1;
        }
        return lo;
    }
#endif
};

#ifdef __CUDACC__
// Programmatic dependent launch.  A kernel launched with the programmatic-serialization attribute may start before the
// kernel in front of it in the stream has finished; wait_for_prerequisites() returns when that one has finished and its
// writes are visible, and every thread that touches global memory another kernel may write or read calls it first.
// launch_dependents() lets the next kernel of the stream start its own set-up (it waits in the same way).
// Such a kernel is alive while its predecessors still write, so it reads whatever another kernel may have written (which
// is every buffer of the caller too: the weights may come from crisp_decode) with plain loads, behind the wait.  The
// read-only path (__ldg, const __restrict__) is for data that stays as it is for the kernel's whole life: its loads may be
// moved above the wait and need not see what the wait makes visible.  (Plain loads take the same time.)
// What a product may read ahead of the wait where its handle is settled (settled.h), walk lists and weight tiles, comes from L2 (__ldcg, and TMA): an
// SM's L1 may hold a line from before the encode.
__device__ __forceinline__ void wait_for_prerequisites() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// The kernels of the mask / encode / decode chain begin with this.  The next kernel may begin as this one's last CTAs end; asked for at the
// start (launch_dependents), its CTAs wait beside this one's on some SMs and leave others empty: mask, encoding and decoding in a row of 2033 x 116
// 35.7 us instead of 27.8, 1024 x 1024 22.9 and 19.9, 4096 x 4096 60.0 and 58.2.
__device__ __forceinline__ void chain_kernels() { wait_for_prerequisites(); }

// Clusters: rank of this CTA, the place of one of its shared-memory addresses in another rank, loads from there, and the barrier
// of all threads of a cluster.
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t peer_address(uint32_t smem, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t lds32_peer(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float4 lds128_peer(uint32_t a) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}

// (`cluster` CTAs form a thread-block cluster; 1: none)
template <typename... Params, typename... Args>
cudaError_t launch_clusters(void (*kern)(Params...), unsigned grid, unsigned threads, size_t smem, cudaStream_t st, unsigned cluster,
                            const Args &...args) {
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
    if (e != cudaSuccess) (void)cudaGetLastError();          // reported here, not to the caller's next check
    return e;
}
template <typename... Params, typename... Args>
cudaError_t launch_chained(void (*kern)(Params...), unsigned grid, unsigned threads, size_t smem, cudaStream_t st, const Args &...args) {
    return launch_clusters(kern, grid, threads, smem, st, 1u, args...);
}
#endif

int sm_count_of(int device);                // multiprocessors of a device, looked up once (spmm_tc.cu)

constexpr int kMaxBlocksPerRowTile = 4096;
constexpr size_t kAlign = 256;
inline size_t align_up(size_t x, size_t a = kAlign) { return (x + a - 1) / a * a; }

}  // namespace crisp

struct crisp_mask_s {
    crisp::Geometry g;
    int32_t *d_blk_col;     // [nrt, kkeep]
    uint32_t *d_nm_bits;    // [mp, wpr]
    int image_kind;         // CRISP_PATH_* of the execution image crisp_encode will lay out: fixed when the
                            // mask is built, so that crisp_encode_sizes and crisp_encode always agree
};

namespace crisp {
// Launch plan of the tensor-core kernel for one set of operands (spmm_tc.cu); cached in the handle so that
// repeated products on the same buffers skip the tensor-map encoding.
struct TcPlan;
void tc_plan_destroy(TcPlan *plan);
struct GatherPlan;          // tensor map of the execution image for the products of spmm_gather.cu
void gather_plan_destroy(GatherPlan *plan);
struct HaloPlan;            // launch plan of the last convolution of spmm_halo.cu
void halo_plan_destroy(HaloPlan *plan);
}  // namespace crisp

struct crisp_handle_s {
    crisp::Geometry g;
    // canonical format
    int32_t *d_blk_col;
    uint16_t *d_vals;
    uint32_t *d_idx;
    // execution image
    int32_t *d_status;      // first word of the exec buffer
    uint8_t *d_exec;        // payload after the 256-byte header
    size_t exec_payload_bytes;
    int exec_kind;          // CRISP_PATH_* the image was laid out for (DIRECT = none)
    int forced_path;        // -1 = default
    crisp::Epilogue epilogue;
    int nt_override;        // tuning: 64-column boxes per CTA tile (0 = chosen by the library)
    int group_override;     // tuning: most kept blocks a pipeline stage may take (0 = chosen by the library)
    unsigned long long wait_limit_cycles;   // bound of every in-kernel wait (0 = default)
    int debug_skip_stage;   // test hook: the producer leaves out the loads of this pipeline fill (-1 = none)
    crisp::TcPlan *plan;    // cached launch plan of the last tensor-core product (or nullptr)
    crisp::HaloPlan *halo;                  // cached launch plan of the last convolution that shares loads among taps (or nullptr)
    crisp::GatherPlan *gather;              // made by the first product on a layout TMA cannot address (or nullptr)
    // Products and convolutions of one handle may come from several host threads: the three plans above and what follows are read and
    // written under this lock, and a launch is made from copies.
    std::mutex plan_lock;
    crisp_launch_info_t last;               // what the last product on this handle launched
    crisp::Settled settled;                 // and whether the next one may read the weights early
    int64_t last_resident;                  // and the bytes of weight tiles it kept in shared memory
};

namespace crisp {

// mask_kernels.cu
cudaError_t launch_build_mask(const float *d_s, int64_t ld, const Geometry &g, int32_t *d_blk_col,
                              uint32_t *d_nm_bits, void *d_workspace, bool max_known, cudaStream_t st);
// One layer of a batched launch: the saliency that is scored, the group bits, scores and what they are made from (in the mask workspace)
// and where the selection writes its block list.
struct ScoreLayer {
    Geometry g;
    const float *s;
    int64_t ld;
    uint32_t *max_key;
    const uint32_t *maxima;              // partial maxima that max_key is made from, n_maxima of them; nullptr: max_key stands
    int n_maxima;
    uint32_t *nm_bits;
    unsigned long long *score, *records;
    int32_t *blk_col;
    int vec_ok;                          // (filled in by the launchers)
};
constexpr int kMaxMaxima = 2048;         // CTAs of the pass over S
void set_workspace(ScoreLayer *L, void *d_workspace);        // max_key, score, records of a layer whose geometry is set
// Whether only a group's n largest values count, so that they are found with minima and maxima (1, 2; 0: no).
inline int top_counted(int n, bool all_count) { return !all_count && n <= 2 ? n : 0; }
cudaError_t launch_clear_scores(const ScoreLayer *layers, int n, cudaStream_t st);     // max_key
cudaError_t launch_block_scores(const ScoreLayer *layers, int n, cudaStream_t st);
cudaError_t launch_block_selects(const ScoreLayer *layers, int n, cudaStream_t st);
// per-row-tile selection alone, on the scores and group bits an earlier launch_build_mask left behind
cudaError_t launch_block_select(const Geometry &g, const void *d_workspace, int32_t *d_blk_col, uint32_t *d_nm_bits,
                                cudaStream_t st);
size_t mask_workspace_bytes(const Geometry &g);
size_t mask_score_bytes(const Geometry &g);                  // its first part: the maximum and the scores

// saliency_kernels.cu: saliency, group bits, score records and layer maxima of a network in one launch (max_key cleared before)
cudaError_t launch_saliency_bits(const crisp_prune_layer_t *layers, const ScoreLayer *scores, int n, cudaStream_t st);

// encode_kernels.cu
constexpr int kMaxBlockWords = kMaxBlocksPerRowTile / 32;
// One layer of an encode launch: canonical blocks, and the execution image of `kind` with its walk lists (kind DIRECT:
// canonical blocks only, walk_col = nullptr).  The layers of one launch share n and m.
struct EncodeLayer {
    Geometry g;
    const uint16_t *w;
    int64_t ld;
    const int32_t *mask_blk_col;
    const uint32_t *nm_bits;
    int32_t *blk_col;
    uint16_t *vals;
    uint32_t *idx;
    uint8_t *image;
    int32_t *walk_col, *walk_len;
    uint32_t *header;                    // 64 words cleared by the kernel (the handle's status block), or nullptr
    int kind, nst, wcap, stack;
    uint32_t a_bytes, entry_bytes;
    int vec_ok;                          // (filled in by the launcher)
};
cudaError_t launch_encode(const EncodeLayer *layers, int n, cudaStream_t st);
cudaError_t launch_decode(const Geometry &g, const int32_t *d_blk_col, const uint16_t *d_vals,
                          const uint32_t *d_idx, uint16_t *d_w, int64_t ld, cudaStream_t st);

// spmm_tc.cu: tensor-core path and its execution image
struct TcImageLayout {
    int r;                  // row tiles per 128-row CTA tile
    int nst;                // 128-row CTA tiles
    int wcap;               // capacity of one CTA tile's walk list (union of its row tiles' kept blocks)
    int stack;              // copies of the image, each shifted by 128 / stack rows (thin single-tile layers)
    uint32_t a_bytes;       // weight tile bytes per walk entry
    uint32_t entry_bytes;   // weight tile + metadata (two of each for the two-addend image)
    int addends;            // sparse tiles per walk entry: 1, or 2 for the two-addend image
    size_t walk_col_off, walk_len_off, image_off, total_bytes;   // offsets inside the exec payload
};
bool tc_pattern_is_sparse(const Geometry &g);
TcImageLayout tc_image_layout(const Geometry &g, int kind);      // kind: CRISP_PATH_DENSE / SPARSE / SPARSE2
bool tc_operands_ok(const void *x, int64_t ldx, const void *y, int64_t ldy, int y_dtype, int64_t ncols);
// Convolution geometry for the implicit-GEMM mode (stride 1): NHWC activation, ho x wo output pixels.
struct ConvGeom { int batch, height, width, channels, kh, kw, pad, ho, wo, nhwc_out; };
inline bool same_conv(const ConvGeom &a, const ConvGeom &b) {
    return a.batch == b.batch && a.height == b.height && a.width == b.width && a.channels == b.channels &&
           a.kh == b.kh && a.kw == b.kw && a.pad == b.pad && a.nhwc_out == b.nhwc_out;
}
// The pixel box tw x th x tb (n pixels) of a column tile of spmm_tc.cu's gather that covers the fewest pixels outside the images, then the
// widest, then the tallest; `row` pixels of Y fill a 128-byte staging row.  -> pixels covered, -1: none fits
int64_t conv_box(int n, int row, const ConvGeom &cv, int *tw, int *th, int *tb);
// spmm_halo.cu: convolutions whose taps share one load of the activation
cudaError_t launch_spmm_halo(crisp_handle_s *h, const uint16_t *d_x, void *d_y, int64_t ldy, int y_dtype, const ConvGeom &cv, int device,
                             cudaStream_t st, bool *done);
extern EncodeCount encodes;                                   // (encode_kernels.cu)
// After the launch of a product: for crisp_last_launch, and for h->settled; moment: encodes.now() before it.
void note_launch(crisp_handle_s *h, const crisp_launch_info_t &info, int64_t resident_bytes, cudaStream_t st, uint64_t moment);
// conv == nullptr: d_x is the [k, ncols] matrix.  Otherwise d_x is the activation and ncols = batch*ho*wo.
// `h->plan` is reused when the operands, shape and epilogue are those of the previous call; `h->last` is filled in.
cudaError_t launch_spmm_tc(crisp_handle_s *h, int kind, const uint16_t *d_x, int64_t ldx, int64_t ncols,
                           void *d_y, int64_t ldy, int y_dtype, const ConvGeom *conv, cudaStream_t st);
// spmm_gather.cu: bf16 products on layouts TMA cannot address, on the same weight tiles
bool gather_supported(const crisp_handle_s *h, int64_t ncols, int y_dtype);
cudaError_t launch_spmm_gather(crisp_handle_s *h, const uint16_t *d_x, int64_t ldx, int64_t ncols, void *d_y, int64_t ldy,
                               cudaStream_t st);
// spmm_direct.cu
cudaError_t launch_spmm_direct(const Geometry &g, const int32_t *d_blk_col, const uint16_t *d_vals,
                               const uint32_t *d_idx, const uint16_t *d_x, int64_t ldx, int64_t ncols,
                               void *d_y, int64_t ldy, int y_dtype, const Epilogue &epi, cudaStream_t st);

}  // namespace crisp
