// Internal declarations shared by the translation units of libfdc (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "fdc.h"

#define FDC_PAIR_COUNTERS 65536
// Work split of the tcgen05 attention kernel: the layers of one forward pass see the same
// per-scene counts, so the split is computed once per pass (by a launch of the kernel that does
// nothing else, before the pass's first attention launch) and kept here with the counts it was
// computed from; the attention launches only check that the counts are unchanged.  Layout, in
// int32: [0..15] header, [16..) n_active[FDC_MEMO_BATCH], tiles[FDC_MEMO_BATCH],
// prev[FDC_MEMO_BATCH + 1], [FDC_MEMO_ENTRIES..) first and last unit of each CTA (2 x int64), [FDC_MEMO_SPREAD..) how each
// CTA's part is spread over its pair's list (4 each).
#define FDC_MEMO_BATCH 256
#define FDC_MEMO_CTAS 256
#define FDC_MEMO_ENTRIES 800
#define FDC_MEMO_SPREAD (FDC_MEMO_ENTRIES + 4 * FDC_MEMO_CTAS)
#define FDC_MEMO_INTS (FDC_MEMO_SPREAD + 4 * FDC_MEMO_CTAS)

namespace fdc {

// Device-resident template tables (built on the host by fdc_plan_graph).
struct PlanDev {
    int32_t  n, m, P, T, W, max_active, ntile_max, pad0;
    uint64_t anc[FDC_MAX_NODES];     // bit u of anc[v]: a path u -> ... -> v exists (Eq. 1)
    uint64_t par[FDC_MAX_NODES];     // bit u of par[v]: edge (u, v)
    int32_t  base[FDC_MAX_NODES + 1];
    int32_t  pad1;
    int32_t  cap[FDC_MAX_NODES];
    int32_t  nfixed[FDC_MAX_NODES];
    int32_t  indeg[FDC_MAX_NODES];   // incoming edges, duplicates counted (Alg. 1's initial d_v)
};

// Per-scene scheduler state (caller-owned device memory, opaque to the caller).
struct alignas(16) SceneState {
    uint64_t ready;                  // S of Algorithm 1 as a node bitset
    uint64_t done;                   // finished fields
    int32_t  n_active;               // width of the last emitted pass
    int32_t  pass;                   // passes emitted so far
    int32_t  pad[2];
    int32_t  d[FDC_MAX_NODES];       // unfinished prerequisites of each field
    int32_t  tok[FDC_MAX_NODES];     // rows of the field present in the cache (after this pass's append)
    int32_t  lim[FDC_MAX_NODES];     // the field is finished when tok reaches lim
    int32_t  node[FDC_MAX_NODES];    // packed list of the last emitted pass
};

}  // namespace fdc

// Arguments of an fdc_kv_append call that has been recorded instead of launched (fused append).
struct fdc_pending_append {
    int            valid;
    fdc_kv_desc    kv;
    int32_t        layer;
    const int32_t* d_n_active;
    const int32_t* d_kv_row;
    const void*    d_k_new;
    const void*    d_v_new;
    void*          stream;
};

namespace fdc {
// How the cluster kernel (fdc_attn_cluster.cu) cuts a launch.
struct ClusterShape {
    int nblk, qsplit, per_sm;        // blocks per cluster, clusters per (scene, KV head) pair, blocks per SM (1 or 2)
};
struct ClusterProblem {
    int64_t pairs;
    int32_t mmax, head_dim, P, T, sm_count;
    bool operator==(const ClusterProblem& o) const
    {
        return pairs == o.pairs && mmax == o.mmax && head_dim == o.head_dim && P == o.P && T == o.T && sm_count == o.sm_count;
    }
};
#ifdef __CUDACC__
#define FDC_HD __host__ __device__ __forceinline__
#else
#define FDC_HD inline
#endif
// First of block `rank`'s run among a pair's `parts` tile parts (cluster kernels): equal runs.  The listed parts beyond the
// prefix count in full: while the last fields of a template are decoded all of them hold rows.  Counted half, a block with many of them took up
// to twice as many.  us a layer, half / full: fp32, 14/2 heads x 64, 9 fields, 4 scenes, prefix 3000, the last field 45.6 / 35.2; 4/2 x 64, 24
// fields, 8 scenes, prefix 2048, the last field 56.9 / 39.3; bf16, 50 pairs of 50 rows x 64, prefix 2215 43.0 / 37.7; 4 pairs of 112 rows x 128, prefix
// 707 12.9 / 11.6.  What it gained was less: fp32, 32/8 x 128, six fields at work, 8 scenes, prefix 2048 75.7 / 79.5.
// (= rank * parts / nblk; `div(x)` is x / nblk, which the kernels do without a division)
template <class Div>
FDC_HD int run_begin(int rank, int nblk, int parts, Div&& div)
{
    const int each = (int)div((uint32_t)parts);
    return rank * each + (int)div((uint32_t)(rank * (parts - each * nblk)));
}
// Division of x < 2^28 by a small n (1 to 16) or of x < 2^24 by any n < 256: div_by(x, div_inverse(n)) = x / n.
inline uint32_t div_inverse(int n) { return n > 1 ? (uint32_t)((1ull << 32) / (uint32_t)n + 1) : 0u; }
FDC_HD uint32_t div_by(uint32_t x, uint32_t inverse)
{
#ifdef __CUDA_ARCH__
    return inverse ? __umulhi(x, inverse) : x;
#else
    return inverse ? (uint32_t)(((uint64_t)x * inverse) >> 32) : x;
#endif
}
// Weights of the tcgen05 kernels' work split (the unit is a quarter of a tile inside the prefix).
constexpr int W_PREFIX = 4;
constexpr int W_MASKED = 6;          // a tile beyond the prefix (bitmap selects, V clean-up): measured about 1.5 prefix tiles
constexpr int W_PAIR = 32;           // finishing a (scene, KV head) pair (drain, partial write, next queries)
// Weighted length of a pair's first `nt` tiles, of which the first `np` are whole tiles of the prefix.
FDC_HD int weighted_tiles(int np, int nt) { return nt <= np ? nt * W_PREFIX : np * W_PREFIX + (nt - np) * W_MASKED; }
// One part per CTA leaves CTAs idle when the parts per pair do not divide the CTAs evenly
// (64 pairs on 148 CTAs: 2 or 3 parts, a CTA carries up to 16 % more than the average).  Where the
// shares are long enough for a pair boundary inside a CTA to cost less than that, equal shares of the
// weighted length win after all: from about 200 prefix tiles per CTA, half of that with more than 64 query
// rows (the row form), whose tiles take longer.  Measured there, us a layer one part / equal shares, 32 / 8
// heads x 128, 32 fields: 26 tiles per CTA (8 scenes, prefix 3840) 57 / 65, 60 tiles 85.9 / 85.1, 100 tiles
// 121 / 116, 150 tiles 165 / 158; 100 tiles in 5 scenes (40 pairs) 124 / 116, in 12 scenes (96 pairs) 153 /
// 125; where the parts divide well (48 pairs in 144 parts) 103 / 107.
// length: of all pairs, W_PAIR for each included; part: the longest part of a cut for one part per CTA.
FDC_HD bool equal_shares(long long length, int part, int n_cta, int mmax)
{
    const long long avg = length / n_cta;
    return avg * (mmax > 64 ? 2 : 1) >= 200 * W_PREFIX && (long long)part * 100 > avg * 108;
}
bool pairs_in_two_parts(int64_t pairs, int mmax, int P, int ntile_max, int n_cta);      // fdc_attn_tc.cu
ClusterShape pick_cluster(const ClusterProblem& c, float* us);      // us (may be NULL): the estimated time
bool route_problem(const ClusterProblem& c, ClusterShape* cut);     // the cut, and whether the cluster kernel is the one to take (head_dim 64: always)
int cluster_ring(int head_dim, int rows, int nblk, int per_sm);     // stages of a block's ring (bf16); 0: no room for the partials beside it
// The largest cluster of at most `nblk` blocks that the device can place (a single block always can).
template <class F>
int largest_placeable(int nblk, F&& placeable)
{
    while (nblk > 1 && !placeable(nblk)) --nblk;
    return nblk;
}
}  // namespace fdc

// Everything the work split of the tcgen05 attention kernel depends on (host side).
struct fdc_split_key {
    uint32_t       tables_gen;
    const int32_t* d_n_active;
    const int32_t* d_ntiles;
    int32_t        batch, hkv, n_cta, P;
    void*          stream;
    int            valid;
};

struct fdc_plan {
    fdc::PlanDev  h;                 // host copy
    fdc::PlanDev* d;                 // device copy
    int32_t*      d_status;          // sticky FDC_DEV_* bits
    int32_t*      d_ticket;          // [2] scratch of the frontier kernel's cross-block reduction
    int32_t*      d_pair_cnt;        // [FDC_PAIR_COUNTERS] arrivals per (scene, KV head) of the fused combine (zero between calls)
    int32_t*      d_split_memo;      // [FDC_MEMO_INTS] work split of the current pass and the counts it was made from
    uint32_t      tables_gen;        // bumped by every call that rewrites the pass tables (state_init, frontier, build_masks)
    uint32_t      split_gen;         // number of the last split launch (stored in the memo's header)
    fdc_split_key split_key;         // what the memo was computed for
    uint32_t      attn_gen;          // tables_gen at the last attention launch of a kernel that reads ahead
    void*         attn_stream;       // and its stream
    int           attn_gen_valid;
    int           fuse_append;       // fdc_set_fused_append
    fdc_pending_append pend;         // recorded append waiting for its attention call
    int           device;
    int           sm_count;
    int           attn_kernel;       // 0 auto
    fdc::ClusterProblem route_for;   // the problem `route_shape` / `route_cluster` were chosen for (sm_count 0: none yet)
    fdc::ClusterShape   route_shape;
    int           route_cluster;     // with attn_kernel 0: the cluster kernel is the faster one
    void*         prof;              // event records of fdc_profile (nullptr when never enabled)
    int           prof_on;
    int32_t*      succ_ptr;          // host CSR successor lists (kept for inspection)
    int32_t*      succ;
};

namespace fdc {

// Attention launch parameters (passed by value).
struct AttnParams {
    const void*     k;               // layer base
    const void*     v;
    int64_t         stride_scene, stride_head, stride_row;   // elements
    const void*     q;               // [batch][max_active][hq][D]
    void*           out;
    const uint64_t* mask;            // [batch][max_active][W]
    const int32_t*  tiles;           // [batch][ntile_max]
    const int32_t*  ntiles;          // [batch]
    const int32_t*  n_active;        // [batch]
    float*          ws_o;            // [slots][mmax][D]
    float*          ws_ml;           // [slots][mmax][2]
    int32_t         batch, hkv, hq, group, max_active, mmax, W, P, rows, ntile_max, n_cta;
    float           scale_log2;      // softmax scale * log2(e)
    int32_t*        status;          // sticky FDC_DEV_* bits
    int32_t*        pair_cnt;        // per (scene, KV head) arrival counters: the split kernel also combines (nullptr: it does not)
    int32_t*        split_memo;      // [FDC_MEMO_INTS] (nullptr: the work split is always computed)
    uint32_t        seq;             // number of the split launch the memo must come from
    int32_t         early;           // the pass tables, the memo and the prefix rows were complete before the kernel
                                     // preceding this one in the stream began: they may be read ahead of the dependency wait
    ClusterShape    cluster;         // cut of the launch (cluster kernel)
    const int32_t*  app_row;         // fused append: [batch][max_active] cache row of each branch's new K/V vector (nullptr: none)
    const void*     app_k;           // [batch][max_active][hkv][D]
    const void*     app_v;
};

extern int64_t g_launches;
void note_launch();
int  set_cuda_error(cudaError_t e);                  // records the message, returns FDC_ERR_CUDA

int launch_attn_ref(const AttnParams& p, int dtype, int head_dim, cudaStream_t st);
int launch_attn_f32(const AttnParams& p, int head_dim, cudaStream_t st);
int launch_attn_cluster(const AttnParams& p, int head_dim, cudaStream_t st);
int launch_attn_tc(const AttnParams& p, int head_dim, cudaStream_t st);
int launch_attn_tc_split(const AttnParams& p, int head_dim, cudaStream_t st);   // computes the work split only (into p.split_memo)
int launch_attn_combine(const AttnParams& p, int dtype, int head_dim, cudaStream_t st);
void prof_destroy(fdc_plan* plan);
int  check_kv_desc(const fdc_plan* plan, const fdc_kv_desc* kv, int32_t layer);
bool takes_cluster_kernel(fdc_plan* plan, const fdc_kv_desc* kv);    // fdc_decode_attn would run the cluster kernel (else: the tcgen05 kernel, for bf16)
bool fuses_append(fdc_plan* plan, const fdc_kv_desc* kv);            // ... and the kernel it would run can carry out a recorded append
int  launch_kv_append(fdc_plan* plan, const fdc_kv_desc* kv, int32_t layer, const int32_t* d_n_active, const int32_t* d_kv_row,
                      const void* d_k_new, const void* d_v_new, void* stream);
int  flush_pending_append(fdc_plan* plan);     // launches a recorded append on its own (no-op when there is none)

// cudaFuncAttributeMaxDynamicSharedMemorySize is kept by the runtime per kernel and device, and the last call wins.  So every call sets the
// same value, all that a block can have: threads that launch with different sizes cannot lower it for one another, in whatever order
// they come.  One SmemLimit per kernel remembers the devices that have been told.
constexpr int kMaxDevices = 64;
struct SmemLimit {
    std::atomic<size_t> set[kMaxDevices] = {};
};
inline int raise_dynamic_smem(const void* kernel, size_t bytes, SmemLimit& limit)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return set_cuda_error(e);
    const bool known = dev >= 0 && dev < kMaxDevices;
    if (known && bytes <= limit.set[dev].load(std::memory_order_acquire)) return FDC_OK;
    int block = 0;
    cudaFuncAttributes own;
    e = cudaDeviceGetAttribute(&block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&own, kernel);
    if (e != cudaSuccess) return set_cuda_error(e);
    const size_t room = (size_t)block > own.sharedSizeBytes ? (size_t)block - own.sharedSizeBytes : 0;
    const size_t most = bytes > room ? bytes : room;            // (more than there is: refused here)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if (e != cudaSuccess) return set_cuda_error(e);
    if (known) limit.set[dev].store(most, std::memory_order_release);
    return FDC_OK;
}

inline cudaLaunchAttribute cluster_of_two()
{
    cudaLaunchAttribute a;
    a.id = cudaLaunchAttributeClusterDimension;
    a.val.clusterDim.x = 2;
    a.val.clusterDim.y = a.val.clusterDim.z = 1;
    return a;
}
// Whether the device holds n_cta blocks of a kernel in clusters of two at once (asked once per device): FDC_OK, or FDC_ERR_SHAPE (another build's launch).
struct PairsPlaceable {
    std::atomic<int> known[kMaxDevices] = {};         // 0: not asked; n + 1: that many clusters
    int all(const void* kernel, int threads, size_t smem, int n_cta, SmemLimit& limit)
    {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return FDC_ERR_SHAPE;
        int n = known[dev].load(std::memory_order_relaxed);
        if (n == 0) {
            const int rc = raise_dynamic_smem(kernel, smem, limit);
            if (rc) return rc;
            cudaLaunchConfig_t one = {};
            cudaLaunchAttribute at = cluster_of_two();
            one.gridDim = dim3((unsigned)n_cta);
            one.blockDim = dim3((unsigned)threads);
            one.dynamicSmemBytes = smem;
            one.attrs = &at;
            one.numAttrs = 1;
            int clusters = 0;
            if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &one) != cudaSuccess) {
                cudaGetLastError();
                clusters = 0;
            }
            known[dev].store(n = clusters + 1, std::memory_order_relaxed);
        }
        return 2 * (n - 1) >= n_cta ? FDC_OK : FDC_ERR_SHAPE;
    }
};

// ----------------------------------------------------------------------------------
// device helpers
// ----------------------------------------------------------------------------------
#ifdef __CUDACC__
// 64 bits of a bitmap of `W` words starting at bit position `start` (may be negative or run
// past the end: bits outside [0, 64*W) read as 0).
__device__ __forceinline__ uint64_t extract64(const uint64_t* __restrict__ words, int W, int start)
{
    if (start <= -64) return 0ull;
    if (start < 0) return W > 0 ? (words[0] << (-start)) : 0ull;
    int w = start >> 6, sh = start & 63;
    if (w >= W) return 0ull;
    uint64_t lo = words[w] >> sh;
    if (sh && w + 1 < W) lo |= words[w + 1] << (64 - sh);
    return lo;
}

// Visibility of the 64 rows of KV tile `tile` for one branch: prefix rows are all visible.
__device__ __forceinline__ uint64_t tile_rowmask(const uint64_t* __restrict__ words, int W, int P, int tile)
{
    int r0 = tile * FDC_TILE_ROWS;
    int npre = P - r0;
    uint64_t pm = npre >= 64 ? ~0ull : (npre <= 0 ? 0ull : ((1ull << npre) - 1ull));
    if (npre >= 64) return pm;
    return pm | extract64(words, W, r0 - P);
}

// Work split shared by the split pass and the combine pass: unit u (one KV tile of one
// (scene, KV head) pair, pairs in scene-major order) belongs to CTA floor(u * n_cta / U).
__device__ __forceinline__ long long cta_first_unit(long long c, long long U, long long n_cta)
{
    return (c * U + n_cta - 1) / n_cta;
}
__device__ __forceinline__ int unit_cta(long long u, long long U, long long n_cta)
{
    return (int)((u * n_cta) / U);
}
#endif

}  // namespace fdc
