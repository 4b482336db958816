// A (scene, KV head) pair's attention by thread-block clusters: what the bf16 kernel (fdc_attn_cluster.cu) and
// the fp32 kernel (fdc_attn_f32.cu) share.  The blocks of a cluster take equal runs of the pair's tile parts (16
// or 32 rows), a block's warps take the run's stages in turn, and the partial results meet in (distributed)
// shared memory.  A kernel's arithmetic is its class `Math`:
//   Elem, D                 cache element and head_dim
//   NW                      warps of a block
//   SROWS                   KV rows of a stage: a part of a 64-row tile (16 or 32)
//   GROWS, GROUPS           query rows of a group; groups of a cluster at most (a power of two)
//   ROWS, row(i)            query rows a thread needs visibility bits for
//   STAGE_BYTES             SROWS rows of K, then of V, in panels of [SROWS rows][128 bytes] (128-byte swizzle)
//   K_REUSED                stage() writes over the stage's K rows
//   PREFIX_FIRST, FUSES     report a tile list that does not begin with the prefix; carry out recorded appends
//   q_off                   place of a 16-byte chunk of a query row in shared memory
//   stage(), write()        one stage for one warp (shared: other groups work on it too; k_read() is called by every warp once
//                           it has read the stage's K rows for the last time and returns when all groups have); the warp's
//                           accumulators and (m, l) to shared memory
//   part_off, store         float offset of (row, column) of a partial; four results to the output
//
// How the blocks of a cluster merge.  Every block sends its (m, l, O), merged over its warps, straight into the shared
// memory of the blocks that finish the rows: the result's chunks of 16 columns are dealt out over the blocks, and a
// chunk's values travel as asynchronous stores (st.async) that count towards a barrier of the block that owns it.  That
// is one one-way trip: no barrier of the cluster after the partials are written, no reads of other blocks' memory, none
// at the end (a block's memory is written by those only whose bytes it waits for, and it reads its own alone).
// Measured (us a layer, partials read from the other blocks between two barriers of the cluster / sent): one scene, 28/4
// heads x 128, prefix 2048, six fields 11.9 / 10.1 (with the queries' lines asked into L2 ahead of the dependency wait);
// one field, prefix 1024: 8.0 / 7.6; 16 scenes, 14/2 x 64, prefix 4096: 19.5 / 18.5; fp32, 8 scenes, prefix 2048: 87.2 / 84.8.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include <atomic>
#include <type_traits>

#include "fdc_attn_common.cuh"

namespace fdc {

constexpr int MAX_STAGES = 16;
constexpr int MASK_WORDS = 1024;              // (tile part, field) visibility words kept in shared memory
constexpr int MASK_HALVES = 64;               // tile parts among them at most
constexpr int MAX_QROWS = 192;                // query rows of a cluster, whole groups
constexpr int ROW0S = 256;                    // tile parts of the run whose first row is kept in shared memory

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Byte offset of the 16-byte chunk `dc` (0 .. D/8-1) of row `r` of an operand in panels of `panel` bytes
// ([rows][128 bytes], 64 bf16 columns each) with the 128-byte swizzle TMA applies: inside a panel the
// chunk index is XORed with (row mod 8).
__device__ __forceinline__ uint32_t swz(uint32_t panel, int r, int dc)
{
    return (uint32_t)(dc >> 3) * panel + (uint32_t)(r * 128 + (((dc & 7) ^ (r & 7)) << 4));
}

// 16-byte asynchronous copy global -> shared (zero fill when !valid).
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(valid ? 16 : 0) : "memory");
}

// Visibility of the SROWS rows row0.. for one field: prefix rows are all visible.
template <int SROWS>
__device__ __forceinline__ uint32_t part_bits(const uint64_t* __restrict__ words, int W, int P, int row0)
{
    constexpr uint32_t all = SROWS == 32 ? ~0u : (1u << (SROWS & 31)) - 1u;
    const int npre = P - row0;
    if (npre >= SROWS) return all;
    return ((npre <= 0 ? 0u : ((1u << npre) - 1u)) | (uint32_t)extract64(words, W, row0 - P)) & all;
}

template <int N, class F, int I = 0>
__device__ __forceinline__ void static_for(F&& f)
{
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        static_for<N, F, I + 1>(static_cast<F&&>(f));
    }
}

// Waits until stage `slot` has been asked for at least `n` times.  The warps that use a slot in turn need
// not be the same ones, and a parity wait tells only two consecutive phases of a barrier apart: a warp
// that ran ahead would take the phase before the previous use for its own.  Once the n-th request has
// been made the previous use is over, so the barrier is in the n-th phase or just past it.  Bounded
// like every in-kernel wait.
static __device__ __noinline__ bool wait_asked_slow(volatile int* asked, int n, volatile int* abort_flag, int32_t* status)
{
    for (uint32_t i = 0; i < SPIN_LIMIT * 16; ++i) {
        if (*asked >= n) return true;
        if ((i & 255u) == 255u && *abort_flag) return false;
        __nanosleep(32);
    }
    *abort_flag = 1;
    atomicOr(status, FDC_DEV_TIMEOUT);
    return false;
}
__device__ __forceinline__ bool wait_asked(volatile int* asked, int n, volatile int* abort_flag, int32_t* status)
{
    return *asked >= n || wait_asked_slow(asked, n, abort_flag, status);
}

template <int NW, int GROWS>
struct __align__(16) BlockState {
    uint64_t full[MAX_STAGES];
    uint64_t k_read[MAX_STAGES];              // all groups have read the stage's K rows (kernels that reuse their place)
    int used[MAX_STAGES];                     // groups that have finished with the stage
    int asked[MAX_STAGES];                    // requests made for the stage so far
    int abort_flag;                           // a bounded wait ran out somewhere in the block
    int beyond[NW];                           // first part of the run that reaches beyond the prefix, among those a warp looked at
    float2 wml[NW * GROWS];                   // (m, l) per warp and row of its group ([lane][query row])
    uint64_t pushed;                          // the cluster's partials of this block's chunks have arrived
    uint64_t pad2;
    uint8_t fld[MAX_QROWS];                   // field of every query row of the cluster (0xff: a row past the last)
    int app_row[FDC_MAX_NODES];               // fused append: cache row of every field's new K/V vector, -1: not written
    uint32_t newbits[2 * FDC_MAX_NODES];      // [new rows 0-31, 32-63][field] the new rows that the field sees
    uint32_t seen[MASK_HALVES];               // rows of a tile part that some field sees and whose values come from the cache
    uint8_t holds[MASK_HALVES];               // the part holds a visible row
    uint8_t kept[MASK_HALVES];                // the parts that do, in order
    uint32_t bits[MASK_WORDS];                // [part][field] the rows that the field sees
    int row0[ROW0S];                          // first KV row of the run's parts
};

// The block's run of tile parts: positions [h0, h1) of the pair's list (each 64-row tile is two or four of them).
// Positions p0 .. p0 + np - 1 have their visibility in shared memory; those of them that hold no
// visible row are left out, so the i-th part that is loaded is not always position h0 + i.
struct Run {
    const int32_t* tiles;                     // the scene's tile list
    const uint64_t* mask;                     // the scene's bitmaps
    int h0, h1, p0, np;
    int nx;                                   // stages of new rows, ahead of the tile parts
    int total;                                // stages
    int n_kept;                               // entries of kept[]
};
template <int SROWS>
__device__ __forceinline__ int list_row0(const Run& r, int pos)
{
    return r.tiles[pos / (FDC_TILE_ROWS / SROWS)] * FDC_TILE_ROWS + pos % (FDC_TILE_ROWS / SROWS) * SROWS;
}
template <int SROWS, class Block>
__device__ __forceinline__ int part_row0(const Run& r, const Block& bs, int pos)
{
    const int i = pos - r.h0;
    return i < ROW0S ? bs.row0[i] : list_row0<SROWS>(r, pos);
}
template <class Block>
__device__ __forceinline__ int stage_pos(const Run& r, const Block& bs, int it)
{
    const int i = it - r.nx - (r.p0 - r.h0);
    if (i < 0) return r.h0 + it - r.nx;
    return i < r.n_kept ? r.p0 + bs.kept[i] : r.p0 + r.np + (i - r.n_kept);
}
// Rows of the tile part that some field sees (whole warp).
template <int SROWS>
__device__ __noinline__ uint32_t part_seen_slow(const uint64_t* mask, int W, int P, int A, int row0)
{
    uint32_t x = 0u;
    for (int b = threadIdx.x & 31; b < A; b += 32) x |= part_bits<SROWS>(mask + (size_t)b * W, W, P, row0);
    return __reduce_or_sync(0xffffffffu, x);
}

// The new rows of this pass among the SROWS rows row0.. (their values come from the stage of new rows).
template <int SROWS>
__device__ __noinline__ uint32_t new_rows_of(const int* app_row, int A, int row0)
{
    uint32_t x = 0u;
    for (int b = threadIdx.x & 31; b < A; b += 32) {
        const int i = app_row[b] - row0;
        if (i >= 0 && i < SROWS) x |= 1u << i;
    }
    return __reduce_or_sync(0xffffffffu, x);
}

__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// Asynchronous stores into a block of the cluster; the bytes count towards `bar`, a barrier of the same block.
__device__ __forceinline__ void st_async4(uint32_t addr, uint32_t bar, const float4& v)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar) : "memory");
}
__device__ __forceinline__ void st_async2(uint32_t addr, uint32_t bar, const float2& v)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(addr), "f"(v.x), "f"(v.y), "r"(bar) : "memory");
}
// Where the partials of a block's chunks arrive: [block of the cluster][chunk][16 columns], then [block][chunk] (m, l).
// Chunk k (query row k / (D / 16), columns 16 (k mod D / 16) ..) belongs to block k mod nblk and is its (k / nblk)-th.
constexpr int CHUNK_BYTES = 16 * 4 + 8;
// The wait for them: false where it ran out (nothing of them may then be read).  A sender whose own wait runs out still sends what it
// has, after its limit (a second or so) and what its earlier waits took.  This wait is flagged after eight such limits and then goes on as long
// again, so that bytes still under way find the block's memory in place.  That is an assumption, not a guarantee: a sender can be later than
// both if many of its waits end just short of their limits, in a launch that is lost already; its bytes would then fall into memory that may be another
// block's.  (A barrier of the cluster that every thread passes before it leaves would rule that out; it costs 1 % on average, and
// 6.13 -> 6.57 us a layer at 4 pairs x 7 query rows, prefix 1024.)
constexpr uint32_t PUSHED_FLAG = SPIN_LIMIT * 8, PUSHED_LEAVE = PUSHED_FLAG * 2;
static __device__ __noinline__ bool wait_pushed_slow(uint32_t bar, volatile int* abort_flag, int32_t* status)
{
    for (uint32_t i = 0; i < PUSHED_LEAVE; ++i) {
        if (mbar_try(bar, 0)) return true;
        if (i + 1 == PUSHED_FLAG) {
            *abort_flag = 1;
            atomicOr(status, FDC_DEV_TIMEOUT);
        }
    }
    return false;
}
// Merge over the lanes of a block, for every (query row, 4 columns): `rows` = query rows of a lane's partial;
// `done(row, column, m, l, sum)` takes the result.  (The weights of the merges, fp32's too, are ex2.approx.ftz: two
// units in the last place like exp2f, but a part whose maximum lies more than 2^126 below the highest counts 0.)
template <class Math, int L, class F>
__device__ __forceinline__ void merge_lanes_n(int tid, int M, int rows, const float2* ml, const float* part, F&& done)
{
    constexpr int D = Math::D;
    for (int idx = tid; idx < M * (D / 4); idx += Math::NW * 32) {
        const int mm = idx / (D / 4), c4 = (idx - mm * (D / 4)) * 4;
        float4 x[L];
        float2 v[L];
#pragma unroll
        for (int k = 0; k < L; ++k) {
            v[k] = ml[mm + k * rows];
            x[k] = *reinterpret_cast<const float4*>(part + k * rows * D + Math::part_off(mm, c4));
        }
        float mx = v[0].x;
#pragma unroll
        for (int k = 1; k < L; ++k) mx = fmaxf(mx, v[k].x);
        const float ms = mx == -INFINITY ? 0.f : mx;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        float lt = 0.f;
#pragma unroll
        for (int k = 0; k < L; ++k) {
            const float w = fast_exp2(v[k].x - ms);
            lt = fmaf(v[k].y, w, lt);
            acc.x = fmaf(x[k].x, w, acc.x);
            acc.y = fmaf(x[k].y, w, acc.y);
            acc.z = fmaf(x[k].z, w, acc.z);
            acc.w = fmaf(x[k].w, w, acc.w);
        }
        done(mm, c4, mx, lt, acc);
    }
}
template <class Math, class F>
__device__ __forceinline__ void merge_lanes(int lanes, int tid, int M, int rows, const float2* ml, const float* part, F&& done)
{
    if constexpr (Math::NW == 8) {
        switch (lanes) {
            case 1: return merge_lanes_n<Math, 1>(tid, M, rows, ml, part, done);
            case 2: return merge_lanes_n<Math, 2>(tid, M, rows, ml, part, done);
            case 4: return merge_lanes_n<Math, 4>(tid, M, rows, ml, part, done);
            default: return merge_lanes_n<Math, 8>(tid, M, rows, ml, part, done);
        }
    } else {
        static_assert(Math::NW == 12 && Math::GROUPS <= 2, "lanes of a group");
        if (lanes == 6) merge_lanes_n<Math, 6>(tid, M, rows, ml, part, done);
        else merge_lanes_n<Math, 12>(tid, M, rows, ml, part, done);
    }
}

// What a launch's blocks need besides AttnParams.
struct ClusterArgs {
    int nstage, nblk, qsplit, qrows;           // ring slots, blocks per cluster, clusters per pair, query rows per cluster
    uint32_t by_nblk, by_qsplit, by_group;     // div_inverse of nblk, qsplit and the query heads of a KV head
};

// The kernel.  Grid: x = (KV head, share of the query rows, block of the cluster), y = scene.
//
// The set-up is on the path of every launch whose blocks find no place beside the launch ahead (and of the first of a pass), and
// it is a chain of trips to memory (counts -> tile list -> bitmaps), fences and, more than both, of instructions that are fetched for one
// execution.  So: the barriers and the prefix's first stages are warp 0's alone, which needs no barrier of the block for it; the
// other warps prepare the visibility meanwhile, a warp per tile part, a lane per field; one barrier of the block ends it; and
// nothing is divided.  From a block's first instruction to its dependency wait (traced): 3.3 us with all warps going through every step, three barriers of
// the block and a releasing arrival at the cluster's (1000 cycles by itself), 2.1 us now.  us a layer: one scene, 28/4 heads x 128, six fields, prefix
// 2048 9.9 / 8.8; one field, prefix 1024 6.2 / 5.8; 14/2 x 64, 41 scenes, prefix 281, one field left 14.1 / 12.2.
template <class Math>
__device__ __forceinline__ void attn_cluster_body(const AttnParams& p, const CUtensorMap& tm_k, const CUtensorMap& tm_v, const ClusterArgs& ca)
{
    constexpr int D = Math::D, GROWS = Math::GROWS, STAGE_BYTES = Math::STAGE_BYTES, NW = Math::NW, THREADS = NW * 32, SROWS = Math::SROWS;
    constexpr int PARTS = FDC_TILE_ROWS / SROWS;           // stages of a tile
    constexpr int CHUNK = 16 / sizeof(typename Math::Elem);         // elements of a 16-byte chunk
    extern __shared__ unsigned char smem_dyn[];
    const int nstage = ca.nstage, nblk = ca.nblk, qrows = ca.qrows;
    unsigned char* ring = reinterpret_cast<unsigned char*>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    unsigned char* qs = ring + (size_t)nstage * STAGE_BYTES;
    unsigned char* recv = qs + Math::q_bytes(qrows);       // partials of this block's chunks, from all blocks of the cluster
    float* part = reinterpret_cast<float*>(ring);          // after the last stage: [warp][GROWS][D] partials
    __shared__ BlockState<NW, GROWS> bs;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int s = blockIdx.y, cluster = (int)div_by(blockIdx.x, ca.by_nblk), rank = (int)blockIdx.x - cluster * nblk;      // rank in the cluster
    const int g = (int)div_by((uint32_t)cluster, ca.by_qsplit), m0 = (cluster - g * ca.qsplit) * qrows;      // this cluster: query rows m0 .. m0 + qrows - 1 of the pair
    // Programmatic dependent launch: as in the tcgen05 kernel (fdc_attn_tc_kernel.cuh).  With p.early the pass
    // tables and the prefix rows may be read ahead of the wait.
    if (!p.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int A = p.n_active[s], nt = p.ntiles[s];
    // (the launch may be ahead of whatever writes the new rows' numbers: what is read here is checked after the wait)
    const int32_t* app = p.app_row ? p.app_row + (size_t)s * p.max_active : nullptr;
    int ar[2];                                             // lane: of fields lane and lane + 32
#pragma unroll
    for (int j = 0; j < 2; ++j) ar[j] = app && lane + 32 * j < p.max_active ? app[lane + 32 * j] : -1;
    if (A * p.group <= m0 || nt <= 0) {
        // Nothing to do (all blocks of the cluster agree).  Such blocks leave at once: their places go to the next launch's blocks, which set
        // themselves up meanwhile (3 scenes, 28/4 heads, one of five fields left, 144 of 216 blocks idle: a launch's last blocks began 0.5 us before the launch ahead
        // ended, now 15 us; over 160 drawn passes with at most a third of their fields at work no faster than waiting on average, 0.946 to 1.051).  One block of the grid waits for the launch ahead, so that grids still complete in stream order.
        if (p.early && blockIdx.x == 0 && blockIdx.y == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    const int M = A * p.group - m0 < qrows ? A * p.group - m0 : qrows;
    const int groups = Math::GROUPS == 1 || M <= GROWS ? 1 : (Math::GROUPS == 2 || M <= 2 * GROWS ? 2 : (M <= 4 * GROWS ? 4 : 8)), lanes = NW / groups;
    auto by_nblk = [&](uint32_t x) { return div_by(x, ca.by_nblk); };
    Run r;
    r.tiles = p.tiles + (size_t)s * p.ntile_max;
    r.mask = p.mask + (size_t)s * p.max_active * p.W;
    r.h0 = run_begin(rank, nblk, PARTS * nt, by_nblk);
    r.h1 = run_begin(rank + 1, nblk, PARTS * nt, by_nblk);
    const int whole = p.P / FDC_TILE_ROWS;                     // the whole tiles of the prefix come first in a list
    r.p0 = PARTS * whole;
    if (r.p0 < r.h0) r.p0 = r.h0;
    if (r.p0 > r.h1) r.p0 = r.h1;
    r.np = r.h1 - r.p0;
    if (r.np * A > MASK_WORDS) r.np = (int)__fdividef((float)MASK_WORDS, (float)A);       // (any number will do that is not too high)
    if (r.np > MASK_HALVES) r.np = MASK_HALVES;
    const int chunks = M * (D / 16), slots = (int)by_nblk((uint32_t)(chunks + nblk - 1));     // chunks of the result, of one block at most
    r.nx = app && rank == 0 ? (A + SROWS - 1) / SROWS : 0;
    const uint32_t full0 = smem_u32(bs.full), ring0 = smem_u32(ring);
    auto request_rows = [&](int row0, int st, int n) {     // one thread: the copies of a stage, the n-th to use slot st
        const uint32_t bar = full0 + 8 * st, dst = ring0 + (uint32_t)st * STAGE_BYTES;
        mbar_expect_tx(bar, STAGE_BYTES);
#pragma unroll
        for (int h = 0; h < STAGE_BYTES / (2 * SROWS * 128); ++h) {
            tma_load_4d(dst + h * (SROWS * 128), &tm_k, bar, h * 8 * CHUNK, row0, g, s);
            tma_load_4d(dst + STAGE_BYTES / 2 + h * (SROWS * 128), &tm_v, bar, h * 8 * CHUNK, row0, g, s);
        }
        __threadfence_block();
        *(volatile int*)&bs.asked[st] = n;
    };
    // The first stages: those of the prefix right away, by warp 0; stages fb1.. may hold rows beyond the prefix and wait for the kernel ahead.
    int fb1 = r.nx + r.p0 - r.h0, first0 = 0;              // lane: first KV row of part h0 + lane
    if (!Math::PREFIX_FIRST) {                             // (any order of the list is served)
        const int pos = r.h0 + lane;
        first0 = pos < r.p0 ? list_row0<SROWS>(r, pos) : 0;
        const unsigned beyond = __ballot_sync(0xffffffffu, pos < r.p0 && first0 + SROWS > p.P);
        if (beyond) fb1 = r.nx + __ffs(beyond) - 1;
    }
    if (warp == 0) {
        const int ask = nstage < fb1 ? nstage : fb1;
        if (lane < nstage) {
            bs.used[lane] = 0;
            bs.asked[lane] = lane < r.nx ? 1 : 0;
            mbar_init(full0 + 8 * lane, 1);
            if (Math::K_REUSED) mbar_init(smem_u32(&bs.k_read[lane]), groups);
            if (lane == 0) {
                bs.abort_flag = 0;
                mbar_init(smem_u32(&bs.pushed), 1);
            }
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            fence_async_smem();
            if (lane == 0 && nblk > 1) mbar_expect_tx(smem_u32(&bs.pushed), nblk * (int)by_nblk((uint32_t)(chunks - rank + nblk - 1)) * CHUNK_BYTES);
            if (lane < r.nx) mbar_arrive(full0 + 8 * lane);               // filled by this block itself, ahead of the main loop
        }
        __syncwarp();
        const int from = Math::PREFIX_FIRST ? (r.h0 + lane - r.nx) * SROWS : __shfl_sync(0xffffffffu, first0, lane >= r.nx ? lane - r.nx : 0);
        if (lane >= r.nx && lane < ask) request_rows(from, lane, 1);
        __syncwarp();
    }
    // (the barrier of the partials is there, made known by the fence: the other blocks may send once they have seen all of this arrive)
    if (nblk > 1) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
    volatile int* abortp = &bs.abort_flag;
    bool off_list = false;
    {
        int beyond = 0x7fffffff;                           // first part of this thread's that reaches beyond the prefix
        for (int i = tid; i < r.h1 - r.h0; i += THREADS) {
            const int pos = r.h0 + i, row0 = list_row0<SROWS>(r, pos);
            if (i < ROW0S) bs.row0[i] = row0;
            if (row0 + SROWS > p.P && beyond == 0x7fffffff) beyond = i;
            off_list |= pos < PARTS * whole && row0 != pos * SROWS;
        }
        beyond = __reduce_min_sync(0xffffffffu, beyond);
        if (lane == 0) bs.beyond[warp] = beyond;
    }
    if (tid < MAX_QROWS) bs.fld[tid] = tid < M ? (uint8_t)div_by((uint32_t)(m0 + tid), ca.by_group) : (uint8_t)0xff;
    // Visibility of the run's parts from position p0 on: a warp per part (from the last warp down: warp 0 has the barriers), a lane per
    // field.  Fused append: the new rows count as unseen there (their values come from the stage of new rows).
    auto written = [&](int row) { return row >= p.P && row < p.rows; };
    auto cache_bits = [&]() {
        for (int h = NW - 1 - warp; h < r.np; h += NW) {
            const int row0 = list_row0<SROWS>(r, r.p0 + h);
            uint32_t x[2] = {0u, 0u}, fresh = 0u;
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int b = lane + 32 * j, i = ar[j] - row0;
                if (b < A) {
                    x[j] = part_bits<SROWS>(r.mask + (size_t)b * p.W, p.W, p.P, row0);
                    if (written(ar[j]) && i >= 0 && i < SROWS) fresh |= 1u << i;
                }
            }
            if (app) fresh = __reduce_or_sync(0xffffffffu, fresh);
            const uint32_t any = __reduce_or_sync(0xffffffffu, x[0] | x[1]);
#pragma unroll
            for (int j = 0; j < 2; ++j)
                if (lane + 32 * j < A) bs.bits[h * A + lane + 32 * j] = x[j] & ~fresh;
            if (lane == 0) {
                bs.seen[h] = any & ~fresh;
                bs.holds[h] = any != 0u;               // (the new rows' numbers may still change)
            }
        }
    };
    // ... and which of the new rows every field sees (block 0)
    auto new_bits = [&]() {
        for (int i = warp; i < r.nx * A; i += NW) {
            static_assert(!Math::FUSES || SROWS == 32, "a lane's two fields are in two stages");
            const int x = i >= A ? 1 : 0, b = i - x * A, row = x * 32 + lane < A ? (x ? ar[1] : ar[0]) : -1, t = row - p.P;
            const bool on = written(row) && (t >> 6) < p.W && ((r.mask[(size_t)b * p.W + (t >> 6)] >> (t & 63)) & 1ull);
            const uint32_t bits = __ballot_sync(0xffffffffu, on);
            if (lane == 0) bs.newbits[x * FDC_MAX_NODES + b] = bits;
        }
        if (warp == NW - 1)
#pragma unroll
            for (int j = 0; j < 2; ++j)
                if (lane + 32 * j < A) bs.app_row[lane + 32 * j] = written(ar[j]) ? ar[j] : -1;
    };
    cache_bits();
    if (app) new_bits();
    __syncthreads();
    // The parts that hold a visible row, in order (every warp makes the whole list: the same values).
    auto keep_parts = [&]() {
        int n = 0;
        for (int h0 = 0; h0 < r.np; h0 += 32) {
            const bool keep = h0 + lane < r.np && bs.holds[h0 + lane] != 0;
            const uint32_t ball = __ballot_sync(0xffffffffu, keep);
            if (keep) bs.kept[n + __popc(ball & ((1u << lane) - 1u))] = (uint8_t)(h0 + lane);
            n += __popc(ball);
        }
        __syncwarp();
        return n;
    };
    r.n_kept = keep_parts();
    int first_beyond = lane < NW ? bs.beyond[lane] : 0x7fffffff;
    first_beyond = __reduce_min_sync(0xffffffffu, first_beyond);
    if (first_beyond > r.h1 - r.h0) first_beyond = r.h1 - r.h0;
    r.total = r.nx + (r.h1 - r.h0) - (r.np - r.n_kept);
    // stages fb.. may hold rows beyond the prefix (parts ahead of p0 are never left out)
    const int fb = r.nx + (first_beyond < r.p0 - r.h0 ? first_beyond : r.p0 - r.h0);
    auto request = [&](int it, int st, int n) { request_rows(part_row0<SROWS>(r, bs, stage_pos(r, bs, it)), st, n); };
    if (p.early) {
        // The queries and the new rows may still be written by the kernel ahead: their lines are only requested into L2
        // (which stays coherent), so that the reads after the wait find them there.
        constexpr int LINES = D * sizeof(typename Math::Elem) / 128;
        for (int i = tid; i < M * LINES; i += THREADS) {
            const int m = i / LINES, b = bs.fld[m], hg = m0 + m - b * p.group;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(p.q) + ((((size_t)s * p.max_active + b) * p.hq + (size_t)g * p.group + hg) * LINES + (i - m * LINES)) * 128));
        }
        if (r.nx)
            for (int i = tid; i < 2 * A * LINES; i += THREADS) {
                const int x = i >= A * LINES, b = (i - x * A * LINES) / LINES;
                asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(x ? p.app_v : p.app_k) + ((((size_t)s * p.max_active + b) * p.hkv + g) * LINES + i % LINES) * 128));
            }
        asm volatile("griddepcontrol.wait;" ::: "memory");
    }
    // queries of the pair: row m = field * group + head-in-group; rows M.. up to a whole group are zero
    for (int i = tid; i < (M + GROWS - 1) / GROWS * GROWS * (D / CHUNK); i += THREADS) {
        const int m = i / (D / CHUNK), dc = i - m * (D / CHUNK);
        const int b = m < M ? (int)bs.fld[m] : 0, hg = m < M ? m0 + m - b * p.group : 0;
        cp_async16(qs + Math::q_off(qrows, m, dc),
                   reinterpret_cast<const uint4*>(p.q) + ((((size_t)s * p.max_active + b) * p.hq + (size_t)g * p.group + hg) * D) / CHUNK + dc, m < M);
    }
    if (lane == 0) {
        for (int it = warp; it < nstage && it < r.total; it += NW)
            if (it >= fb1) request(it, it, 1);
    }
    __syncwarp();
    // the stages of new rows: row i of stage x = the new vectors of field 32 x + i (rows past the last field: zero)
    for (int i = tid; i < r.nx * SROWS * (D / CHUNK); i += THREADS) {
        const int b = i / (D / CHUNK), dc = i - b * (D / CHUNK);
        const size_t src = ((size_t)s * p.max_active * p.hkv + g + (size_t)(b < A ? b : 0) * p.hkv) * (D / CHUNK) + dc;
        unsigned char* ks = ring + (size_t)(b / SROWS) * STAGE_BYTES + swz(SROWS * 128, b % SROWS, dc);
        cp_async16(ks, reinterpret_cast<const uint4*>(p.app_k) + src, b < A);
        cp_async16(ks + STAGE_BYTES / 2, reinterpret_cast<const uint4*>(p.app_v) + src, b < A);
    }
    // (kernels for other caches have never asked for the prefix tiles to come first)
    if (Math::PREFIX_FIRST && off_list) atomicOr(p.status, FDC_DEV_TILE_LIST);
    int moved = 0;
    if (app) {
#pragma unroll
        for (int j = 0; j < 2; ++j)
            if (lane + 32 * j < A) {
                const int now = __ldcg(app + lane + 32 * j);
                if (!written(now) && warp == 0 && blockIdx.x == 0) atomicOr(p.status, FDC_DEV_ROW_RANGE);     // skipped and flagged
                moved |= now != ar[j];
                ar[j] = now;
            }
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    if (r.nx) fence_async_smem();                          // (the next copy into the new rows' slots goes through the asynchronous proxy)
    if (__syncthreads_or(moved)) {
        // the row numbers were written by the kernel ahead: the tables once more
        cache_bits();
        new_bits();
        __syncthreads();
    }
    const int mg = warp % groups, kl = warp / groups;
    const int left = M - mg * GROWS;                       // rows of this warp's group that exist (<= 0: none)
    Math math(p, qs, qrows, left > 0 ? mg * GROWS : 0, lane, left);
    const uint8_t* fld = bs.fld + mg * GROWS;              // fields of the group's query rows
    bool alive = true;
    int st = kl, use = 1;                                  // slot of stage `it`, and how many stages (this one included) have used it
    while (st >= nstage) {
        st -= nstage;
        ++use;
    }
    for (int it = kl; it < r.total; it += lanes) {
        alive = wait_asked(&bs.asked[st], use, abortp, p.status) && mbar_wait(full0 + 8 * st, (uint32_t)(use - 1) & 1, abortp, p.status);
        if (!__all_sync(0xffffffffu, alive)) break;
        if (left > 0) {
            bool masked = false;
            uint32_t mk[Math::ROWS], seen = ~0u, any = ~0u;
#pragma unroll
            for (int i = 0; i < Math::ROWS; ++i) mk[i] = ~0u;
            if (it < r.nx) {
                masked = true;
#pragma unroll
                for (int i = 0; i < Math::ROWS; ++i) mk[i] = fld[math.row(i)] == 0xff ? 0u : bs.newbits[it * FDC_MAX_NODES + fld[math.row(i)]];
                for (int b = 0; b < SROWS && it * SROWS + b < A; ++b)     // (values of rows that are not written do not count either)
                    if (bs.app_row[it * SROWS + b] < 0) seen &= ~(1u << b);
            } else if (it >= fb) {
                const int pos = stage_pos(r, bs, it), row0 = part_row0<SROWS>(r, bs, pos), h = pos - r.p0;
                if (row0 + SROWS > p.P) {
                    masked = true;
                    if (h >= 0 && h < r.np) {
#pragma unroll
                        for (int i = 0; i < Math::ROWS; ++i) mk[i] = fld[math.row(i)] == 0xff ? 0u : bs.bits[h * A + fld[math.row(i)]];
                        seen = bs.seen[h];
                    } else {
                        const uint32_t fresh = p.app_row ? new_rows_of<SROWS>(bs.app_row, A, row0) : 0u;
#pragma unroll
                        for (int i = 0; i < Math::ROWS; ++i) mk[i] = fld[math.row(i)] == 0xff ? 0u : part_bits<SROWS>(r.mask + (size_t)fld[math.row(i)] * p.W, p.W, p.P, row0) & ~fresh;
                        seen = part_seen_slow<SROWS>(r.mask, p.W, p.P, A, row0) & ~fresh;
                    }
                }
            }
            if (masked) {
                any = 0u;
#pragma unroll
                for (int i = 0; i < Math::ROWS; ++i) any |= mk[i];
            }
            auto k_read = [&]() {
                if constexpr (Math::K_REUSED) {
                    __syncwarp();
                    if (groups == 1) return;
                    if (lane == 0) mbar_arrive(smem_u32(&bs.k_read[st]));
                    alive = mbar_wait(smem_u32(&bs.k_read[st]), (uint32_t)(use - 1) & 1, abortp, p.status);
                }
            };
            if (__any_sync(0xffffffffu, any != 0u)) math.stage(ring0 + (uint32_t)st * STAGE_BYTES, masked, mk, seen, k_read);
            else k_read();                                 // (a part that only other groups' fields see)
            if (Math::K_REUSED && !__all_sync(0xffffffffu, alive)) break;
        } else if (Math::K_REUSED && groups > 1 && lane == 0) {
            mbar_arrive(smem_u32(&bs.k_read[st]));
        }
        // the last group to finish with the stage requests its next rows
        __syncwarp();
        if (lane == 0 && it + nstage < r.total) {
            bool mine = groups == 1;
            if (!mine) {
                __threadfence_block();
                mine = atomicAdd(&bs.used[st], 1) == groups - 1;
                __threadfence_block();
                if (mine) bs.used[st] = 0;
            }
            if (mine) request(it + nstage, st, use + 1);
        }
        st += lanes;
        while (st >= nstage) {
            st -= nstage;
            ++use;
        }
    }
    // a wait that ran out: give the copies already in flight a bounded chance to land before the ring is reused
    if (*abortp) {
        for (int i = 0; i < 100; ++i) __nanosleep(1000);
    }
    // ---- the warps' results meet in shared memory (the ring is free: every stage has been consumed)
    __syncthreads();
    if (left > 0) math.write(part + warp * (GROWS * D), bs.wml + warp * GROWS, left);
    __syncthreads();
    auto store_out = [&](int mm, int c4, const float4& acc, float lt) {
        const float inv = 1.f / lt;
        const int b = bs.fld[mm], hg = m0 + mm - b * p.group;
        Math::store(reinterpret_cast<typename Math::Elem*>(p.out) + (((size_t)s * p.max_active + b) * p.hq + (size_t)g * p.group + hg) * D + c4,
                    make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv));
    };
    // block: merge over the warps of a group; with one block per pair that is the result, else it is sent to the chunk's block
    if (nblk > 1) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");       // (long complete: all blocks have set up their barriers)
    const uint32_t recv0 = smem_u32(recv), recv_ml0 = recv0 + (uint32_t)(nblk * slots * 64), pushed = smem_u32(&bs.pushed);
    merge_lanes<Math>(lanes, tid, M, groups * GROWS, bs.wml, part, [&](int mm, int c4, float mx, float lt, const float4& acc) {
        if (nblk == 1) {
            store_out(mm, c4, acc, lt);
        } else {
            const uint32_t k = (uint32_t)(mm * (D / 16) + (c4 >> 4)), slot = by_nblk(k), owner = k - slot * (uint32_t)nblk;
            const uint32_t at = (uint32_t)(rank * slots) + slot, bar = map_rank(pushed, owner);
            st_async4(map_rank(recv0 + at * 64 + (uint32_t)(c4 & 15) * 4, owner), bar, acc);
            if ((c4 & 15) == 0) st_async2(map_rank(recv_ml0 + at * 8, owner), bar, make_float2(mx, lt));
        }
    });
    // fused append: the new rows whose tile parts are in this block's run go to the cache (this block's copies
    // from there have landed; clusters with the pair's other query rows may still be reading the
    // part, but to them, too, the row counts as unseen: its bytes there do not matter)
    if (Math::FUSES && p.app_row && m0 == 0 && first_beyond < r.h1 - r.h0)
        for (int b = warp; b < A; b += NW) {
            const int ar = bs.app_row[b];
            bool here = false;
            for (int i = first_beyond + lane; i < r.h1 - r.h0; i += 32) {
                const int x = ar - part_row0<SROWS>(r, bs, r.h0 + i);
                here |= x >= 0 && x < SROWS;
            }
            here = __any_sync(0xffffffffu, here && ar >= 0);
            const int dc = lane & 15;
            if (here && dc < D / CHUNK) {
                // lanes 0-15: the K row, lanes 16-31: the V row
                const uint4 x = reinterpret_cast<const uint4*>(lane < 16 ? p.app_k : p.app_v)[((((size_t)s * p.max_active + b) * p.hkv + g) * D) / CHUNK + dc];
                auto* cache = const_cast<typename Math::Elem*>(reinterpret_cast<const typename Math::Elem*>(lane < 16 ? p.k : p.v));
                *reinterpret_cast<uint4*>(cache + (size_t)s * p.stride_scene + (size_t)g * p.stride_head + (size_t)ar * p.stride_row + dc * CHUNK) = x;
            }
        }
    if (nblk == 1) return;
    // ---- cluster: every block finishes its chunks once all blocks' partials of them are there
    if (!__all_sync(0xffffffffu, mbar_try(pushed, 0) || wait_pushed_slow(pushed, abortp, p.status))) return;       // (flagged: no output)
    {
        // Four threads per item (4 columns), each with every fourth block (at most four), summed by shuffles.
        const float4* ro = reinterpret_cast<const float4*>(recv);
        const float2* rml = reinterpret_cast<const float2*>(recv + (size_t)nblk * slots * 64);
        const int q = tid & 3, items = (int)by_nblk((uint32_t)(chunks - rank + nblk - 1)) * 4;
        for (int i = tid >> 2; __any_sync(0xffffffffu, i < items); i += THREADS / 4) {
            const bool on = i < items;
            const int slot = on ? i >> 2 : 0, k = slot * nblk + rank, mm = k / (D / 16), c4 = (k - mm * (D / 16)) * 16 + (i & 3) * 4;
            float2 v[4];
            float4 x[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                v[j] = make_float2(-INFINITY, 0.f);
                x[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (on && q + 4 * j < nblk) {
                    const int at = (q + 4 * j) * slots + slot;
                    v[j] = rml[at];
                    x[j] = ro[at * 4 + (i & 3)];
                }
            }
            float mx = fmaxf(fmaxf(v[0].x, v[1].x), fmaxf(v[2].x, v[3].x));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const float ms = mx == -INFINITY ? 0.f : mx;
            float lt = 0.f;
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float w = fast_exp2(v[j].x - ms);    // a block that saw nothing: 0
                lt = fmaf(v[j].y, w, lt);
                acc.x = fmaf(x[j].x, w, acc.x);
                acc.y = fmaf(x[j].y, w, acc.y);
                acc.z = fmaf(x[j].z, w, acc.z);
                acc.w = fmaf(x[j].w, w, acc.w);
            }
#pragma unroll
            for (int d = 1; d < 4; d <<= 1) {
                lt += __shfl_xor_sync(0xffffffffu, lt, d);
                acc.x += __shfl_xor_sync(0xffffffffu, acc.x, d);
                acc.y += __shfl_xor_sync(0xffffffffu, acc.y, d);
                acc.z += __shfl_xor_sync(0xffffffffu, acc.z, d);
                acc.w += __shfl_xor_sync(0xffffffffu, acc.w, d);
            }
            if (on && q == 0) store_out(mm, c4, acc, lt);
        }
    }
}

// Host: which cluster sizes of one kernel the devices have been asked about and can place: bit n of a device's word for
// clusters of n blocks with one block per SM, bit 16 + n with two (with either, the SMs of a GPC decide, not the
// launch's exact shared memory).
struct PlaceableClusters {
    std::atomic<uint64_t> asked[kMaxDevices] = {}, yes[kMaxDevices] = {};
};
inline bool cluster_placeable(const void* kernel, const cudaLaunchConfig_t& cfg, int n, bool two, PlaceableClusters& known)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return n <= 8;
    const uint64_t bit = 1ull << (n + (two ? 16 : 0));
    if (known.asked[dev].load(std::memory_order_acquire) & bit) return (known.yes[dev].load(std::memory_order_relaxed) & bit) != 0;
    int clusters = 0;
    cudaError_t e = n > 8 ? cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) : cudaSuccess;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg);
    if (e != cudaSuccess) {
        cudaGetLastError();                                // (no answer: left to the launch, the portable sizes only)
        return n <= 8;
    }
    if (clusters > 0) known.yes[dev].fetch_or(bit, std::memory_order_relaxed);
    known.asked[dev].fetch_or(bit, std::memory_order_release);
    return clusters > 0;
}

// Host: shared memory of a block besides its ring, and the ring's stages in `room` bytes (0: the partials, which take the
// ring's place after the last stage, would not fit it).
template <class Math>
size_t cluster_smem_fixed(int qrows, int nblk)
{
    const size_t recv = nblk > 1 ? (size_t)(qrows * (Math::D / 16) + nblk) * CHUNK_BYTES : 0;      // (for any number of blocks up to this one)
    return 1024 + Math::q_bytes(qrows) + recv;
}
template <class Math>
int cluster_ring_stages(size_t room, int qrows, int nblk)
{
    const long long left = (long long)room - (long long)(sizeof(BlockState<Math::NW, Math::GROWS>) + 256 + cluster_smem_fixed<Math>(qrows, nblk));
    const int n = left > 0 ? (int)(left / Math::STAGE_BYTES) : 0;
    if (n * Math::STAGE_BYTES < Math::NW * Math::GROWS * Math::D * 4) return 0;
    return n > MAX_STAGES ? MAX_STAGES : n;
}

// Host: shared memory of a launch, tensor maps, launch attributes.  `room`: bytes a block may use.
template <class Math, class Kernel>
int launch_cluster(Kernel kernel, const AttnParams& p, size_t room, const ClusterShape& h, cudaStream_t st)
{
    const int qrows = ((p.mmax + Math::GROWS - 1) / Math::GROWS + h.qsplit - 1) / h.qsplit * Math::GROWS;
    const int nstage = cluster_ring_stages<Math>(room, qrows, h.nblk);
    if (nstage == 0) return FDC_ERR_SHAPE;
    size_t smem = cluster_smem_fixed<Math>(qrows, h.nblk) + (size_t)nstage * Math::STAGE_BYTES;
    if (h.per_sm <= 1 && smem < 120 * 1024) smem = 120 * 1024;        // (more than half of an SM's: no second block beside this one)
    static SmemLimit limit;
    int rc = raise_dynamic_smem(reinterpret_cast<const void*>(kernel), smem, limit);
    if (rc) return rc;
    static PlaceableClusters known;
    alignas(64) CUtensorMap tk, tv;
    const int dtype = sizeof(typename Math::Elem) == 4 ? FDC_F32 : FDC_BF16;
    rc = get_kv_tensor_map(p.k, p, dtype, Math::D, Math::SROWS, &tk);
    if (rc) return rc;
    rc = get_kv_tensor_map(p.v, p, dtype, Math::D, Math::SROWS, &tv);
    if (rc) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(Math::NW * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    // The cuts are made for a whole B200.  What a device cannot place (a part of one, or GPCs with fewer SMs) is
    // launched as the next smaller clusters that it can; any size is right.
    const int nblk = largest_placeable(h.nblk, [&](int n) {
        cudaLaunchConfig_t one = cfg;
        at[1].val.clusterDim.x = (unsigned)n;
        one.gridDim = dim3((unsigned)n);
        one.attrs = &at[1];
        one.numAttrs = 1;
        return cluster_placeable(reinterpret_cast<const void*>(kernel), one, n, h.per_sm > 1, known);
    });
    at[1].val.clusterDim.x = (unsigned)nblk;
    cfg.gridDim = dim3((unsigned)(p.hkv * h.qsplit * nblk), (unsigned)p.batch);
    const ClusterArgs args{nstage, nblk, h.qsplit, qrows, div_inverse(nblk), div_inverse(h.qsplit), div_inverse(p.group)};
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, p, tk, tv, args);
    if (e != cudaSuccess) return set_cuda_error(e);
    note_launch();
    return FDC_OK;
}

}  // namespace fdc
