// Attention of one (scene, KV head) pair by ONE thread-block cluster (bf16, head_dim 64 or 128): split,
// softmax and merge in a single kernel, the partial results exchanged through distributed shared
// memory instead of a workspace.
//
// What bounds it.  A pass of one or a few scenes moves a few MB per layer: streaming them takes 1 to
// 5 us, and the rest of a layer's time is a chain of latencies (dependency wait -> queries -> scores
// -> softmax -> output -> merge -> end of the grid).  This kernel is made for a short chain: no TMEM, no
// arrival counters, no partials in global memory, no second kernel and no split table.  The blocks
// of a pair take equal runs of its 32-row half tiles; everything of the prefix that fits the ring is
// requested before the dependency wait; the merge is two trips inside the cluster.  The tensor work
// is small here (a pair has 1 to 128 query rows), so it is done by mma.sync from registers, which
// needs no hand-over between issuing thread, tensor memory and softmax threads.
//
// Sec. 3.3: all queries of a pair (parallel fields x GQA heads) share ONE read of its KV rows (one
// per cluster where the query rows are cut, see pick_cluster).
//
// Measured (a layer, graphs of whole passes, against the kernels that served these shapes before): 1 scene, 28/4
// heads x 128, prefix 1024, one field: 14.6 -> 8.0 us; prefix 2048, six fields: 19.3 -> 11.9; 1 scene, 14/2 heads x
// 64, prefix 1531, six fields, append apart: 56.2 -> 16.1; 16 scenes, 14/2 x 64, prefix 4096: 56.4 -> 19.4.
//
// Block = 8 warps, two blocks per SM (128 registers a thread: the accumulators of 16 query rows take
// half of them).  A stage is 32 KV rows of K and V (TMA, 128-byte swizzle).  The query rows form 1, 2, 4
// or 8 groups of 16; the 8, 4, 2 or 1 warps of a group take its stages in turn, each with an online
// softmax of its own (running maximum, fp32 accumulators).  There is no producer warp: the warp that is
// the last to have used a stage requests the stage's next rows.
//   S = Q K^T, Eq. 1 by select from the fields' bitmaps, P (bf16), O += P V, and the softmax denominators
//   as P times ones (the same rounded values that meet V).
// Beyond the prefix, rows that no field may see can hold anything (NaN included), and 0 * NaN must not reach
// the accumulator: their V values are cleared in the registers on the way to the multiplication.
// Half tiles without any visible row are not loaded at all.
// Fused append: the pass's new K/V rows are a stage of their own, filled straight from k_new / v_new by the
// first block of the cluster; in the stages of the cache the same rows count as unseen.  The block whose
// run holds a row's half tile writes it to the cache after its last stage, while it waits for the cluster.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <atomic>
#include <cmath>
#include <mutex>
#include <type_traits>
#include <vector>

#include "fdc_attn_common.cuh"

using namespace fdc;

namespace {

constexpr int NW = 8;                         // warps
constexpr int THREADS = NW * 32;
constexpr int SROWS = 32;                     // KV rows per stage (half a tile)
constexpr int GROWS = 16;                     // query rows of a group
constexpr int MAX_STAGES = 16;
constexpr int MASK_WORDS = 1024;              // (half tile, field) visibility words kept in shared memory
constexpr int MASK_HALVES = 64;               // half tiles among them at most
constexpr int ROW0S = 256;                    // half tiles of the run whose first row is kept in shared memory

template <int OFF>
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4 + %5];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr), "n"(OFF) : "memory");
}
template <int OFF>
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4 + %5];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr), "n"(OFF) : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
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

// Visibility of the 32 rows row0.. for one field: prefix rows are all visible.
__device__ __forceinline__ uint32_t half_bits(const uint64_t* __restrict__ words, int W, int P, int row0)
{
    const int npre = P - row0;
    if (npre >= 32) return ~0u;
    return (npre <= 0 ? 0u : ((1u << npre) - 1u)) | (uint32_t)extract64(words, W, row0 - P);
}

template <int N, class F, int I = 0>
__device__ __forceinline__ void static_for(F&& f)
{
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        static_for<N, F, I + 1>(static_cast<F&&>(f));
    }
}

// One stage (32 KV rows) for one warp (16 query rows).  The swizzled chunk of a fragment differs between the
// steps of an operand by an XOR of address bits 5 and 6 only, everything else is a constant offset: two
// to four addresses per operand serve all its loads.
//   ka, qa  lane addresses of K (rows 0-7, chunks 0-3) and Q (chunks 0, 1);  va  of V (rows 0-15, chunks 0, 1)
template <int D>
__device__ __forceinline__ void process_stage(const uint32_t ka, const uint32_t va, const uint32_t qa, const uint32_t qpanel,
                                              float (&o)[D / 8][4], float (&l)[4], float (&m)[2], const bool masked, const uint32_t mk0,
                                              const uint32_t mk1, const uint32_t seen, const float c, const int lane)
{
    constexpr int NT = SROWS / 8;
    constexpr int panel = SROWS * 128;
    float s[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
    // S = Q K^T (the queries' fragments come from shared memory every time: registers hold the accumulators)
    static_for<D / 32>([&](auto KP) {
        constexpr int kp = KP;                             // 32 columns: chunks 4 kp .. 4 kp + 3
        uint32_t q[2][4], b[NT][4];
        const uint32_t qk = qa + (kp >> 1) * qpanel;
        ldsm_x4<0>(qk ^ ((kp & 1) * 64), q[0]);
        ldsm_x4<0>(qk ^ ((kp & 1) * 64 + 32), q[1]);
        static_for<NT>([&](auto N) { ldsm_x4<(kp >> 1) * panel + N * 1024>(ka ^ ((kp & 1) * 64), b[N]); });
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) mma_bf16(s[nt], q[0], b[nt][0], b[nt][1]);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) mma_bf16(s[nt], q[1], b[nt][2], b[nt][3]);
    });
    if (masked) {
        const int cb = 2 * (lane & 3);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const int col = nt * 8 + cb;
            if (!((mk0 >> col) & 1)) s[nt][0] = -INFINITY;
            if (!((mk0 >> (col + 1)) & 1)) s[nt][1] = -INFINITY;
            if (!((mk1 >> col) & 1)) s[nt][2] = -INFINITY;
            if (!((mk1 >> (col + 1)) & 1)) s[nt][3] = -INFINITY;
        }
    }
    // online softmax (scores in raw units; c = scale * log2 e is folded into the exponent)
    float x0 = -INFINITY, x1 = -INFINITY;
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        x0 = fmaxf(x0, fmaxf(s[nt][0], s[nt][1]));
        x1 = fmaxf(x1, fmaxf(s[nt][2], s[nt][3]));
    }
    x0 = fmaxf(x0, __shfl_xor_sync(0xffffffffu, x0, 1));
    x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, 1));
    x0 = fmaxf(x0, __shfl_xor_sync(0xffffffffu, x0, 2));
    x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, 2));
    const float n0 = fmaxf(m[0], x0), n1 = fmaxf(m[1], x1);
    const float r0 = n0 == -INFINITY ? 0.f : n0 * c;                   // a row that has seen nothing yet
    const float r1 = n1 == -INFINITY ? 0.f : n1 * c;
    // the running maxima settle after a few stages: rescale only when one of them moved
    if (__any_sync(0xffffffffu, (n0 != m[0]) || (n1 != m[1]))) {
        const float a0 = fast_exp2(m[0] * c - r0), a1 = fast_exp2(m[1] * c - r1);
        l[0] *= a0;
        l[2] *= a1;
#pragma unroll
        for (int n = 0; n < D / 8; ++n) {
            o[n][0] *= a0;
            o[n][1] *= a0;
            o[n][2] *= a1;
            o[n][3] *= a1;
        }
        m[0] = n0;
        m[1] = n1;
    }
    uint32_t pa[SROWS / 16][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        pa[nt >> 1][(nt & 1) * 2 + 0] = pack_bf16(fast_exp2(fmaf(s[nt][0], c, -r0)), fast_exp2(fmaf(s[nt][1], c, -r0)));
        pa[nt >> 1][(nt & 1) * 2 + 1] = pack_bf16(fast_exp2(fmaf(s[nt][2], c, -r1)), fast_exp2(fmaf(s[nt][3], c, -r1)));
    }
    // O += P V, l += P 1
    static_for<SROWS / 16>([&](auto KK) {
        constexpr int kk = KK;
        mma_bf16(l, pa[kk], 0x3F803F80u, 0x3F803F80u);
        // rows of this thread's V fragments that nobody sees: cleared
        const uint32_t two = seen >> (kk * 16 + 2 * (lane & 3));
        const uint32_t z0 = ((two & 1u) ? 0xffffu : 0u) | ((two & 2u) ? 0xffff0000u : 0u);
        const uint32_t z1 = ((two & 0x100u) ? 0xffffu : 0u) | ((two & 0x200u) ? 0xffff0000u : 0u);
        static_for<D / 64>([&](auto N4) {
            uint32_t b[4][4];
            static_for<4>([&](auto J) { ldsm_x4_t<N4 * panel + kk * 2048>(va ^ (J * 32), b[J]); });
            if (masked) {                                              // (uniform)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    b[j][0] &= z0;
                    b[j][1] &= z1;
                    b[j][2] &= z0;
                    b[j][3] &= z1;
                }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                mma_bf16(o[8 * N4 + 2 * j], pa[kk], b[j][0], b[j][1]);
                mma_bf16(o[8 * N4 + 2 * j + 1], pa[kk], b[j][2], b[j][3]);
            }
        });
    });
}

// Waits until stage `slot` has been asked for at least `n` times.  The warps that use a slot in turn need
// not be the same ones, and a parity wait tells only two consecutive phases of a barrier apart: a warp
// that ran ahead would take the phase before the previous use for its own.  Once the n-th request has
// been made the previous use is over, so the barrier is in the n-th phase or just past it.  Bounded
// like every in-kernel wait.
__device__ __noinline__ bool wait_asked_slow(volatile int* asked, int n, volatile int* abort_flag, int32_t* status)
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

struct __align__(16) BlockState {
    uint64_t full[MAX_STAGES];
    int used[MAX_STAGES];                     // groups that have finished with the stage
    int asked[MAX_STAGES];                    // requests made for the stage so far
    int abort_flag;                           // a bounded wait ran out somewhere in the block
    int first_beyond;                         // first half tile of the run that reaches beyond the prefix
    int n_kept;                               // entries of kept[]
    int pad;
    float2 wml[NW * GROWS];                   // (m, l) per warp and row of its group ([lane][query row])
    float2 cml[128];                          // (m, l) of the block per query row
    int app_row[FDC_MAX_NODES];               // fused append: cache row of every field's new K/V vector, -1: not written
    uint32_t newbits[2 * FDC_MAX_NODES];      // [new rows 0-31, 32-63][field] the new rows that the field sees
    uint32_t seen[MASK_HALVES];               // rows of a half tile that some field sees
    uint8_t kept[MASK_HALVES];                // those of them that hold a visible row, in order
    uint32_t bits[MASK_WORDS];                // [half tile][field] the rows that the field sees
    int row0[ROW0S];                          // first KV row of the run's half tiles
};

// The block's run of half tiles: positions [h0, h1) of the pair's list (64-row tile i = positions 2i, 2i + 1).
// Positions p0 .. p0 + np - 1 have their visibility in shared memory; those of them that hold no
// visible row are left out, so the i-th half tile that is loaded is not always position h0 + i.
struct Run {
    const int32_t* tiles;                     // the scene's tile list
    const uint64_t* mask;                     // the scene's bitmaps
    int h0, h1, p0, np;
    int nx;                                   // stages of new rows, ahead of the half tiles
    int total;                                // stages
};
__device__ __forceinline__ int half_row0(const Run& r, const BlockState& bs, int pos)
{
    const int i = pos - r.h0;
    return i < ROW0S ? bs.row0[i] : r.tiles[pos >> 1] * FDC_TILE_ROWS + (pos & 1) * SROWS;
}
__device__ __forceinline__ int stage_pos(const Run& r, const BlockState& bs, int it)
{
    const int i = it - r.nx - (r.p0 - r.h0);
    if (i < 0) return r.h0 + it - r.nx;
    return i < bs.n_kept ? r.p0 + bs.kept[i] : r.p0 + r.np + (i - bs.n_kept);
}
// Rows of the half tile that some field sees (whole warp).
__device__ __noinline__ uint32_t half_seen_slow(const uint64_t* mask, int W, int P, int A, int row0)
{
    uint32_t x = 0u;
    for (int b = threadIdx.x & 31; b < A; b += 32) x |= half_bits(mask + (size_t)b * W, W, P, row0);
    return __reduce_or_sync(0xffffffffu, x);
}

// The new rows of this pass among the 32 rows row0.. (their values come from the stage of new rows).
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
__device__ __forceinline__ float2 ld_cluster2(uint32_t addr)
{
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float4 ld_cluster4(uint32_t addr)
{
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
// Float offset of (row, column) of a partial [rows][D]: the columns' groups of 8 are permuted by the row
// so that the accumulator fragments' stores spread over the banks.
template <int D>
__device__ __forceinline__ int part_off(int row, int col) { return row * D + (col ^ ((row & 3) << 3)); }

// Merge over the lanes of a block, for every (query row, 4 columns): `rows` = query rows of a lane's partial;
// `done(row, column, m, l, sum)` takes the result.
template <int D, int L, class F>
__device__ __forceinline__ void merge_lanes_n(int tid, int M, int rows, const float2* ml, const float* part, F&& done)
{
    for (int idx = tid; idx < M * (D / 4); idx += THREADS) {
        const int mm = idx / (D / 4), c4 = (idx - mm * (D / 4)) * 4;
        float4 x[L];
        float2 v[L];
#pragma unroll
        for (int k = 0; k < L; ++k) {
            v[k] = ml[mm + k * rows];
            x[k] = *reinterpret_cast<const float4*>(part + k * rows * D + part_off<D>(mm, c4));
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
template <int D, class F>
__device__ __forceinline__ void merge_lanes(int lanes, int tid, int M, int rows, const float2* ml, const float* part, F&& done)
{
    switch (lanes) {
        case 1: merge_lanes_n<D, 1>(tid, M, rows, ml, part, done); break;
        case 2: merge_lanes_n<D, 2>(tid, M, rows, ml, part, done); break;
        case 4: merge_lanes_n<D, 4>(tid, M, rows, ml, part, done); break;
        default: merge_lanes_n<D, 8>(tid, M, rows, ml, part, done); break;
    }
}

template <int D>
__global__ void __launch_bounds__(THREADS, 2)
attn_cluster_kernel(const __grid_constant__ AttnParams p, const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                    const int nstage, const int nblk, const int qsplit, const int qrows)
{
    constexpr int STAGE_BYTES = 2 * SROWS * D * 2;         // K rows + V rows
    extern __shared__ unsigned char smem_dyn[];
    unsigned char* ring = reinterpret_cast<unsigned char*>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    unsigned char* qs = ring + (size_t)nstage * STAGE_BYTES;
    const uint32_t qpanel = (uint32_t)qrows * 128;
    float* part = reinterpret_cast<float*>(ring);          // after the last stage: [warp][16][D] partials
    __shared__ BlockState bs;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = blockIdx.x % nblk;                    // = rank in the cluster (the grid is cut into runs of nblk blocks)
    const int cluster = blockIdx.x / nblk;
    const int pair = cluster / qsplit, m0 = (cluster - pair * qsplit) * qrows;      // this cluster: query rows m0 .. m0 + qrows - 1 of the pair
    const int s = pair / p.hkv, g = pair - s * p.hkv;
    // Programmatic dependent launch: as in the tcgen05 kernel (fdc_attn_tc_kernel.cuh).  With p.early the pass
    // tables and the prefix rows may be read ahead of the wait; every thread passes the wait.
    if (!p.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int A = p.n_active[s], nt = p.ntiles[s];
    if (A * p.group <= m0 || nt <= 0) {                    // nothing to do (all blocks of the cluster agree)
        if (p.early) asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    const int M = A * p.group - m0 < qrows ? A * p.group - m0 : qrows;
    const int groups = M <= GROWS ? 1 : (M <= 2 * GROWS ? 2 : (M <= 4 * GROWS ? 4 : 8)), lanes = NW / groups;
    Run r;
    r.tiles = p.tiles + (size_t)s * p.ntile_max;
    r.mask = p.mask + (size_t)s * p.max_active * p.W;
    r.h0 = (int)((long long)rank * 2 * nt / nblk);
    r.h1 = (int)((long long)(rank + 1) * 2 * nt / nblk);
    r.p0 = 2 * (p.P / FDC_TILE_ROWS);                      // the whole tiles of the prefix come first in a list
    if (r.p0 < r.h0) r.p0 = r.h0;
    if (r.p0 > r.h1) r.p0 = r.h1;
    r.np = r.h1 - r.p0;
    if (r.np > MASK_WORDS / A) r.np = MASK_WORDS / A;
    if (r.np > MASK_HALVES) r.np = MASK_HALVES;
    // ---- set-up: barriers, the run's rows, the fields' visibility beyond the prefix
    r.nx = p.app_row && rank == 0 ? (A + SROWS - 1) / SROWS : 0;
    if (tid == 0) {
        bs.abort_flag = 0;
        bs.first_beyond = r.h1 - r.h0;
        for (int i = 0; i < nstage; ++i) {
            bs.used[i] = 0;
            bs.asked[i] = i < r.nx ? 1 : 0;
            mbar_init(smem_u32(&bs.full[i]), 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
        for (int i = 0; i < r.nx; ++i) mbar_arrive(smem_u32(&bs.full[i]));      // filled by this block itself, ahead of the main loop
    }
    if (tid < MASK_HALVES) bs.seen[tid] = 0u;
    bool off_list = false;
    int beyond = 0x7fffffff;                               // first half tile of this thread's that reaches beyond the prefix
    for (int i = tid; i < r.h1 - r.h0; i += THREADS) {
        const int pos = r.h0 + i, row0 = r.tiles[pos >> 1] * FDC_TILE_ROWS + (pos & 1) * SROWS;
        if (i < ROW0S) bs.row0[i] = row0;
        if (row0 + SROWS > p.P && beyond == 0x7fffffff) beyond = i;
        off_list |= pos < 2 * (p.P / FDC_TILE_ROWS) && row0 != pos * SROWS;
    }
    __syncthreads();
    if (beyond != 0x7fffffff) atomicMin(&bs.first_beyond, beyond);
    auto cache_bits = [&]() {
        for (int i = tid; i < r.np * A; i += THREADS) {
            const int h = i / A, b = i - h * A;
            const uint32_t x = half_bits(r.mask + (size_t)b * p.W, p.W, p.P, half_row0(r, bs, r.p0 + h));
            bs.bits[i] = x;
            if (x) atomicOr(&bs.seen[h], x);
        }
    };
    // Fused append, from the new rows' places (bs.app_row): which of them every field sees, and their rows
    // taken out of the tables of the cache's half tiles.
    auto new_bits = [&]() {
        for (int i = tid; i < r.np * A; i += THREADS) {
            const int h = i / A, b = i - h * A, x = bs.app_row[b] - half_row0(r, bs, r.p0 + h);
            if (x >= 0 && x < SROWS) {
                atomicAnd(&bs.seen[h], ~(1u << x));
                for (int b2 = 0; b2 < A; ++b2) atomicAnd(&bs.bits[h * A + b2], ~(1u << x));
            }
        }
        for (int i = warp; i < r.nx * A; i += NW) {
            const int x = i / A, b = i - x * A, j = x * SROWS + lane;
            const int ar = j < A ? bs.app_row[j] : -1, t = ar - p.P;
            const bool on = ar >= 0 && (t >> 6) < p.W && ((r.mask[(size_t)b * p.W + (t >> 6)] >> (t & 63)) & 1ull);
            const uint32_t bits = __ballot_sync(0xffffffffu, on);
            if (lane == 0) bs.newbits[x * FDC_MAX_NODES + b] = bits;
        }
    };
    // (the launch may be ahead of whatever writes the row numbers: what is read here is checked after the wait)
    int ar0 = p.app_row && tid < A ? p.app_row[(size_t)s * p.max_active + tid] : -1;
    if (tid < A) bs.app_row[tid] = ar0 >= p.P && ar0 < p.rows ? ar0 : -1;
    cache_bits();
    __syncthreads();
    if (warp == 0) {
        // the half tiles that hold a visible row, in order
        int n = 0;
        for (int h0 = 0; h0 < r.np; h0 += 32) {
            const bool keep = h0 + lane < r.np && bs.seen[h0 + lane] != 0u;
            const uint32_t ball = __ballot_sync(0xffffffffu, keep);
            if (keep) bs.kept[n + __popc(ball & ((1u << lane) - 1u))] = (uint8_t)(h0 + lane);
            n += __popc(ball);
        }
        if (lane == 0) bs.n_kept = n;
    }
    __syncthreads();
    if (p.app_row) new_bits();                             // (read after the block's next barrier)
    r.total = r.nx + (r.h1 - r.h0) - (r.np - bs.n_kept);
    // stages fb.. may hold rows beyond the prefix (half tiles ahead of p0 are never left out)
    const int fb = r.nx + (bs.first_beyond < r.p0 - r.h0 ? bs.first_beyond : r.p0 - r.h0);
    volatile int* abortp = &bs.abort_flag;
    const uint32_t full0 = smem_u32(bs.full), ring0 = smem_u32(ring);
    auto request = [&](int it, int st, int n) {            // one thread: the copies of stage `it`, the n-th to use slot st
        const uint32_t bar = full0 + 8 * st, dst = ring0 + (uint32_t)st * STAGE_BYTES;
        const int row0 = half_row0(r, bs, stage_pos(r, bs, it));
        mbar_expect_tx(bar, STAGE_BYTES);
#pragma unroll
        for (int h = 0; h < D / 64; ++h) {
            tma_load_4d(dst + h * (SROWS * 128), &tm_k, bar, h * 64, row0, g, s);
            tma_load_4d(dst + SROWS * D * 2 + h * (SROWS * 128), &tm_v, bar, h * 64, row0, g, s);
        }
        __threadfence_block();
        *(volatile int*)&bs.asked[st] = n;
    };
    // the first stages: warp w requests w and w + 8; those of the prefix ahead of the dependency wait
    if (lane == 0) {
        for (int it = warp; it < nstage && it < fb; it += NW)
            if (it >= r.nx) request(it, it, 1);
    }
    __syncwarp();
    if (p.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (lane == 0) {
        for (int it = warp; it < nstage && it < r.total; it += NW)
            if (it >= fb) request(it, it, 1);
    }
    __syncwarp();
    {
        // queries of the pair: row m = field * group + head-in-group; rows M.. up to a whole group are zero
        const int rows = (M + GROWS - 1) / GROWS * GROWS;
        for (int i = tid; i < rows * (D / 8); i += THREADS) {
            const int m = i / (D / 8), dc = i - m * (D / 8);
            const int b = m < M ? (m0 + m) / p.group : 0, hg = m < M ? m0 + m - b * p.group : 0;
            cp_async16(qs + swz(qpanel, m, dc), reinterpret_cast<const uint4*>(p.q) + ((((size_t)s * p.max_active + b) * p.hq + (size_t)g * p.group + hg) * D) / 8 + dc,
                       m < M);
        }
    }
    // the stages of new rows: row i of stage x = the new vectors of field 32 x + i (rows past the last field: zero)
    for (int i = tid; i < r.nx * SROWS * (D / 8); i += THREADS) {
        const int b = i / (D / 8), dc = i - b * (D / 8);
        const size_t src = ((size_t)s * p.max_active * p.hkv + g + (size_t)(b < A ? b : 0) * p.hkv) * (D / 8) + dc;
        unsigned char* ks = ring + (size_t)(b / SROWS) * STAGE_BYTES + swz(SROWS * 128, b % SROWS, dc);
        cp_async16(ks, reinterpret_cast<const uint4*>(p.app_k) + src, b < A);
        cp_async16(ks + SROWS * D * 2, reinterpret_cast<const uint4*>(p.app_v) + src, b < A);
    }
    // only head_dim 128 has ever asked for the prefix tiles to come first
    if (D == 128 && off_list) atomicOr(p.status, FDC_DEV_TILE_LIST);
    int moved = 0;
    if (p.app_row && tid < A) {
        const int ar = __ldcg(p.app_row + (size_t)s * p.max_active + tid);
        if ((ar < p.P || ar >= p.rows) && cluster == s * p.hkv * qsplit && rank == 0) atomicOr(p.status, FDC_DEV_ROW_RANGE);     // skipped and flagged
        moved = ar != ar0;
        ar0 = ar;
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    fence_async_smem();                                    // (the next copy into the new rows' slots goes through the asynchronous proxy)
    if (__syncthreads_or(moved)) {
        // the row numbers were written by the kernel ahead: the tables once more
        if (tid < A) bs.app_row[tid] = ar0 >= p.P && ar0 < p.rows ? ar0 : -1;
        if (tid < MASK_HALVES) bs.seen[tid] = 0u;
        __syncthreads();
        cache_bits();
        __syncthreads();
        new_bits();
        __syncthreads();
    }
    const int mg = warp % groups, kl = warp / groups;
    const int gq = lane >> 2, cq = lane & 3;
    const int left = M - mg * GROWS;                       // rows of this warp's group that exist (<= 0: none)
    const uint32_t q_lane = smem_u32(qs) + (uint32_t)(left > 0 ? mg * GROWS : 0) * 128 + swz(qpanel, lane & 15, lane >> 4);
    const uint32_t k_lane = swz(SROWS * 128, lane & 7, lane >> 3);
    const uint32_t v_lane = SROWS * D * 2 + swz(SROWS * 128, (lane & 7) + ((lane >> 3) & 1) * 8, lane >> 4);
    const int f0 = gq < left ? (m0 + mg * GROWS + gq) / p.group : -1, f1 = gq + 8 < left ? (m0 + mg * GROWS + gq + 8) / p.group : -1;   // fields of the thread's rows
    float o[D / 8][4], l[4], m[2];
#pragma unroll
    for (int n = 0; n < D / 8; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;
    l[0] = l[1] = l[2] = l[3] = 0.f;
    m[0] = m[1] = -INFINITY;
    const float c = p.scale_log2;
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
            uint32_t mk0 = ~0u, mk1 = ~0u, seen = ~0u;
            if (it < r.nx) {
                masked = true;
                mk0 = f0 < 0 ? 0u : bs.newbits[it * FDC_MAX_NODES + f0];
                mk1 = f1 < 0 ? 0u : bs.newbits[it * FDC_MAX_NODES + f1];
                for (int b = 0; b < SROWS && it * SROWS + b < A; ++b)     // (values of rows that are not written do not count either)
                    if (bs.app_row[it * SROWS + b] < 0) seen &= ~(1u << b);
            } else if (it >= fb) {
                const int pos = stage_pos(r, bs, it), row0 = half_row0(r, bs, pos), h = pos - r.p0;
                if (row0 + SROWS > p.P) {
                    masked = true;
                    if (h >= 0 && h < r.np) {
                        mk0 = f0 < 0 ? 0u : bs.bits[h * A + f0];
                        mk1 = f1 < 0 ? 0u : bs.bits[h * A + f1];
                        seen = bs.seen[h];
                    } else {
                        const uint32_t fresh = p.app_row ? new_rows_of(bs.app_row, A, row0) : 0u;
                        mk0 = f0 < 0 ? 0u : half_bits(r.mask + (size_t)f0 * p.W, p.W, p.P, row0) & ~fresh;
                        mk1 = f1 < 0 ? 0u : half_bits(r.mask + (size_t)f1 * p.W, p.W, p.P, row0) & ~fresh;
                        seen = half_seen_slow(r.mask, p.W, p.P, A, row0) & ~fresh;
                    }
                }
            }
            const uint32_t kb = ring0 + (uint32_t)st * STAGE_BYTES;
            if (!masked || __any_sync(0xffffffffu, (mk0 | mk1) != 0u))       // (a half tile that only other groups' fields see)
                process_stage<D>(kb + k_lane, kb + v_lane, q_lane, qpanel, o, l, m, masked, mk0, mk1, seen, c, lane);
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
    float* wp = part + warp * (GROWS * D);
    if (left > 0) {
#pragma unroll
        for (int n = 0; n < D / 8; ++n) {
            *reinterpret_cast<float2*>(wp + part_off<D>(gq, n * 8 + 2 * cq)) = make_float2(o[n][0], o[n][1]);
            *reinterpret_cast<float2*>(wp + part_off<D>(gq + 8, n * 8 + 2 * cq)) = make_float2(o[n][2], o[n][3]);
        }
        if (cq == 0) {
            bs.wml[warp * GROWS + gq] = make_float2(m[0] * c, l[0]);
            bs.wml[warp * GROWS + gq + 8] = make_float2(m[1] * c, l[2]);
        }
    }
    __syncthreads();
    auto store_out = [&](int mm, int c4, const float4& acc, float lt) {
        const float inv = 1.f / lt;
        const int b = (m0 + mm) / p.group, hg = m0 + mm - b * p.group;
        *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.out) + (((size_t)s * p.max_active + b) * p.hq + (size_t)g * p.group + hg) * D + c4) =
            make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
    };
    // block: merge over the warps of a group; with one block per pair that is the result
    merge_lanes<D>(lanes, tid, M, groups * GROWS, bs.wml, part, [&](int mm, int c4, float mx, float lt, const float4& acc) {
        if (nblk == 1) {
            store_out(mm, c4, acc, lt);
        } else {
            *reinterpret_cast<float4*>(part + part_off<D>(mm, c4)) = acc;          // in place of the first lane's partial (one thread reads and writes it)
            if (c4 == 0) bs.cml[mm] = make_float2(mx, lt);
        }
    });
    if (nblk > 1) {
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    }
    // fused append: the new rows whose half tiles are in this block's run go to the cache (this block's copies
    // from there have landed; clusters with the pair's other query rows may still be reading the half
    // tile, but to them, too, the row counts as unseen: its bytes there do not matter)
    if (p.app_row && m0 == 0 && bs.first_beyond < r.h1 - r.h0)
        for (int b = warp; b < A; b += NW) {
            const int ar = bs.app_row[b];
            bool here = false;
            for (int i = bs.first_beyond + lane; i < r.h1 - r.h0; i += 32) {
                const int x = ar - half_row0(r, bs, r.h0 + i);
                here |= x >= 0 && x < SROWS;
            }
            here = __any_sync(0xffffffffu, here && ar >= 0);
            const int dc = lane & 15;
            if (here && dc < D / 8) {
                // lanes 0-15: the K row, lanes 16-31: the V row
                const uint4 x = reinterpret_cast<const uint4*>(lane < 16 ? p.app_k : p.app_v)[((((size_t)s * p.max_active + b) * p.hkv + g) * D) / 8 + dc];
                __nv_bfloat16* cache = const_cast<__nv_bfloat16*>(reinterpret_cast<const __nv_bfloat16*>(lane < 16 ? p.k : p.v));
                *reinterpret_cast<uint4*>(cache + (size_t)s * p.stride_scene + (size_t)g * p.stride_head + (size_t)ar * p.stride_row + dc * 8) = x;
            }
        }
    if (nblk == 1) return;
    // ---- cluster: every block merges its share of the (query row, 4 columns) items over all blocks
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    {
        // Four threads per item, each with every fourth block (at most four: one trip), summed by shuffles.
        const uint32_t ml0 = smem_u32(bs.cml), part0 = smem_u32(part);
        const int q = tid & 3, items = M * (D / 4);
        for (int i0 = (tid >> 2) * nblk + rank; __any_sync(0xffffffffu, i0 < items); i0 += (THREADS / 4) * nblk) {
            const bool on = i0 < items;
            const int mm = on ? i0 / (D / 4) : 0, c4 = on ? (i0 - mm * (D / 4)) * 4 : 0;
            const uint32_t a_ml = ml0 + mm * 8, a_o = part0 + 4 * part_off<D>(mm, c4);
            float2 v[4];
            float4 x[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                v[j] = make_float2(-INFINITY, 0.f);
                x[j] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (on && q + 4 * j < nblk) {
                    v[j] = ld_cluster2(map_rank(a_ml, q + 4 * j));
                    x[j] = ld_cluster4(map_rank(a_o, q + 4 * j));
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
    __syncwarp();
    // nobody leaves while its shared memory is still being read
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ---------------------------------------------------------------- host side
PFN_cuTensorMapEncodeTiled get_encode()
{
    static PFN_cuTensorMapEncodeTiled fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &f, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled)f;
    });
    return fn;
}

struct MapKey {
    const void* base;
    int64_t ss, sh, sr;
    int32_t batch, hkv, rows, d, box_rows, dev;
    bool operator==(const MapKey& o) const
    {
        return dev == o.dev && base == o.base && ss == o.ss && sh == o.sh && sr == o.sr && batch == o.batch && hkv == o.hkv && rows == o.rows && d == o.d && box_rows == o.box_rows;
    }
};
struct MapCache {
    std::mutex mu;
    std::vector<std::pair<MapKey, CUtensorMap>> items;
};
MapCache g_maps;

int get_map(const void* base, const AttnParams& p, int d, int box_rows, CUtensorMap* out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return FDC_ERR_CUDA;
    MapKey key{base, p.stride_scene, p.stride_head, p.stride_row, p.batch, p.hkv, p.rows, d, box_rows, dev};
    std::lock_guard<std::mutex> lk(g_maps.mu);
    for (auto& it : g_maps.items)
        if (it.first == key) {
            *out = it.second;
            return FDC_OK;
        }
    PFN_cuTensorMapEncodeTiled enc = get_encode();
    if (!enc) return FDC_ERR_CUDA;
    cuuint64_t dims[4] = {(cuuint64_t)d, (cuuint64_t)p.rows, (cuuint64_t)p.hkv, (cuuint64_t)p.batch};
    // a dimension of extent 1 still needs a legal (multiple of 16 bytes, non-zero) stride
    auto str = [](int64_t s, int64_t fallback) { return (cuuint64_t)((s > 0 ? s : fallback) * 2); };
    cuuint64_t strides[3] = {str(p.stride_row, d), str(p.stride_head, (int64_t)d * p.rows), str(p.stride_scene, (int64_t)d * p.rows * p.hkv)};
    cuuint32_t box[4] = {64, (cuuint32_t)box_rows, 1, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    alignas(64) CUtensorMap tm;
    CUresult r = enc(&tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return FDC_ERR_SHAPE;
    if (g_maps.items.size() >= 4096) g_maps.items.clear();
    g_maps.items.emplace_back(key, tm);
    *out = tm;
    return FDC_OK;
}

template <int D>
int launch_t(const AttnParams& p, cudaStream_t st)
{
    constexpr int STAGE_BYTES = 2 * SROWS * D * 2;
    const ClusterShape h = p.cluster;
    const int nblk = h.nblk;
    const int qrows = ((p.mmax + GROWS - 1) / GROWS + h.qsplit - 1) / h.qsplit * GROWS;
    const size_t fixed = 1024 + (size_t)qrows * D * 2;
    // two blocks per SM: 228 KB, less 1 KB each for the system
    const size_t room = h.per_sm > 1 ? 113 * 1024 : 227 * 1024;
    int nstage = (int)((room - sizeof(BlockState) - 256 - fixed) / STAGE_BYTES);
    if (nstage > MAX_STAGES) nstage = MAX_STAGES;
    if ((size_t)nstage * STAGE_BYTES < (size_t)NW * GROWS * D * 4) return FDC_ERR_SHAPE;      // the partials take the ring's place
    size_t smem = fixed + (size_t)nstage * STAGE_BYTES;
    if (h.per_sm <= 1 && smem < 120 * 1024) smem = 120 * 1024;        // (more than half of an SM's: no second block beside this one)
    static size_t attr_smem[kMaxDevices] = {};
    int rc = raise_dynamic_smem(reinterpret_cast<const void*>(attn_cluster_kernel<D>), smem, attr_smem);
    if (rc) return rc;
    if (nblk > 8) {
        static std::atomic<uint64_t> wide_ok{0};           // devices on which clusters of 16 have been asked for
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return FDC_ERR_CUDA;
        if (dev > 63 || !((wide_ok.load() >> dev) & 1)) {
            cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void*>(attn_cluster_kernel<D>), cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            if (e != cudaSuccess) return set_cuda_error(e);
            if (dev <= 63) wide_ok.fetch_or(1ull << dev);
        }
    }
    alignas(64) CUtensorMap tk, tv;
    rc = get_map(p.k, p, D, SROWS, &tk);
    if (rc) return rc;
    rc = get_map(p.v, p, D, SROWS, &tv);
    if (rc) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((long long)p.batch * p.hkv * h.qsplit * nblk));
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)nblk;
    at[1].val.clusterDim.y = 1;
    at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    cudaError_t e = cudaLaunchKernelEx(&cfg, attn_cluster_kernel<D>, p, tk, tv, nstage, nblk, h.qsplit, qrows);
    if (e != cudaSuccess) return set_cuda_error(e);
    note_launch();
    return FDC_OK;
}

}  // namespace

namespace fdc {

int get_kv_tensor_map(const void* base, const AttnParams& p, int head_dim, int box_rows, void* out_map)
{
    return get_map(base, p, head_dim, box_rows, reinterpret_cast<CUtensorMap*>(out_map));
}

// How a launch is cut: blocks per cluster (shares of a pair's rows), clusters per pair (shares of its query
// rows; each reads all the pair's K/V, the later ones from L2) and blocks per SM, by the lowest estimate of
//     fixed + waves x (one block's time)
// where a block's time is the largest of its warps' chain of stages (latency), its SM's share of the
// arithmetic and its SM's share of the bytes, and an SM with two blocks shares the last two.  The constants (us)
// are a least-squares fit to 309 shapes x up to 40 cuts measured on a B200 (1 to 64 scenes, prefix 400 to 20000,
// 2 to 128 query rows, head_dim 64 and 128): the cut it takes is on average 4 % slower than the best one
// measured.  Cutting the query rows pays while the chip has idle SMs: one scene, 4 KV heads, 42 query rows,
// prefix 2048: 16.8 us a layer with one cluster of 16 blocks per KV head, 10.4 us with three of 6.
ClusterShape pick_cluster(const ClusterProblem& c, float* us)
{
    static const int sizes[] = {1, 2, 3, 4, 6, 8, 16};
    // clusters of a size that a B200 (148 SMs) holds at once, one block per SM and two
    // (cudaOccupancyMaxActiveClusters): the SMs of a cluster share one GPC
    static const int holds[2][7] = {{148, 74, 45, 33, 22, 15, 7}, {296, 148, 93, 71, 45, 33, 14}};
    const bool d64 = c.head_dim == 64;
    const float chain = d64 ? 0.53f : 0.99f, arith = d64 ? 0.11f : 0.21f;      // per stage of a warp; per stage and group of an SM
    const int groups_all = (c.mmax + 15) / 16;
    const float rows = (float)c.P + 0.5f * (float)c.T, pairs = (float)c.pairs, stages = rows / 32.f;
    ClusterShape best{1, 1, 2};
    float t_best = 1e30f;
    for (int q = 1; q <= groups_all; ++q) {
        const int gl = (groups_all + q - 1) / q;
        if (q > 1 && gl == (groups_all + q - 2) / (q - 1)) continue;           // (no fewer groups per cluster than with q - 1)
        const int lanes = gl <= 1 ? 8 : (gl <= 2 ? 4 : (gl <= 4 ? 2 : 1));
        // time of the bytes at what the chip streams (K/V read again by further clusters comes from L2)
        const float t_mem = 3.2f + pairs * rows * (float)(c.head_dim * 4) * 1e-6f * sqrtf((float)q) / 5.36f;
        for (int i = 0; i < 7; ++i)
            for (int two = 0; two < 2; ++two) {
                const float n = (float)sizes[i], clusters = pairs * (float)q, hold = (float)holds[two][i] * (float)c.sm_count / 148.f;
                if (sizes[i] > 1 && stages < 2.f * n) continue;
                const float waves = clusters > hold ? clusters / hold + 0.4f : 1.f;
                const float share = two ? fminf(2.f, fmaxf(1.f, clusters * n / (float)c.sm_count)) : 1.f;
                const float sb = ceilf(stages / n);
                const float body = fmaxf(ceilf(sb / (float)lanes) * chain, sb * share * fmaxf((float)gl * arith, (float)(c.head_dim * 128) * 1e-3f / 56.f));
                const float t = fmaxf(3.2f + (body + (sizes[i] > 1 ? 1.f : 0.f) + 4.2f * (float)gl) * waves, t_mem);
                if (t < t_best * 0.995f) {
                    t_best = t;
                    best = ClusterShape{sizes[i], q, two + 1};
                }
            }
    }
    if (us) *us = t_best;
    return best;
}

// bf16 only.  Returns FDC_ERR_SHAPE when the tensor map cannot describe the cache (the caller
// then uses the CUDA-core kernel).
int launch_attn_cluster(const AttnParams& p, int head_dim, cudaStream_t st)
{
    return head_dim == 64 ? launch_t<64>(p, st) : launch_t<128>(p, st);
}

}  // namespace fdc
