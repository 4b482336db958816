// Attention of one (scene, KV head) pair by ONE thread-block cluster (bf16, head_dim 64 or 128): split,
// softmax and merge in a single kernel, the partial results exchanged through distributed shared
// memory instead of a workspace.
//
// What bounds it.  A pass of one or a few scenes moves a few MB per layer: streaming them takes 1 to
// 5 us, and the rest of a layer's time is a chain of latencies (dependency wait -> queries -> scores
// -> softmax -> output -> merge -> end of the grid).  This kernel is made for a short chain: no TMEM, no
// arrival counters, no partials in global memory, no second kernel and no split table.  The blocks
// of a pair take equal runs of its 32-row half tiles; everything of the prefix that fits the ring is
// requested before the dependency wait; the merge is one one-way trip inside the cluster (fdc_cluster.cuh).  The tensor work
// is small here (a pair has 1 to 128 query rows), so it is done by mma.sync from registers, which
// needs no hand-over between issuing thread, tensor memory and softmax threads.
//
// Sec. 3.3: all queries of a pair (parallel fields x GQA heads) share ONE read of its KV rows (one
// per cluster where the query rows are cut, see pick_cluster).
//
// Measured (a layer, graphs of whole passes, against the kernels that served these shapes before): 1 scene, 28/4
// heads x 128, prefix 1024, one field: 14.6 -> 6.1 us; prefix 2048, six fields: 19.3 -> 9.8; 1 scene, 14/2 heads x
// 64, prefix 1531, six fields, append apart and issued by the host: 56.2 -> 12.4; 16 scenes, 14/2 x 64, prefix 4096: 56.4 -> 18.4.
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
// run holds a row's half tile writes it to the cache after it has sent its partials.
#include <cudaTypedefs.h>

#include <cmath>
#include <mutex>
#include <vector>

#include "fdc_cluster.cuh"

using namespace fdc;

namespace {

constexpr int SROWS = 32;                     // KV rows per stage (half a tile)

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

template <int HEAD_DIM>
struct MathBf16 {
    using Elem = __nv_bfloat16;
    static constexpr int D = HEAD_DIM, NW = 8, SROWS = ::SROWS, GROWS = 16, GROUPS = 8, ROWS = 2, STAGE_BYTES = 2 * SROWS * D * 2;
    static constexpr bool PREFIX_FIRST = D == 128, FUSES = true, K_REUSED = false;
    float o[D / 8][4], l[4], m[2];
    const float c;
    const int lane;
    const uint32_t qpanel, q_lane, k_lane, v_lane;         // lane addresses of the operands' fragments

    static __host__ __device__ __forceinline__ size_t q_bytes(int qrows) { return (size_t)qrows * D * 2; }
    static __device__ __forceinline__ uint32_t q_off(int qrows, int m, int dc) { return swz((uint32_t)qrows * 128, m, dc); }
    // Float offset of (row, column) of a partial [rows][D]: the columns' groups of 8 are permuted by the row
    // so that the accumulator fragments' stores spread over the banks.
    static __device__ __forceinline__ int part_off(int row, int col) { return row * D + (col ^ ((row & 3) << 3)); }
    static __device__ __forceinline__ void store(Elem* out, const float4& x)
    {
        *reinterpret_cast<uint2*>(out) = make_uint2(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w));
    }
    __device__ __forceinline__ MathBf16(const AttnParams& p, const unsigned char* qs, int qrows, int q0, int ln, int)
        : c(p.scale_log2), lane(ln), qpanel((uint32_t)qrows * 128), q_lane(smem_u32(qs) + (uint32_t)q0 * 128 + swz((uint32_t)qrows * 128, ln & 15, ln >> 4)),
          k_lane(swz(SROWS * 128, ln & 7, ln >> 3)), v_lane(STAGE_BYTES / 2 + swz(SROWS * 128, (ln & 7) + ((ln >> 3) & 1) * 8, ln >> 4))
    {
#pragma unroll
        for (int n = 0; n < D / 8; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;
        l[0] = l[1] = l[2] = l[3] = 0.f;
        m[0] = m[1] = -INFINITY;
    }
    __device__ __forceinline__ int row(int i) const { return (lane >> 2) + 8 * i; }
    template <class F>
    __device__ __forceinline__ void stage(uint32_t kb, bool masked, const uint32_t (&mk)[ROWS], uint32_t seen, F&&)
    {
        process_stage<D>(kb + k_lane, kb + v_lane, q_lane, qpanel, o, l, m, masked, mk[0], mk[1], seen, c, lane);
    }
    __device__ __forceinline__ void write(float* part, float2* ml, int rows) const      // (of the first `rows` query rows)
    {
        const int gq = lane >> 2, cq = lane & 3;
#pragma unroll
        for (int n = 0; n < D / 8; ++n) {
            if (gq < rows) *reinterpret_cast<float2*>(part + part_off(gq, n * 8 + 2 * cq)) = make_float2(o[n][0], o[n][1]);
            if (gq + 8 < rows) *reinterpret_cast<float2*>(part + part_off(gq + 8, n * 8 + 2 * cq)) = make_float2(o[n][2], o[n][3]);
        }
        if (cq == 0) {
            ml[gq] = make_float2(m[0] * c, l[0]);
            ml[gq + 8] = make_float2(m[1] * c, l[2]);
        }
    }
};

template <int D>
__global__ void __launch_bounds__(MathBf16<D>::NW * 32, 2)
attn_cluster_kernel(const __grid_constant__ AttnParams p, const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                    const __grid_constant__ ClusterArgs args)
{
    attn_cluster_body<MathBf16<D>>(p, tm_k, tm_v, args);
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
    int32_t batch, hkv, rows, d, box_rows, dev, dtype;
    bool operator==(const MapKey& o) const
    {
        return dev == o.dev && base == o.base && ss == o.ss && sh == o.sh && sr == o.sr && batch == o.batch && hkv == o.hkv && rows == o.rows && d == o.d && box_rows == o.box_rows && dtype == o.dtype;
    }
};
struct MapCache {
    std::mutex mu;
    std::vector<std::pair<MapKey, CUtensorMap>> items;
};
MapCache g_maps;

int get_map(const void* base, const AttnParams& p, int dtype, int d, int box_rows, CUtensorMap* out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return FDC_ERR_CUDA;
    MapKey key{base, p.stride_scene, p.stride_head, p.stride_row, p.batch, p.hkv, p.rows, d, box_rows, dev, dtype};
    std::lock_guard<std::mutex> lk(g_maps.mu);
    for (auto& it : g_maps.items)
        if (it.first == key) {
            *out = it.second;
            return FDC_OK;
        }
    // A cache expanded over scenes or heads (stride 0, extent > 1) is nothing that a tensor map describes.
    if ((p.batch > 1 && p.stride_scene == 0) || (p.hkv > 1 && p.stride_head == 0)) return FDC_ERR_SHAPE;
    PFN_cuTensorMapEncodeTiled enc = get_encode();
    if (!enc) return FDC_ERR_CUDA;
    cuuint64_t dims[4] = {(cuuint64_t)d, (cuuint64_t)p.rows, (cuuint64_t)p.hkv, (cuuint64_t)p.batch};
    const int64_t es = dtype == FDC_F32 ? 4 : 2;
    // a dimension of extent 1 still needs a legal (multiple of 16 bytes, non-zero) stride
    auto str = [es](int64_t s, int64_t fallback) { return (cuuint64_t)((s > 0 ? s : fallback) * es); };
    cuuint64_t strides[3] = {str(p.stride_row, d), str(p.stride_head, (int64_t)d * p.rows), str(p.stride_scene, (int64_t)d * p.rows * p.hkv)};
    cuuint32_t box[4] = {(cuuint32_t)(128 / es), (cuuint32_t)box_rows, 1, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    alignas(64) CUtensorMap tm;
    CUresult r = enc(&tm, dtype == FDC_F32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return FDC_ERR_SHAPE;
    if (g_maps.items.size() >= 4096) g_maps.items.clear();
    g_maps.items.emplace_back(key, tm);
    *out = tm;
    return FDC_OK;
}

}  // namespace

namespace fdc {

int get_kv_tensor_map(const void* base, const AttnParams& p, int dtype, int head_dim, int box_rows, void* out_map)
{
    return get_map(base, p, dtype, head_dim, box_rows, reinterpret_cast<CUtensorMap*>(out_map));
}

static size_t block_room(int per_sm) { return per_sm > 1 ? 113 * 1024 : 227 * 1024; }       // two blocks per SM: 228 KB, less 1 KB each for the system
// Stages in the ring of a block of a cluster of n with `rows` query rows; 0: it finds no room for what the other blocks send it
// beside a ring that its own partials fit.  (With two blocks per SM and head_dim 128: more than 48 rows in clusters of several blocks.)
int cluster_ring(int head_dim, int rows, int nblk, int per_sm)
{
    return head_dim == 64 ? cluster_ring_stages<MathBf16<64>>(block_room(per_sm), rows, nblk) : cluster_ring_stages<MathBf16<128>>(block_room(per_sm), rows, nblk);
}

// How a launch is cut: blocks per cluster (shares of a pair's rows), clusters per pair (shares of its query
// rows; each reads all the pair's K/V, the later ones from L2) and blocks per SM, by the lowest estimate of
//     fixed + waves x (one block's time) + a launch that does not fit beside the one ahead
// where a block's time is the largest of its warps' chain of stages (latency), its SM's share of the arithmetic and its SM's share
// of the bytes (an SM with two blocks shares the last two), and its ring's turns.  Two things decide besides the work:
//  - consecutive launches overlap only where both find a place: else the later one's set-up begins when the one ahead ends.  4
//    pairs, 7 query rows, prefix 1024: 7.2 us a layer with clusters of 16 and one block per SM (7 fit the chip), 6.1 with two;
//  - a run longer than the ring gets a ring's stages per turn (a copy's latency and the stage's work: 2.5 us and 0.7 more per group of
//    query rows), and with two blocks per SM a ring is half as deep.  56 pairs, 12 query rows, prefix 4737: 33.3 us a layer with
//    (3, 1, 2), 25.0 with (3, 1, 1).
// The constants (us) are the best of a grid over 1110 (head_dim 128) and 650 (64) shapes drawn over 2 to 500 pairs, prefix 256 to 32700, 2 to 128 query
// rows, at any pass of their templates, with up to 60 cuts of each timed on a B200: the cut taken with head_dim 64 is on average 8 % slower than the
// best one timed, 12 % without the last two terms.  562 of the 650 are faster by more than 4 % than with the cuts (and the merge) of before, 8 are slower by
// more than that (60 pairs of 35 rows, prefix 4802: 35.0 -> 44.9 us a layer).  Cutting the query rows pays while the chip has idle SMs: one
// scene, 4 KV heads, 42 query rows, prefix 2048: 10.8 us a layer with one cluster of 16 blocks per KV head, 9.8 with three.
ClusterShape pick_cluster(const ClusterProblem& c, float* us)
{
    static const int sizes[] = {1, 2, 3, 4, 6, 8, 16};
    // clusters of a size that a B200 (148 SMs) holds at once, one block per SM and two
    // (cudaOccupancyMaxActiveClusters): the SMs of a cluster share one GPC
    static const int holds[2][7] = {{148, 74, 45, 33, 22, 15, 7}, {296, 148, 93, 71, 45, 33, 14}};
    const bool d64 = c.head_dim == 64;
    const float chain = d64 ? 0.65f : 1.2f, arith = d64 ? 0.11f : 0.21f;       // per stage of a warp; per stage and group of an SM
    const float merge = 1.f, late = 0.7f;
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
                const int ring = cluster_ring(c.head_dim, gl * 16, sizes[i], two + 1);
                if (ring == 0) continue;                   // (no room for the partials)
                const float waves = clusters > hold ? clusters / hold + 0.4f : 1.f;
                const float share = two ? fminf(2.f, fmaxf(1.f, clusters * n / (float)c.sm_count)) : 1.f;
                const float sb = ceilf(stages / n);
                const float turns = sb > (float)ring ? (sb - (float)ring) / (float)ring * (2.5f + 0.7f * (float)gl) + chain : 0.f;
                const float body = fmaxf(fmaxf(ceilf(sb / (float)lanes) * chain, turns), sb * share * fmaxf((float)gl * arith, (float)(c.head_dim * 128) * 1e-3f / 56.f));
                const float over = fminf(fmaxf((2.f * clusters - hold) / hold, 0.f), 1.f);
                const float t = fmaxf(3.2f + (body + (sizes[i] > 1 ? merge : 0.f) + 4.2f * (float)gl) * waves + late * over, t_mem);
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
    const size_t room = block_room(p.cluster.per_sm);
    return head_dim == 64 ? launch_cluster<MathBf16<64>>(attn_cluster_kernel<64>, p, room, p.cluster, st)
                          : launch_cluster<MathBf16<128>>(attn_cluster_kernel<128>, p, room, p.cluster, st);
}

}  // namespace fdc
