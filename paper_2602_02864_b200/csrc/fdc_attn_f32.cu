// Attention over fp32 caches: clusters as in fdc_cluster.cuh, the arithmetic in plain fp32 FMAs (no TF32: the
// fp32 configuration is exact to rounding) from register tiles.
//
// What bounds it.  A KV row of 32-bit values costs 2 x head_dim FMAs per query row, and an SM does 128 a cycle; the
// operands come from shared memory at 128 bytes a cycle, so every value that is read has to serve several FMAs.
// A warp takes a whole stage (16 KV rows) times the query rows of its group (4 QL), a lane a tile of QL query rows x 2
// KV rows of the scores and of QL query rows x head_dim / 8 columns of the result; the 8 lanes of a quarter warp
// share their query rows and differ in KV rows and columns.  A 16-byte read of a warp takes the port 4 cycles when the
// lanes of a quarter differ and 2 when they agree (measured).  FMAs go two to an instruction (about 80 % of their
// rate with three different operands), which leaves issue slots for the reads.
// A stage keeps its slot for as long as it is worked on, so what an SM does is the number of slots (10 to 12 of 16 KB with head_dim 128)
// over a stage's time.  Which tile and how many warps: see launch_attn_f32.  The kernel that ran before this one (one warp per query
// row) took 955 us a layer at 8 scenes with six fields, 32/8 heads x 128, prefix 2000, where this one takes 80.
#include "fdc_cluster.cuh"

using namespace fdc;

namespace {

template <int HEAD_DIM, int QLANE, int NWARPS, int NGROUPS>
struct MathF32 {
    using Elem = float;
    static constexpr int D = HEAD_DIM, NW = NWARPS, SROWS = 16, JR = SROWS / 8, QL = QLANE, GROWS = 4 * QL, GROUPS = NGROUPS, ROWS = QL, STAGE_BYTES = 2 * SROWS * D * 4;
    static constexpr bool PREFIX_FIRST = false, FUSES = false, K_REUSED = true;
    static constexpr int QP = (QL + 1) / 2 * 2;            // weights per lane and KV row in shared memory (pairs)
    static constexpr int QROW = (D + 4) * 4;               // bytes of a query row in shared memory (16 more: neighbouring rows on other banks)
    static constexpr int PROW = (4 * QP + 4) * 4;          // bytes of a KV row's weights, the same way
    static_assert(GROUPS * SROWS * PROW <= STAGE_BYTES / 2, "the weights take the place of the stage's K rows");
    // Lane = (qg, rg): query rows qg + 4 i (i < QL), KV rows rg + 8 j of the scores, columns 32 h + 4 rg .. + 3 of the result.
    uint64_t o[QL][D / 32][2];                             // pairs of columns
    float l[QL], m[QL];
    const float scale;
    const int qg, rg;
    const uint32_t q_lane, p_off;                          // p_off: place of the group's weights in the stage
    const bool few;                                        // at most half of the group's rows exist: half tiles serve them

    static __host__ __device__ __forceinline__ size_t q_bytes(int qrows) { return (size_t)qrows * QROW; }
    static __device__ __forceinline__ uint32_t q_off(int, int m, int dc) { return (uint32_t)(m * QROW + dc * 16); }
    static __device__ __forceinline__ int part_off(int row, int col) { return row * D + col; }
    static __device__ __forceinline__ void store(float* out, const float4& x) { *reinterpret_cast<float4*>(out) = x; }
    __device__ __forceinline__ MathF32(const AttnParams& p, const unsigned char* qs, int, int q0, int lane, int rows)
        : scale(p.scale_log2), qg(lane >> 3), rg(lane & 7), q_lane(smem_u32(qs) + (q0 + (lane >> 3)) * QROW), p_off(q0 ? SROWS * PROW : 0), few(rows <= GROWS / 2)
    {
#pragma unroll
        for (int i = 0; i < QL; ++i) {
#pragma unroll
            for (int h = 0; h < D / 32; ++h) o[i][h][0] = o[i][h][1] = 0ull;
            l[i] = 0.f;
            m[i] = -INFINITY;
        }
    }
    __device__ __forceinline__ int row(int i) const { return qg + 4 * i; }
    // Two fp32 FMAs in one instruction, each rounded like any other: the FMA pipe takes two cycles for it, so half of
    // the issue slots are left for the loads and the addresses.
    static __device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
    {
        uint64_t d;
        asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
        return d;
    }
    static __device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b)
    {
        uint64_t d;
        asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
        return d;
    }
    static __device__ __forceinline__ uint64_t pair(float lo, float hi)
    {
        uint64_t d;
        asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
        return d;
    }
    static __device__ __forceinline__ float2 halves(uint64_t x)
    {
        float2 v;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(x));
        return v;
    }
    static __device__ __forceinline__ void lds4(uint32_t a, uint64_t& lo, uint64_t& hi)
    {
        asm volatile("ld.shared.v2.b64 {%0,%1}, [%2];" : "=l"(lo), "=l"(hi) : "r"(a) : "memory");
    }
    // Weights and values of one KV row.
    struct Row {
        float w[QP];
        uint64_t v[D / 32][2];
        template <int N>
        __device__ __forceinline__ void load(uint32_t pr, uint32_t vb, int rg, int r)
        {
#pragma unroll
            for (int i = 0; i < (N + 1) / 2 * 2; i += 2)
                asm volatile("ld.shared.v2.f32 {%0,%1}, [%2];" : "=f"(w[i]), "=f"(w[i + 1]) : "r"(pr + (uint32_t)(r * PROW + i * 4)) : "memory");
            const uint32_t a = vb + (uint32_t)(r * 128) + (uint32_t)((rg ^ (r & 7)) << 4);
#pragma unroll
            for (int h = 0; h < D / 32; ++h) lds4(a + (uint32_t)(h * (SROWS * 128)), v[h][0], v[h][1]);
        }
        // SOME: only for the query rows that see the KV row, r (a weight of 0 is no help against an infinite or NaN value)
        template <int N, bool SOME>
        __device__ __forceinline__ void fma(uint64_t (&o)[QL][D / 32][2], const uint32_t (&mk)[ROWS], int r) const
        {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                if (SOME && !((mk[i] >> r) & 1u)) continue;
                const uint64_t w2 = pair(w[i], w[i]);
#pragma unroll
                for (int h = 0; h < D / 32; ++h) {
                    o[i][h][0] = fma2(w2, v[h][0], o[i][h][0]);
                    o[i][h][1] = fma2(w2, v[h][1], o[i][h][1]);
                }
            }
        }
    };
    template <class F>
    __device__ __forceinline__ void stage(uint32_t kb, bool masked, const uint32_t (&mk)[ROWS], uint32_t, F&& k_read)
    {
        // (one group: its tile is made for the widest frontier, and a single field would pay for all of it)
        if (GROUPS == 1 && few) stage_rows<QL / 2>(kb, masked, mk, k_read);
        else stage_rows<QL>(kb, masked, mk, k_read);
    }
    template <int N, class F>
    __device__ __forceinline__ void stage_rows(uint32_t kb, bool masked, const uint32_t (&mk)[ROWS], F&& k_read)
    {
        uint64_t s2[N][JR];                               // (sum over even columns, sum over odd columns)
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int j = 0; j < JR; ++j) s2[i][j] = 0ull;
        // S = Q K^T: columns 4 d4 .. + 3 sit in chunk d4 of their panel, XORed with the row.  With two warps per scheduler (8 warps) a
        // step's operands are read a step ahead; with three that costs registers and gains nothing.
        constexpr int AHEAD = NW == 8 ? 1 : 0;
        uint64_t k[AHEAD + 1][JR][2], q[AHEAD + 1][N][2];
        auto load = [&](auto B, uint32_t kc, uint32_t qc) {
#pragma unroll
            for (int j = 0; j < JR; ++j) lds4(kc + j * 1024, k[B][j][0], k[B][j][1]);
#pragma unroll
            for (int i = 0; i < N; ++i) lds4(qc + i * 4 * QROW, q[B][i][0], q[B][i][1]);
        };
        uint32_t ka = kb + (uint32_t)rg * 128, qa = q_lane;
        if (AHEAD) load(std::integral_constant<int, 0>{}, ka + (uint32_t)(rg << 4), qa);
#pragma unroll 1
        for (int h = 0; h < D / 32; ++h) {
            static_for<8>([&](auto D4) {
                constexpr int d4 = D4, at = (d4 + AHEAD) & 7, step = (d4 + AHEAD) >> 3;     // (past the last panel: what lies there is not used)
                load(std::integral_constant<int, AHEAD ? (d4 + 1) & 1 : 0>{}, ka + step * (SROWS * 128) + (uint32_t)((at ^ rg) << 4), qa + step * 128 + at * 16);
                constexpr int use = AHEAD ? d4 & 1 : 0;
#pragma unroll
                for (int i = 0; i < N; ++i) {
#pragma unroll
                    for (int j = 0; j < JR; ++j) s2[i][j] = fma2(q[use][i][0], k[use][j][0], s2[i][j]);
#pragma unroll
                    for (int j = 0; j < JR; ++j) s2[i][j] = fma2(q[use][i][1], k[use][j][1], s2[i][j]);
                }
            });
            ka += SROWS * 128;
            qa += 128;
        }
        float s[N][JR];
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int j = 0; j < JR; ++j) {
                const float2 x = halves(s2[i][j]);
                s[i][j] = x.x + x.y;
            }
        k_read();                                          // both groups have read the K rows: the weights take their place
#pragma unroll
        for (int i = 0; i < N; ++i) {
#pragma unroll
            for (int j = 0; j < JR; ++j) {
                s[i][j] *= scale;
                if (masked && !((mk[i] >> (rg + 8 * j)) & 1u)) s[i][j] = -INFINITY;
            }
            float x = s[i][0];
#pragma unroll
            for (int j = 1; j < JR; ++j) x = fmaxf(x, s[i][j]);
#pragma unroll
            for (int d = 1; d < 8; d <<= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, d));
            const float mn = fmaxf(m[i], x), ms = mn == -INFINITY ? 0.f : mn;
            if (mn != m[i]) {                              // (uniform over the lanes that share the row)
                const float a = exp2f(m[i] - ms);
                l[i] *= a;
                const uint64_t a2 = pair(a, a);
#pragma unroll
                for (int h = 0; h < D / 32; ++h) {
                    o[i][h][0] = mul2(o[i][h][0], a2);
                    o[i][h][1] = mul2(o[i][h][1], a2);
                }
                m[i] = mn;
            }
#pragma unroll
            for (int j = 0; j < JR; ++j) {
                s[i][j] = exp2f(s[i][j] - ms);
                l[i] += s[i][j];
            }
        }
        // weights [KV row][qg][i]
        const uint32_t pw = kb + p_off + (uint32_t)rg * PROW + (uint32_t)qg * (QP * 4);
#pragma unroll
        for (int j = 0; j < JR; ++j)
#pragma unroll
            for (int i = 0; i < (N + 1) / 2 * 2; i += 2)
                asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(pw + (uint32_t)(j * 8 * PROW + i * 4)), "f"(s[i][j]), "f"(i + 1 < N ? s[i + 1 < N ? i + 1 : 0][j] : 0.f) : "memory");
        const uint32_t vb = kb + STAGE_BYTES / 2, pr = kb + p_off + (uint32_t)qg * (QP * 4);
        __syncwarp();
        // O += P V, a KV row a step.  Rows that a query row does not see can hold anything, a sibling field's infinities
        // and NaN among them: a stage that reaches beyond the prefix goes by the query rows' bits.
        if (masked) {
            Row x;
#pragma unroll 1
            for (int r = 0; r < SROWS; ++r) {
                x.template load<N>(pr, vb, rg, r);
                x.template fma<N, true>(o, mk, r);
            }
        } else if (GROUPS == 1 && NW == 12) {              // (tiles of 6 rows at 168 registers: no room for a second row's operands)
            Row x;
#pragma unroll 1
            for (int r = 0; r < SROWS; ++r) {
                x.template load<N>(pr, vb, rg, r);
                x.template fma<N, false>(o, mk, r);
            }
        } else {
            // the next row's operands are read while this one's FMAs run
            Row x, y;
            x.template load<N>(pr, vb, rg, 0);
#pragma unroll 1
            for (int r = 0; r < SROWS; r += 2) {
                y.template load<N>(pr, vb, rg, r + 1);
                x.template fma<N, false>(o, mk, r);
                if (r + 2 < SROWS) x.template load<N>(pr, vb, rg, r + 2);
                y.template fma<N, false>(o, mk, r + 1);
            }
        }
        __syncwarp();
        fence_async_smem();                                // the stage's next copy goes through the asynchronous proxy
    }
    __device__ __forceinline__ void write(float* part, float2* ml, int)
    {
#pragma unroll
        for (int i = 0; i < QL; ++i) {
#pragma unroll
            for (int d = 1; d < 8; d <<= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], d);
            if (rg == 0) ml[row(i)] = make_float2(m[i], l[i]);
#pragma unroll
            for (int h = 0; h < D / 32; ++h)
                *reinterpret_cast<ulonglong2*>(part + part_off(row(i), h * 32 + rg * 4)) = make_ulonglong2(o[i][h][0], o[i][h][1]);
        }
    }
};

template <int D, int QL, int NW, int GROUPS>
__global__ void __launch_bounds__(NW * 32, 1)
attn_f32_kernel(const __grid_constant__ AttnParams p, const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                const __grid_constant__ ClusterArgs args)
{
    attn_cluster_body<MathF32<D, QL, NW, GROUPS>>(p, tm_k, tm_v, args);
}

template <int D>
int launch_d(const AttnParams& p, const ClusterShape& h, int ql, cudaStream_t st)
{
    const size_t room = 227 * 1024;
    switch (ql) {
        case 2: return launch_cluster<MathF32<D, 2, 12, 2>>(attn_f32_kernel<D, 2, 12, 2>, p, room, h, st);
        case 4: return launch_cluster<MathF32<D, 4, 12, 2>>(attn_f32_kernel<D, 4, 12, 2>, p, room, h, st);
        default: {
            constexpr int NW = D == 64 ? 12 : 8;
            return launch_cluster<MathF32<D, 6, NW, 1>>(attn_f32_kernel<D, 6, NW, 1>, p, room, h, st);
        }
    }
}

}  // namespace

namespace fdc {

// fp32 only.  Clusters per pair: as many as 32 query rows each need, all of the same width.  Blocks per cluster: what keeps all
// clusters on the chip at once (one block per SM; clusters of 2, 3, 4, 6, 8 that fit a B200 at once: 74, 45, 33, 22, 15), and no more
// than give every block at least two tiles (eight stages).  The tile, by a cluster's query rows:
//   1 to 8, 9 to 16   QL 2, 4: 12 warps in one group.
//   17 to 24          QL 6, one group: in two, every K and V row is read twice, and the shared memory port (14 cycles for 6 of FMAs in the
//                     scores, 18 for 12 in the result, against 20 for 12 and 20 for 24) is what they wait for.  head_dim 128 has 8 warps (an
//                     accumulator of 96 registers), 64 has 12: a pass with few fields at work has a warp per stage as its only
//                     parallelism, and 8 of them took 73.2 -> 91.8 us a layer with 24 fields done, 48 pairs of 48 rows.  us a layer, QL 3 in two
//                     groups of 12 warps / this: 8 scenes, 32/8 x 128, six fields, prefix 2048 88.8 / 79.6, one field left 61.8 / 58.2; 24 scenes,
//                     prefix 256, one field left 77.3 / 80.5 (here two groups are better); 8 scenes, 4/2 x 64, 24 fields, prefix 2048 47.7 / 42.4, one
//                     field left 36.9 / 37.3.
//   25 to 32          QL 4 in two groups of 12 warps: one group with tiles of 8 rows is 1 to 10 % slower with head_dim 128, and with 64
//                     slower where few fields are at work (48 pairs of 56 rows, prefix 256, one field left 40.4 / 43.3).
int launch_attn_f32(const AttnParams& p, int head_dim, cudaStream_t st)
{
    ClusterShape h{1, (p.mmax + 31) / 32, 1};
    const int per = (p.mmax + h.qsplit - 1) / h.qsplit;
    const int ql = per <= 8 ? 2 : (per <= 16 ? 4 : (per <= 24 ? 6 : 4));
    if (ql == 6) h.qsplit = (p.mmax + 23) / 24;
    const long long clusters = (long long)p.batch * p.hkv * h.qsplit;
    static const int sizes[] = {2, 3, 4, 6, 8}, holds[] = {74, 45, 33, 22, 15};
    for (int i = 0; i < 5; ++i)
        if (clusters <= (long long)holds[i] * p.n_cta / 148 && p.ntile_max >= 2 * sizes[i]) h.nblk = sizes[i];
    return head_dim == 64 ? launch_d<64>(p, h, ql, st) : launch_d<128>(p, h, ql, st);
}

}  // namespace fdc
