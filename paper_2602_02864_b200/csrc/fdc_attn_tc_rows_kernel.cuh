// Split-KV pass for bf16 caches (head_dim 128) on the 5th-generation tensor cores (tcgen05 + TMEM), query rows on the M
// side of the multiplications: for pairs of more than 64 query rows (the transposed form, fdc_attn_tc_kernel.cuh,
// serves the narrower ones).
//
// What bounds it.  With 128 query rows a tile of 64 KV rows is 8192 exponentials (512 cycles of the SM's MUFU pipe), and
// in the transposed form the weights also go through shared memory twice (written by the softmax, read by two
// multiplications): its rounds took twice the time their K/V rows take to arrive.  Here the weights never leave tensor
// memory, a thread owns a whole query row (no maximum or sum across threads), and K, V and the copies have shared memory
// for themselves:
//     S = Q K^T     M = 128 query rows, N = 64 KV rows (one tile of the list), K = head_dim; A = Q in TMEM, B = the K tile
//                   as TMA left it
//     O += P V      M = 128, N = head_dim, K = 64; A = P (bf16) in TMEM, in the place of S; B = the V tile (N-major)
// In steady state a tile takes about 1150 cycles, which is what its 32 KB take at an SM's share of the memory (the
// softmax warps need 1130 for every other tile); the first build of this form, with Q in shared memory, rounds of 128
// rows and one thread at a time issuing behind "lane 0", took 2400.
// One persistent CTA per SM, 12 warps (168 registers a thread, 112 bytes of spill stores and 68 of loads):
//   warps 0-7    softmax, two groups on alternate tiles, each with an accumulator and (m, l) of its own (softmax_loop)
//   warp 8       TMA producer of both rings (K and V stages of 16 KB, six each)
//   warp 9       issues S = Q K^T; allocates / frees TMEM
//   warp 10      with fdc_set_fused_append, first writes the pass's new K/V rows that fall into this CTA's tiles
//   warp 11      issues O += P V
// Compiled twice, by the translation units that include it (FDC_TC_TWO: see fdc_tc_common.cuh).
#if !defined(FDC_TC_KERNEL) || !defined(FDC_TC_LAUNCH)
#error "include from a translation unit that defines FDC_TC_TWO (0 or 1), FDC_TC_KERNEL and FDC_TC_LAUNCH"
#endif
#include "fdc_tc_common.cuh"

namespace {

constexpr int MROWS = 128;                   // query rows of a pair at most = M of the multiplications
constexpr int NSOFT = 8;                     // softmax warps: 2 groups x 4 row quadrants
constexpr int W_PROD = NSOFT, W_QK = NSOFT + 1, W_AUX = NSOFT + 2, W_PV = NSOFT + 3;
constexpr int THREADS = (NSOFT + 4) * 32;
constexpr uint32_t TMEM_COLS = 512;          // Q [0,64) | three S / P buffers of 64 columns [64,256) | the groups' accumulators [256,384), [384,512)
constexpr uint32_t TM_S = 64, TM_O = 256;
constexpr int NBUF = 3;                      // tile g (counted over the CTA's run) uses buffer g mod 3 and belongs to group g mod 2, so
constexpr int NBAR = 6;                      // its barriers are numbered g mod 6: a barrier's phases are then all of one group
constexpr int PANEL = TILE * 128;            // 64 rows x 128 bytes (64 bf16 columns)
constexpr int STAGE = (D / 64) * PANEL;      // one K (or V) stage: a tile, 64 rows x head_dim
constexpr int MAXST = 6;                     // stages per ring at most
constexpr float RAISE_LOG2 = 8.f;             // a row's reference is raised when a score exceeds it by more than 2^8
constexpr int MBUF = 1024;                   // bitmap words of a scene kept in shared memory (max_active * W): one buffer

// Instruction descriptor of kind::f16: fp32 accumulate, bf16 A and B, M x N; A K-major, B K-major or (b_mn = 1)
// MN-major (contiguous along N).
__device__ __forceinline__ uint32_t instr_desc(int m, int n, uint32_t b_mn)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (b_mn << 16) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(m >> 4) << 24);
}
// One MMA (cta_group::1, kind::f16) with A in tensor memory (bf16 pairs, 8 columns per 16 values of K).  B's descriptor
// is given as (low, high) words: the address field sits in the low word, so stepping through an operand is
// 32-bit arithmetic for the issuing thread.
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t b_hi, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Barrier of the softmax warps (a named barrier).  Every call site is reached by all eight warps
// the same number of times whatever happens: a warp whose bounded wait ran out goes on without
// waiting but still takes every one of these.
__device__ __forceinline__ void soft_sync() { asm volatile("bar.sync 1, %0;" ::"n"(NSOFT * 32) : "memory"); }

// Small per-CTA state in static shared memory.
struct CtaFlags {
    int abort_flag;                  // a bounded wait ran out somewhere in the CTA
    int v_steps[NBAR];
    int merge[3];                    // last arriver of the pair, first and last CTA of the pair
};

// Everything a role needs to find its barriers and buffers.
struct Ctx : Split {
    // mbarriers: one base address, fixed offsets (kept as functions so that a single register serves them all)
    uint32_t bar0;
    __device__ __forceinline__ uint32_t k_full() const { return bar0; }
    __device__ __forceinline__ uint32_t k_empty() const { return bar0 + 8 * MAXST; }
    __device__ __forceinline__ uint32_t v_full() const { return bar0 + 16 * MAXST; }
    __device__ __forceinline__ uint32_t v_empty() const { return bar0 + 24 * MAXST; }
    __device__ __forceinline__ uint32_t s_full() const { return bar0 + 32 * MAXST; }
    __device__ __forceinline__ uint32_t p_full() const { return bar0 + 32 * MAXST + 8 * NBAR; }
    __device__ __forceinline__ uint32_t pv_done() const { return bar0 + 32 * MAXST + 16 * NBAR; }
    __device__ __forceinline__ uint32_t q_ready() const { return bar0 + 32 * MAXST + 24 * NBAR; }
    __device__ __forceinline__ uint32_t o_free() const { return bar0 + 32 * MAXST + 24 * NBAR + 8; }
    __device__ __forceinline__ uint32_t app_done() const { return bar0 + 32 * MAXST + 24 * NBAR + 16; }
    __device__ __forceinline__ uint32_t peer_done() const { return bar0 + 32 * MAXST + 24 * NBAR + 24; }
    uint32_t tmem;
    unsigned char *kring, *vring;
    float2* ml;                      // [2][128] (reference, sum) of each group's rows at the end of a segment
    int* merge;
    uint64_t* smask;                 // [2][mbuf] the current segment's scene bitmaps (when mstaged)
    int mbuf;                        // words per buffer
    uint64_t* sunion;                // [2][UW] their OR over the scene's active branches (when mstaged and W <= UW)
    int mstaged;
    volatile int* abortp;
    volatile int* v_steps;           // [NBAR] the 16-row steps of the tile to multiply (bit k: rows 16k..)
    int nk, nv;                      // ring depths
};

// Row bitmap (Eq. 1) of branch b of the segment's scene.  While the K/V stream saturates the
// memory system a global read costs microseconds, so the softmax warps copy the scene's bitmaps
// to shared memory at the start of a segment whenever they fit.
__device__ __forceinline__ const uint64_t* mask_row(const AttnParams& p, const Ctx& cx, uint32_t seg, int s, int b)
{
    return cx.mstaged ? cx.smask + (seg & 1) * cx.mbuf + (size_t)b * p.W : p.mask + ((size_t)s * p.max_active + b) * p.W;
}
// One elected thread: S[g mod 3] = Q K(stage)^T for every tile g.  A buffer's scores are replaced in place by the
// weights P, so it is free again when the multiplication P V of tile g - 3 has completed.
__device__ __forceinline__ void qk_loop(const AttnParams& p, const Ctx& cx, long long lo, long long hi)
{
    const uint64_t k_desc0 = smem_desc(smem_u32(cx.kring), 16, 1024);
    const uint32_t k_lo0 = (uint32_t)k_desc0, k_hi = (uint32_t)(k_desc0 >> 32);
    const uint32_t idesc = instr_desc(MROWS, TILE, 0);
    int s = 0;
    uint32_t g = 0, seg = 0;
    int st = 0;
    uint32_t kph = 0;                               // ring position and phase of the K stage of tile g
    long long u = lo;
    bool good = true;
    while (u < hi && good) {
        const Segment sg = decode_segment(u, hi, cx.pre, p.hkv, s);
        const int ntile = sg.j1 - sg.j0;
        good = mbar_wait_warp(cx.q_ready(), seg & 1, cx.abortp, p.status);
        for (int t = 0; t < ntile && good; ++t, ++g) {
            good = mbar_wait(cx.k_full() + 8 * st, kph, cx.abortp, p.status);
            if (good && g >= NBUF) good = mbar_wait(cx.pv_done() + 8 * ((g - NBUF) % NBAR), ((g - NBUF) / NBAR) & 1, cx.abortp, p.status);
            good = __all_sync(0xffffffffu, good);
            if (!good) break;
            tc_fence_after();
            if (elect_one()) {
                const uint32_t kd = k_lo0 + (uint32_t)((st * STAGE) >> 4), d = cx.tmem + TM_S + (g % NBUF) * TILE;
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks)
                    umma_ts(d, cx.tmem + ks * 8, kd + (uint32_t)(((ks >> 2) * PANEL + (ks & 3) * 32) >> 4), k_hi, idesc, ks > 0);
                umma_commit(cx.k_empty() + 8 * st);
                umma_commit(cx.s_full() + 8 * (g % NBAR));
            }
            __syncwarp();
            if (++st == cx.nk) {
                st = 0;
                kph ^= 1;
            }
        }
        ++seg;
        u = sg.next_u;
    }
}

// One elected thread: O[g & 1] += P V(stage) for every tile g, once the stage has landed and the tile's softmax
// warps have delivered P (and, beyond the prefix, cleared the stage's unseen rows).  The multiplication runs in steps
// of 16 KV rows; the softmax warps say which steps hold a visible row, the others are left out.
__device__ __forceinline__ void pv_loop(const AttnParams& p, const Ctx& cx, long long lo, long long hi)
{
    const uint64_t v_desc0 = smem_desc(smem_u32(cx.vring), PANEL, 1024);
    const uint32_t v_lo0 = (uint32_t)v_desc0, v_hi = (uint32_t)(v_desc0 >> 32);
    const uint32_t idesc = instr_desc(MROWS, D, 1);
    int s = 0;
    uint32_t g = 0, seg = 0;
    int st = 0;
    uint32_t vph = 0;
    long long u = lo;
    bool good = true;
    while (u < hi && good) {
        const Segment sg = decode_segment(u, hi, cx.pre, p.hkv, s);
        const int ntile = sg.j1 - sg.j0, npre = prefix_tiles(sg, cx.npre);
        uint32_t begun = 0;                         // groups whose accumulator holds something of this segment
        for (int t = 0; t < ntile && good; ++t, ++g) {
            const uint32_t b = g % NBAR, grp = g & 1;
            good = mbar_wait(cx.v_full() + 8 * st, vph, cx.abortp, p.status);
            if (good) good = mbar_wait(cx.p_full() + 8 * b, (g / NBAR) & 1, cx.abortp, p.status);
            if (good && t == 0 && seg > 0) good = mbar_wait(cx.o_free(), (seg - 1) & 1, cx.abortp, p.status);
            good = __all_sync(0xffffffffu, good);
            if (!good) break;
            const uint32_t steps = t < npre ? 0xfu : (uint32_t)cx.v_steps[b];      // (all steps of a prefix tile)
            tc_fence_after();
            if (elect_one()) {
                const uint32_t vd = v_lo0 + (uint32_t)((st * STAGE) >> 4), od = cx.tmem + TM_O + grp * 128, pa = cx.tmem + TM_S + (g % NBUF) * TILE;
                uint32_t acc = (begun >> grp) & 1u;
                if (steps == 0xfu) {
#pragma unroll
                    for (int kk = 0; kk < TILE / 16; ++kk) umma_ts(od, pa + kk * 8, vd + kk * 128, v_hi, idesc, kk > 0 ? 1u : acc);
                } else {
#pragma unroll
                    for (int kk = 0; kk < TILE / 16; ++kk)
                        if ((steps >> kk) & 1u) {
                            umma_ts(od, pa + kk * 8, vd + kk * 128, v_hi, idesc, acc);
                            acc = 1u;
                        }
                }
                umma_commit(cx.v_empty() + 8 * st);
                umma_commit(cx.pv_done() + 8 * b);
            }
            __syncwarp();
            if (steps) begun |= 1u << grp;
            if (++st == cx.nv) {
                st = 0;
                vph ^= 1;
            }
        }
        ++seg;
        u = sg.next_u;
    }
}

// A pair's queries go to tensor memory (lane = query row, 64 columns of bf16 pairs: the row as it is in memory), from
// where they are the A operand of all the pair's Q K^T: shared memory serves K alone.  Called by the 128 threads of
// one group; rows past the pair's last are zero up to the next multiple of 32, and left as they are beyond that
// (their results are never looked at).
__device__ __noinline__ void load_queries(const uint4* qg, int max_active, int hq, int G, int s, int g, int M, int row, uint32_t taddr)
{
    if ((row & ~31) >= M) return;                  // (uniform over the warp)
    const int b = row < M ? row / G : 0, hg = row < M ? row - b * G : 0;
    const uint4* src = qg + ((((size_t)s * max_active + b) * hq + (size_t)g * G + hg) * D) / 8;
    uint32_t w[2][32];
#pragma unroll
    for (int i = 0; i < 8; ++i) {                  // whole 32-byte sectors (q may be no more than 16-byte aligned: then two halves)
        uint32_t* x = &w[i >> 2][(i & 3) * 8];
        if (row >= M) {
            x[0] = x[1] = x[2] = x[3] = x[4] = x[5] = x[6] = x[7] = 0u;
        } else if (!((uintptr_t)qg & 31)) {
            asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                         : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]), "=r"(x[5]), "=r"(x[6]), "=r"(x[7])
                         : "l"(src + 2 * i)
                         : "memory");
        } else {
            const uint4 a = __ldcg(src + 2 * i), b2 = __ldcg(src + 2 * i + 1);
            x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
            x[4] = b2.x; x[5] = b2.y; x[6] = b2.z; x[7] = b2.w;
        }
    }
    tmem_st<32>(taddr, w[0]);
    tmem_st<32>(taddr + 32, w[1]);
    tmem_wait_st();
}
// The scene's bitmaps, asynchronous (128 threads; completed with cp_async_wait_all).
__device__ __forceinline__ void stage_bitmaps(const uint64_t* mask, int max_active, int W, int s, uint64_t* dst, int tid)
{
    const uint64_t* src = mask + (size_t)s * max_active * W;
    for (int idx = tid; idx < max_active * W; idx += 128) cp_async8(dst + idx, src + idx);
}
// The first pair when the kernel runs ahead of the dependency wait: the queries may still be written by the
// kernel ahead, so their lines are only requested into L2 (which stays coherent).
__device__ __noinline__ void request_pair(const uint4* qg, int max_active, int hq, int G, int s, int g, int M, int tid)
{
    for (int idx = tid * 8; idx < M * (D / 8); idx += 128 * 8) {             // one request per 128-byte line
        const int n = idx / (D / 8), ch = idx - n * (D / 8);
        const int bb = n / G, hg = n - bb * G;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(qg + ((((size_t)s * max_active + bb) * hq + (size_t)g * G + hg) * D) / 8 + ch));
    }
}

// Merge of the partials of one (scene, KV head) pair by the CTA that delivered the last one
// (all softmax threads).  Every thread owns eight accumulator columns of MI query rows at a time and merges
// the parts' (m, l, O) for them in ONE pass, MB parts per turn with all loads ahead of the
// arithmetic (a turn costs one trip to L2, so it carries as many rows and parts as registers allow; the running
// maximum is carried like in the online softmax, so more parts need no second pass):
//     m = max_c m_c,  l = sum_c l_c 2^(m_c - m),  O = sum_c O_c 2^(m_c - m) / l.
// Out of line, arguments by value.
__device__ __noinline__ void merge_pair(const float* ws_ml, const float* ws_o, __nv_bfloat16* out, int pair, int mmax, int M, int G, int s, int g,
                                        int max_active, int hq, int c_first, int c_last)
{
    constexpr int MB = 3, MI = 4, RSTEP = NSOFT * 32 / (D / 8);    // rows between a thread's items
    const int c8 = threadIdx.x % (D / 8), r0 = threadIdx.x / (D / 8);
    for (int mb = r0; mb < M; mb += MI * RSTEP) {
        float acc[MI][8], mx[MI], lt[MI];
#pragma unroll
        for (int i = 0; i < MI; ++i) {
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[i][e] = 0.f;
            mx[i] = -INFINITY;
            lt[i] = 0.f;
        }
        for (int c0 = c_first; c0 <= c_last; c0 += MB) {
            float2 v[MI][MB];
            float o[MI][MB][8];
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int j = 0; j < MB; ++j) {
                    const int m = mb + i * RSTEP;
                    const bool on = m < M && c0 + j <= c_last;
                    const size_t at = (size_t)(pair + c0 + j) * mmax + m;
                    v[i][j] = make_float2(-INFINITY, 0.f);
#pragma unroll
                    for (int e = 0; e < 8; ++e) o[i][j][e] = 0.f;
                    if (on) {
                        v[i][j] = __ldcg(reinterpret_cast<const float2*>(ws_ml) + at);
                        asm volatile("ld.global.cg.v4.f32 {%0,%1,%2,%3}, [%8];\n\tld.global.cg.v4.f32 {%4,%5,%6,%7}, [%8+16];"
                                     : "=f"(o[i][j][0]), "=f"(o[i][j][1]), "=f"(o[i][j][2]), "=f"(o[i][j][3]), "=f"(o[i][j][4]), "=f"(o[i][j][5]), "=f"(o[i][j][6]),
                                       "=f"(o[i][j][7])
                                     : "l"(ws_o + at * D + c8 * 8)
                                     : "memory");
                    }
                }
#pragma unroll
            for (int i = 0; i < MI; ++i) {
                float nm = mx[i];
#pragma unroll
                for (int j = 0; j < MB; ++j) nm = fmaxf(nm, v[i][j].x);
                const float sc = mx[i] == nm ? 1.f : fast_exp2(mx[i] - nm);           // (-inf) - (-inf) must not be formed
                lt[i] *= sc;
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[i][e] *= sc;
#pragma unroll
                for (int j = 0; j < MB; ++j) {
                    const float w = v[i][j].x == -INFINITY ? 0.f : fast_exp2(v[i][j].x - nm);   // a part that saw nothing
                    lt[i] = fmaf(v[i][j].y, w, lt[i]);
#pragma unroll
                    for (int e = 0; e < 8; ++e) acc[i][e] = fmaf(o[i][j][e], w, acc[i][e]);
                }
                mx[i] = nm;
            }
        }
#pragma unroll
        for (int i = 0; i < MI; ++i) {
            const int m = mb + i * RSTEP;
            if (m < M) {
                const float inv = 1.f / lt[i];
                const int b = m / G, hg = m - b * G;
                *reinterpret_cast<uint4*>(out + (((size_t)s * max_active + b) * hq + (size_t)g * G + hg) * D + c8 * 8) =
                    make_uint4(pack2(acc[i][0] * inv, acc[i][1] * inv), pack2(acc[i][2] * inv, acc[i][3] * inv), pack2(acc[i][4] * inv, acc[i][5] * inv),
                               pack2(acc[i][6] * inv, acc[i][7] * inv));
            }
        }
    }
}

// Two fp32 operations in one instruction.
__device__ __forceinline__ uint64_t pair2(float lo, float hi)
{
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ float2 halves2(uint64_t x)
{
    float2 v;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(x));
    return v;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// The accumulator of a row whose reference moves from m to a higher one: times a.
__device__ __forceinline__ void rescale_row(const uint32_t o_addr, const float a)
{
#pragma unroll 1
    for (int k = 0; k < D; k += 16) {
        uint32_t ov[16];
        tmem_ld<16>(o_addr + k, ov);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 16; ++i) ov[i] = __float_as_uint(__uint_as_float(ov[i]) * a);
        tmem_st<16>(o_addr + k, ov);
    }
}
// One tile (64 KV rows) of one query row: the scores leave TMEM, the weights take their place (bf16 pairs in the first
// 32 columns of the buffer).  o_addr: the row's accumulator; settled() returns when no multiplication is in flight on it.
//
// Prefix tiles: the weights are made with the row's present reference while the maximum is taken; where it turns out too
// low the reference is raised and the weights are made once more.
template <class F>
__device__ __forceinline__ void softmax_tile(const uint32_t s_addr, const uint32_t o_addr, const float c, float& m, float& l, const bool begun, F&& settled)
{
    if (__any_sync(0xffffffffu, m == -INFINITY)) {
        // a row that has not seen anything yet takes the maximum of this tile's scores
        float x = -INFINITY;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            uint32_t sv[32];
            tmem_ld<32>(s_addr + k * 32, sv);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 32; ++i) x = fmaxf(x, __uint_as_float(sv[i]));
        }
        if (m == -INFINITY) m = x * c;
    }
    uint32_t pk[2][16];
    float lr;
#pragma unroll 1
    for (;;) {
        uint32_t sv[2][32];
        tmem_ld<32>(s_addr, sv[0]);
        tmem_ld<32>(s_addr + 32, sv[1]);
        const float nm = m == -INFINITY ? 0.f : -m;
        const uint64_t c2 = pair2(c, c), nm2 = pair2(nm, nm);
        uint64_t l2 = 0ull;
        float x0 = -INFINITY, x1 = -INFINITY;
        tmem_wait_ld();
#pragma unroll
        for (int k = 0; k < 2; ++k) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float a = __uint_as_float(sv[k][2 * i]), b = __uint_as_float(sv[k][2 * i + 1]);
                if (i & 1) x1 = fmaxf(fmaxf(x1, a), b);
                else x0 = fmaxf(fmaxf(x0, a), b);
                const float2 t = halves2(fma2(pair2(a, b), c2, nm2));
                pk[k][i] = pack2(fast_exp2(t.x), fast_exp2(t.y));
                l2 = add2(l2, pair2(__uint_as_float(pk[k][i] << 16), __uint_as_float(pk[k][i] & 0xffff0000u)));      // the rounded values
            }
        }
        const float2 lh = halves2(l2);
        const float l0 = lh.x, l1 = lh.y;
        lr = l0 + l1;
        const float mx = fmaxf(x0, x1) * c;
        const bool raise = mx > m + RAISE_LOG2;        // (no score: mx = m = -inf)
        if (!__any_sync(0xffffffffu, raise)) break;
        const float mn = raise ? mx : m;
        const float a = raise ? fast_exp2(m - mn) : 1.f;
        l *= a;
        m = mn;
        if (begun) {
            settled();
            rescale_row(o_addr, a);
        }
    }
    l += lr;
    tmem_st<16>(s_addr, pk[0]);
    tmem_st<16>(s_addr + 16, pk[1]);
    tmem_wait_st();
}
// Tiles beyond the prefix, w = the KV rows that this query row sees.  Few rows of the warp see the tile, as a rule those of one
// field, and of the tile only the part that has been decoded: the maximum comes first, so that no pass is made twice (a row's
// first scores, or a higher reference, are the usual case here), and 16 KV rows that nobody in the warp sees get weights of 0
// without an exponential (a warp's 64 exponentials a thread are 512 cycles of its MUFU pipe).  Measured, 32 / 8 heads, 32 fields, 8 scenes, prefix
// 1024, us a layer with one loop for both kinds of tile / with this one: 40.8 / 39.2.
template <class F>
__device__ __forceinline__ void softmax_tile_masked(const uint32_t s_addr, const uint32_t o_addr, const uint64_t w, const float c, float& m, float& l,
                                                    const bool begun, F&& settled)
{
    uint32_t sv[2][32];
    tmem_ld<32>(s_addr, sv[0]);
    tmem_ld<32>(s_addr + 32, sv[1]);
    const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)w), hi = __reduce_or_sync(0xffffffffu, (uint32_t)(w >> 32));
    float x0 = -INFINITY, x1 = -INFINITY;
    tmem_wait_ld();
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const uint32_t bits = (uint32_t)(w >> (k * 32));
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (((k ? hi : lo) >> (h * 16)) & 0xffffu) {              // (uniform)
#pragma unroll
                for (int i = h * 16; i < h * 16 + 16; i += 2) {
                    if (!((bits >> i) & 1u)) sv[k][i] = 0xff800000u;
                    if (!((bits >> (i + 1)) & 1u)) sv[k][i + 1] = 0xff800000u;
                    x0 = fmaxf(x0, __uint_as_float(sv[k][i]));
                    x1 = fmaxf(x1, __uint_as_float(sv[k][i + 1]));
                }
            }
    }
    const float mx = fmaxf(x0, x1) * c;
    const bool first = m == -INFINITY, raise = !first && mx > m + RAISE_LOG2;
    if (__any_sync(0xffffffffu, raise)) {
        const float mn = raise ? mx : m, a = raise ? fast_exp2(m - mn) : 1.f;
        l *= a;
        m = mn;
        if (begun) {
            settled();
            rescale_row(o_addr, a);
        }
    }
    if (first) m = mx;                                 // (a row that has not seen anything has weights of 0 so far)
    const float nm = m == -INFINITY ? 0.f : -m;
    const uint64_t c2 = pair2(c, c), nm2 = pair2(nm, nm);
    uint64_t l2 = 0ull;
    uint32_t pk[2][16];
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (((k ? hi : lo) >> (h * 16)) & 0xffffu) {
#pragma unroll
                for (int i = h * 8; i < h * 8 + 8; ++i) {
                    const float2 t = halves2(fma2(pair2(__uint_as_float(sv[k][2 * i]), __uint_as_float(sv[k][2 * i + 1])), c2, nm2));
                    pk[k][i] = pack2(fast_exp2(t.x), fast_exp2(t.y));
                    l2 = add2(l2, pair2(__uint_as_float(pk[k][i] << 16), __uint_as_float(pk[k][i] & 0xffff0000u)));      // the rounded values
                }
            } else {
#pragma unroll
                for (int i = h * 8; i < h * 8 + 8; ++i) pk[k][i] = 0u;
            }
        }
    const float2 lh = halves2(l2);
    l += lh.x + lh.y;
    tmem_st<16>(s_addr, pk[0]);
    tmem_st<16>(s_addr + 16, pk[1]);
    tmem_wait_st();
}
// No row of this warp sees anything in the tile: weights 0.
__device__ __forceinline__ void zero_weights(const uint32_t s_addr)
{
    uint32_t z[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) z[i] = 0u;
    tmem_st<32>(s_addr, z);
    tmem_wait_st();
}

// The softmax warps' work on a CTA's run.  Warps 0-3 are group 0 and take the even tiles, warps 4-7 group 1 and the odd
// ones; a group has two S / P buffers, an accumulator and (m, l) of its own, so the groups meet only at the ends of a
// segment.  Thread = one query row (TMEM lane) x all 64 KV rows of the tile.
//   m: the row's reference (in log2 units): the maximum of its first scores, raised only when a score exceeds it by
//      more than 2^8 (then l and the accumulator are rescaled);
//   l: the sum of the bf16-rounded weights that are multiplied with V.
__device__ __forceinline__ void softmax_loop(const AttnParams& p, const Ctx& cx, long long lo, long long hi, const int warp, const int lane)
{
    const int tid = threadIdx.x;                   // 0 .. NSOFT * 32 - 1
    const int grp = warp >> 2, q4 = warp & 3, gtid = tid & 127;
    const int row = q4 * 32 + lane;                // query row
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
    const uint32_t o_addr = cx.tmem + lane_base + TM_O + grp * 128;
    const float c = p.scale_log2;
    const int G = p.group;
    bool dead = false;                             // a bounded wait ran out somewhere in the CTA
    auto wait_u = [&](uint32_t bar, uint32_t parity) {    // warp-uniform outcome
        if (dead || __all_sync(0xffffffffu, mbar_try(bar, parity))) return;          // usually satisfied already
        if (!mbar_wait_slow(bar, parity, cx.abortp, p.status)) dead = true;
        dead = __any_sync(0xffffffffu, dead);
    };
    const uint4* qg = reinterpret_cast<const uint4*>(p.q);
    int s = 0;
    uint32_t g = 0, seg = 0;                       // tile (counted over all segments), segment
    long long u = lo;
    bool staged = false;                           // the segment's queries and bitmaps were staged and announced by the segment before
    while (u < hi) {
        const Segment sg = decode_segment(u, hi, cx.pre, p.hkv, s);
        const int A = cx.nact[sg.s], M = A * G;
        uint64_t* sm = cx.smask + (seg & 1) * cx.mbuf;
        if (!staged) {
            // (the first segment) group 0 stages the queries and the bitmaps
            if (grp == 0 && p.early) request_pair(qg, p.max_active, p.hq, G, sg.s, sg.g, M, gtid);
            if (p.early) asm volatile("griddepcontrol.wait;" ::: "memory");
            if (grp == 0) {
                if (cx.mstaged) stage_bitmaps(p.mask, p.max_active, p.W, sg.s, sm, gtid);
                load_queries(qg, p.max_active, p.hq, G, sg.s, sg.g, M, row, cx.tmem + lane_base);
                cp_async_wait_all();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(cx.q_ready());
            }
        }
        staged = false;
        // (first use of the bitmaps and of their OR: after the prefix)
        const uint64_t* un = (cx.mstaged && p.W <= UW) ? cx.sunion + (seg & 1) * UW : nullptr;
        const bool rows_here = q4 * 32 < M;        // this warp has query rows
        const uint64_t* words = mask_row(p, cx, seg, sg.s, row < M ? row / G : 0);
        const int ntile = sg.j1 - sg.j0;
        float m = -INFINITY, l = 0.f;
        bool begun = false;                        // the group's accumulator holds something of this segment
        uint32_t last = 0;                         // the group's last tile
        bool any_tile = false;
        const uint32_t g0 = g;                     // the segment's first tile
        const int npre = prefix_tiles(sg, cx.npre);      // whole prefix tiles come first in a list
        auto settled = [&]() {
            // the group's tile before this one (the ones before that are known to be done)
            wait_u(cx.pv_done() + 8 * (last % NBAR), (last / NBAR) & 1);
            tc_fence_after();
        };
        int t = (int)((g0 ^ (uint32_t)grp) & 1u);  // the group's tiles are t, t + 2, ...
        const int32_t* ids = p.tiles + (size_t)sg.s * p.ntile_max + (tile_entry(sg, npre) - npre);
        int id0 = npre + lane;                     // ids of the tiles beyond the prefix, a warp's width at a time
        int my_tile = id0 < ntile ? ids[id0] : 0;
#pragma unroll 1
        for (; t < npre; t += 2) {
            const uint32_t gt = g0 + (uint32_t)t, b = gt % NBAR;
            wait_u(cx.s_full() + 8 * b, (gt / NBAR) & 1);
            tc_fence_after();
            if (rows_here && !dead) softmax_tile(cx.tmem + lane_base + TM_S + (gt % NBUF) * TILE, o_addr, c, m, l, begun, settled);
            begun = true;
            last = gt;
            any_tile = true;
            tc_fence_before();
            __syncwarp();
            if (!dead && lane == 0) mbar_arrive(cx.p_full() + 8 * b);
        }
        if (npre < ntile) {
            soft_sync();                           // the bitmaps are in place
            if (cx.mstaged && p.W <= UW) {
                // OR of the scene's bitmaps: the rows that some branch may see (the others are cleared in V)
                if (tid < p.W) {
                    uint64_t x = 0ull;
                    for (int b = 0; b < A; ++b) x |= sm[(size_t)b * p.W + tid];
                    cx.sunion[(seg & 1) * UW + tid] = x;
                }
                soft_sync();
            }
        }
#pragma unroll 1
        for (; t < ntile; t += 2) {
            const uint32_t gt = g0 + (uint32_t)t, b = gt % NBAR;
            if (t - (id0 - lane) >= 32) {
                id0 += 32;
                my_tile = id0 < ntile ? ids[id0] : 0;
            }
            const int tile = __shfl_sync(0xffffffffu, my_tile, t - (id0 - lane));
            // Eq. 1 for this thread's query row
            const uint64_t w = row < M ? tile_rowmask(words, p.W, p.P, tile) : 0ull;
            const bool some = __any_sync(0xffffffffu, w != 0ull);
            const uint64_t seen = tile_seen_rows(un, mask_row(p, cx, seg, sg.s, 0), p.W, p.P, A, tile);
            wait_u(cx.s_full() + 8 * b, (gt / NBAR) & 1);
            tc_fence_after();
            const uint32_t s_addr = cx.tmem + lane_base + TM_S + (gt % NBUF) * TILE;
            if (some && !dead) softmax_tile_masked(s_addr, o_addr, w, c, m, l, begun, settled);
            else if (rows_here && !dead) zero_weights(s_addr);
            // Rows that no branch of the scene may see can hold anything (NaN, Inf: slots that were never written), and
            // 0 * NaN must not reach the accumulator: steps of 16 KV rows without a visible row are left out of the
            // multiplication, in the others the unseen rows are cleared once the stage has landed (two threads of the
            // group a row).
            wait_u(cx.v_full() + 8 * (gt % (uint32_t)cx.nv), (gt / (uint32_t)cx.nv) & 1);
            const int r = gtid & (TILE - 1);
            const uint32_t step_seen = (uint32_t)(seen >> (r & 48)) & 0xffffu;
            if (!dead && step_seen != 0u && !((seen >> r) & 1ull)) {
                const uint32_t va = smem_u32(cx.vring) + (gt % (uint32_t)cx.nv) * STAGE + (uint32_t)(gtid / TILE) * PANEL + (uint32_t)r * 128;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(va + (uint32_t)((i + lane) & 7) * 16), "r"(0u) : "memory");
            }
            uint32_t steps = 0u;
#pragma unroll
            for (int i = 0; i < 4; ++i) steps |= ((seen >> (16 * i)) & 0xffffull) ? (1u << i) : 0u;
            if (steps) begun = true;
            last = gt;
            any_tile = true;
            if (gtid == 0) cx.v_steps[b] = (int)steps;
            // every thread orders its own TMEM accesses and shared-memory writes, then one lane per warp signals
            fence_async_smem();
            tc_fence_before();
            __syncwarp();
            if (!dead && lane == 0) mbar_arrive(cx.p_full() + 8 * b);
        }
        g = g0 + (uint32_t)ntile;
        // the whole tiles of the prefix come first in a tile list (entry j = tile j): everything above relies on it
        for (int j = tile_entry(sg, 0) + tid; j < tile_entry(sg, 0) + npre; j += NSOFT * 32)
            if (p.tiles[(size_t)sg.s * p.ntile_max + j] != j) atomicOr(p.status, FDC_DEV_TILE_LIST);
        // The group that does not have the segment's last tile asks for the next pair's queries and bitmaps meanwhile, puts
        // them in place once the last scores are complete and announces them, so that the next pair's Q K^T runs on
        // while this pair is finished off.  (The last tile's barrier is the other group's, but its phase before that
        // one is known to be over: the scores of the tile ahead of the last one, this group's, came after it.)
        if (sg.next_u < hi) {
            if ((int)((g - 1) & 1) != grp) {
                int s2 = sg.s;
                const Segment nx = decode_segment(sg.next_u, hi, cx.pre, p.hkv, s2);
                const int M2 = cx.nact[nx.s] * G;
                if (cx.mstaged) stage_bitmaps(p.mask, p.max_active, p.W, nx.s, cx.smask + ((seg + 1) & 1) * cx.mbuf, gtid);
                request_pair(qg, p.max_active, p.hq, G, nx.s, nx.g, M2, gtid);
                wait_u(cx.s_full() + 8 * ((g - 1) % NBAR), ((g - 1) / NBAR) & 1);
                tc_fence_after();
                if (!dead) load_queries(qg, p.max_active, p.hq, G, nx.s, nx.g, M2, row, cx.tmem + lane_base);
                cp_async_wait_all();
                tc_fence_before();
                __syncwarp();
                if (!dead && lane == 0) mbar_arrive(cx.q_ready());
            }
            staged = true;
        }
        // ---- end of segment: the two groups' results of a row are one row's result
        if (any_tile) wait_u(cx.pv_done() + 8 * (last % NBAR), (last / NBAR) & 1);
        tc_fence_after();
        cx.ml[grp * MROWS + row] = make_float2(begun ? m : -INFINITY, l);
        if (lane == 0 && q4 == 0) cx.merge[grp] = begun;
        soft_sync();
        if (TWO && half_of_pair(cx, sg, p.hkv) >= 0) break;           // (one part a CTA: the run's only segment)
        const float2 a0 = cx.ml[row], a1 = cx.ml[MROWS + row];
        const bool has0 = cx.merge[0] != 0, has1 = cx.merge[1] != 0;
        const float mx = fmaxf(a0.x, a1.x), ms = mx == -INFINITY ? 0.f : mx;
        const float f0 = fast_exp2(a0.x - ms), f1 = fast_exp2(a1.x - ms), lt = a0.y * f0 + a1.y * f1;
        soft_sync();                               // (merge[] is used again below)
        const int pair = sg.s * p.hkv + sg.g;
        const int slot = blockIdx.x + pair;
        const bool whole = sg.j0 == 0 && sg.j1 == sg.nt;   // this CTA saw every tile of the pair
        const bool direct = p.pair_cnt && whole;           // no other partial exists: normalise and write the output
        if (rows_here && !dead) {
            const float inv = direct ? 1.f / lt : 1.f, g0 = f0 * inv, g1 = f1 * inv;
            const int b = row / G, hg = row - b * G;
            __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(p.out) + (((size_t)sg.s * p.max_active + b) * p.hq + (size_t)sg.g * G + hg) * D;
            float* wo = p.ws_o + ((size_t)slot * p.mmax + row) * D;
            // group 0 takes the first half of the columns of both accumulators, group 1 the second
#pragma unroll 1
            for (int c0 = grp * (D / 2); c0 < (grp + 1) * (D / 2); c0 += 16) {
                uint32_t x[16], y[16];
                if (has0) tmem_ld<16>(cx.tmem + lane_base + TM_O + c0, x);
                if (has1) tmem_ld<16>(cx.tmem + lane_base + TM_O + 128 + c0, y);
                tmem_wait_ld();
                float v[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = (has0 ? __uint_as_float(x[i]) * g0 : 0.f) + (has1 ? __uint_as_float(y[i]) * g1 : 0.f);
                if (row < M) {
                    if (direct) {
#pragma unroll
                        for (int i = 0; i < 16; i += 8)
                            *reinterpret_cast<uint4*>(out + c0 + i) = make_uint4(pack2(v[i], v[i + 1]), pack2(v[i + 2], v[i + 3]), pack2(v[i + 4], v[i + 5]), pack2(v[i + 6], v[i + 7]));
                    } else {
#pragma unroll
                        for (int i = 0; i < 16; i += 8)          // whole 32-byte sectors
                            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(wo + c0 + i), "f"(v[i]), "f"(v[i + 1]), "f"(v[i + 2]), "f"(v[i + 3]),
                                         "f"(v[i + 4]), "f"(v[i + 5]), "f"(v[i + 6]), "f"(v[i + 7])
                                         : "memory");
                    }
                }
            }
            if (!direct && grp == 0 && row < M) *reinterpret_cast<float2*>(p.ws_ml + ((size_t)slot * p.mmax + row) * 2) = make_float2(mx, lt);
        }
        if (p.pair_cnt && !whole) {
            // the CTA that delivers the last partial of a pair merges them all (no second kernel)
            soft_sync();
            if (tid == 0) {
                __threadfence();                   // (everybody's stores: they came before the barrier)
                int c_first, c_last;
                pair_ctas(p, cx, sg.s, sg.g, c_first, c_last);
                const int expected = c_last - c_first + 1;               // every CTA in between owns tiles of the pair
                const int old = dead ? -1 : atomicAdd(&p.pair_cnt[pair], 1);
                cx.merge[0] = old == expected - 1;
                cx.merge[1] = c_first;
                cx.merge[2] = c_last;
                __threadfence();                   // (the other CTAs' partials are read after the barrier below, past L1)
                if (old == expected - 1) p.pair_cnt[pair] = 0;          // ready for the next call
            }
            soft_sync();
            if (cx.merge[0])
                merge_pair(p.ws_ml, p.ws_o, reinterpret_cast<__nv_bfloat16*>(p.out), pair, p.mmax, M, G, sg.s, sg.g, p.max_active, p.hq, cx.merge[1], cx.merge[2]);
        }
        soft_sync();                               // (merge[] and ml[] are free again)
        tc_fence_before();
        __syncwarp();
        if (!dead && lane == 0) mbar_arrive(cx.o_free());
        ++seg;
        u = sg.next_u;
    }
    if (!TWO || lo >= hi) return;
    // A pair in two parts: group `half` finishes its columns with what the other CTA's group of that number hands over (through the free K ring instead of
    // registers).
    s = 0;
    const Segment sg = decode_segment(lo, hi, cx.pre, p.hkv, s);
    const int half = half_of_pair(cx, sg, p.hkv), M = cx.nact[sg.s] * G, has = (cx.merge[0] ? 1 : 0) | (cx.merge[1] ? 2 : 0);
    if (half < 0) return;
    const float2 a0 = cx.ml[row], a1 = cx.ml[MROWS + row];
    const float m = fmaxf(a0.x, a1.x), ms = m == -INFINITY ? 0.f : m;
    float s0 = fast_exp2(a0.x - ms), s1 = fast_exp2(a1.x - ms);
    const float l = a0.y * s0 + a1.y * s1;
    if (q4 * 32 < M && !dead) {
        const int b = row < M ? row / G : 0, hg = row - b * G;
        const size_t slot = blockIdx.x + sg.s * p.hkv + sg.g;
        float* wo = p.ws_o + slot * p.mmax * D + (size_t)(grp * (D / 8) * p.mmax + row) * 4;      // [4 columns][query row][4]: a warp's accesses are whole lines
        float* wml = p.ws_ml + (slot * p.mmax + row) * 2;
        float4* mine = reinterpret_cast<float4*>(cx.kring) + row;
        float s2 = 0.f;
        bool ok = true;
        if (grp == half) {
            ok = wait_for_peer(cx.peer_done(), cx.abortp, p.status);
            const long long other = half ? -(long long)p.mmax : (long long)p.mmax;                // to the other CTA's slot, in rows
            if (ok && row < M) {
#pragma unroll 4
                for (int i = 0; i < D / 8; ++i)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(mine + i * MROWS)), "l"(wo + other * D + (size_t)i * p.mmax * 4) : "memory");
                const float2 v = __ldcg(reinterpret_cast<const float2*>(wml + other * 2));
                const float nm = fmaxf(m, v.x), nms = nm == -INFINITY ? 0.f : nm, a = fast_exp2(m - nms), w = fast_exp2(v.x - nms);     // (a part that saw nothing: 0)
                const float inv = 1.f / fmaf(v.y, w, l * a);
                s0 *= a * inv;
                s1 *= a * inv;
                s2 = w * inv;
            }
            cp_async_wait_all();
        } else if (row < M) {
            *reinterpret_cast<float2*>(wml) = make_float2(m, l);
        }
        __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(p.out) + (((size_t)sg.s * p.max_active + b) * p.hq + (size_t)sg.g * G + hg) * D + grp * (D / 2);
        const uint32_t o0 = o_addr - grp * 128 + grp * (D / 2);
#pragma unroll 1
        for (int c0 = 0; c0 < D / 2 && ok; c0 += 16) {
            uint32_t x[16], y[16];
            if (has & 1) tmem_ld<16>(o0 + c0, x);
            if (has & 2) tmem_ld<16>(o0 + 128 + c0, y);
            tmem_wait_ld();
            float v[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = ((has & 1) ? __uint_as_float(x[i]) * s0 : 0.f) + ((has & 2) ? __uint_as_float(y[i]) * s1 : 0.f);
            if (row < M && grp != half) {
#pragma unroll
                for (int i = 0; i < 16; i += 4)
                    *reinterpret_cast<float4*>(wo + (size_t)((c0 + i) / 4) * p.mmax * 4) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
            } else if (row < M) {
#pragma unroll
                for (int i = 0; i < 16; i += 4) {
                    const float4 z = mine[(c0 + i) / 4 * MROWS];
                    v[i] = fmaf(z.x, s2, v[i]);
                    v[i + 1] = fmaf(z.y, s2, v[i + 1]);
                    v[i + 2] = fmaf(z.z, s2, v[i + 2]);
                    v[i + 3] = fmaf(z.w, s2, v[i + 3]);
                }
#pragma unroll
                for (int i = 0; i < 16; i += 8)
                    *reinterpret_cast<uint4*>(out + c0 + i) = make_uint4(pack2(v[i], v[i + 1]), pack2(v[i + 2], v[i + 3]), pack2(v[i + 4], v[i + 5]), pack2(v[i + 6], v[i + 7]));
            }
        }
    }
    if (grp != half) {
        __threadfence();
        __syncwarp();
        if (!dead && lane == 0) arrive_at_peer(cx.peer_done());
    }
}
__global__ void __launch_bounds__(THREADS, 1)
FDC_TC_KERNEL(const AttnParams p, const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
               const int nk, const int nv, const int split_only)
{
    extern __shared__ unsigned char smem_dyn[];
    unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    Ctx cx;
    cx.nk = nk;
    cx.nv = nv;
    cx.kring = smem;
    cx.vring = cx.kring + (size_t)nk * STAGE;
    uint64_t* bars = reinterpret_cast<uint64_t*>(cx.vring + (size_t)nv * STAGE);
    cx.bar0 = smem_u32(bars);
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 4 * MAXST + 3 * NBAR + 6);
    cx.ml = reinterpret_cast<float2*>(tmem_holder + 4);
    cx.pre = reinterpret_cast<int*>(cx.ml + 2 * MROWS);
    cx.nact = cx.pre + p.batch + 1;
    cx.prev = cx.nact + p.batch;
    cx.smask = reinterpret_cast<uint64_t*>(((uintptr_t)(cx.prev + p.batch + 1) + 15) & ~(uintptr_t)15);
    cx.mbuf = MBUF;
    cx.sunion = cx.smask + 2 * cx.mbuf;
    cx.mstaged = p.max_active * p.W <= cx.mbuf;
    __shared__ CtaFlags cta_flags;
    cx.abortp = &cta_flags.abort_flag;
    cx.v_steps = cta_flags.v_steps;
    cx.merge = cta_flags.merge;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        cta_flags.abort_flag = 0;
    }
    SplitFinder<THREADS> split(p, split_only);
    if (p.early) split.issue(p);
    // ---- set-up that needs no global memory: barriers, TMEM
    if (threadIdx.x == 0) {
        for (int i = 0; i < MAXST; ++i) {
            mbar_init(cx.k_full() + 8 * i, 1);
            mbar_init(cx.k_empty() + 8 * i, 1);
            mbar_init(cx.v_full() + 8 * i, 1);
            mbar_init(cx.v_empty() + 8 * i, 1);
        }
        for (int i = 0; i < NBAR; ++i) {
            mbar_init(cx.s_full() + 8 * i, 1);
            mbar_init(cx.p_full() + 8 * i, NSOFT / 2);       // the warps of the tile's group
            mbar_init(cx.pv_done() + 8 * i, 1);
        }
        mbar_init(cx.q_ready(), NSOFT / 2);
        mbar_init(cx.o_free(), NSOFT);
        mbar_init(cx.app_done(), 1);
        mbar_init(cx.peer_done(), NSOFT / 2);        // the group that hands over
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_smem();
    }
    if (warp == W_QK && !split_only) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)), "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    if (TWO) cluster_arrive();
    tc_fence_after();
    const uint32_t tmem = split_only ? 0u : *reinterpret_cast<volatile uint32_t*>(tmem_holder);
    cx.tmem = tmem;
    // Programmatic dependent launch: this grid may have been scheduled while the kernel before it in
    // the stream was still running, and the kernel after this one may be scheduled early in the same
    // way.  Ordinarily nothing of global memory is touched before the kernel ahead has completed, and
    // only then is the next one let in.  With p.early the host vouches that the pass tables (counts,
    // tile lists, bitmaps), the work split and the prefix rows of the cache were complete before the
    // kernel ahead even began: then the work split is looked up and the first K/V stages of the prefix
    // are requested right away, while that kernel's last blocks are still running, and only what it
    // may have written (queries, the pass's new K/V rows, the rows beyond the prefix) waits for it.
    // Every thread passes the wait before the block ends, so grids complete in stream order.
    if (!p.early) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (!p.early) split.issue(p);
    long long lo = 0, hi = 0;
    bool active = split.find(p, cx, split_only, lo, hi);
    if (TWO) cluster_wait();
    // Two roles run ahead of the dependency wait (with p.early): the TMA producer, which takes the wait
    // itself once nothing more of the prefix can be requested, and the softmax warps, which first stage
    // the first pair's bitmaps.
    if (p.early && !(active && (warp == W_PROD || warp < NSOFT))) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!active) {
    } else if (warp == W_PROD) {
        producer_loop<1>(p, cx, &tm_k, &tm_v, lo, hi, lane);
    } else if (warp == W_AUX) {
        if (p.app_row) {
            append_rows<16>(const_cast<char*>(reinterpret_cast<const char*>(p.k)), const_cast<char*>(reinterpret_cast<const char*>(p.v)), p.stride_scene * 2,
                        p.stride_head * 2, p.stride_row * 2, p.app_row, reinterpret_cast<const char*>(p.app_k), reinterpret_cast<const char*>(p.app_v), p.tiles,
                        p.ntile_max, p.max_active, p.hkv, p.rows, p.P, cx.pre, cx.nact, lo, hi, p.status);
            if (lane == 0) mbar_arrive(cx.app_done());
        }
    } else if (warp == W_PV) {
        pv_loop(p, cx, lo, hi);
    } else if (warp == W_QK) {
        qk_loop(p, cx, lo, hi);
    } else {
        softmax_loop(p, cx, lo, hi, warp, lane);
    }
    // ---- teardown: everybody is done with TMEM before it is freed
    tc_fence_before();
    __syncthreads();
    if (warp == W_QK && !split_only) {
        // TMEM is freed only when no multiplication can still be writing it.  In an orderly run they were
        // all seen to complete before the last result was written.  After a wait that ran out, some may
        // still be on their way: their operands are all on chip, so they finish within microseconds, and
        // the block lingers for about a hundred before it lets go of TMEM.
        if (*cx.abortp)
            for (int i = 0; i < 100; ++i) __nanosleep(1000);
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
    if (TWO) {
        cluster_arrive();
        cluster_wait();
    }
}

}  // namespace

namespace fdc {

// bf16, head_dim 128, at most 128 query rows per (scene, KV head); FDC_ERR_SHAPE otherwise (the
// caller then takes another kernel).  split_only: the launch only computes the work split of the
// pass into p.split_memo (an ordinary launch; no rings, no TMEM).
int FDC_TC_LAUNCH(const AttnParams& p, int head_dim, cudaStream_t st, int split_only)
{
    if (head_dim != D || p.mmax > MROWS) return FDC_ERR_SHAPE;
    const size_t fixed = 1024 + 8 * (4 * MAXST + 3 * NBAR + 6) + 16 + 8 * 2 * MROWS + sizeof(int) * (3 * p.batch + 2) +
                         8 * (2 * MBUF + 2 * UW + 2) + 64;
    int stages = (int)((227 * 1024 - 256 - fixed) / STAGE);
    if (stages > 2 * MAXST) stages = 2 * MAXST;
    if (stages < 2 * NBUF) return FDC_ERR_SHAPE;  // (a V stage's use before is known to be over when its next one is waited for: NBUF of them at least)
    static SmemLimit limit;
    int rc = FDC_OK;
    if (TWO) {
        static PairsPlaceable placeable;
        rc = placeable.all(reinterpret_cast<const void*>(FDC_TC_KERNEL), THREADS, fixed + (size_t)stages * STAGE, p.n_cta, limit);
        if (rc) return rc;
    }
    if (split_only) stages = 0;
    const int nk = stages / 2, nv = stages - nk;
    const size_t smem = fixed + (size_t)stages * STAGE;
    alignas(64) CUtensorMap tk, tv;
    rc = get_kv_tensor_map(p.k, p, FDC_BF16, D, TILE, &tk);
    if (rc) return rc;
    rc = get_kv_tensor_map(p.v, p, FDC_BF16, D, TILE, &tv);
    if (rc) return rc;
    rc = raise_dynamic_smem(reinterpret_cast<const void*>(FDC_TC_KERNEL), smem, limit);
    if (rc) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.n_cta);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = split_only ? 0 : 1;
    if (TWO && !split_only) at[cfg.numAttrs++] = cluster_of_two();
    cudaError_t e = cudaLaunchKernelEx(&cfg, FDC_TC_KERNEL, p, tk, tv, nk, nv, split_only);
    if (e != cudaSuccess) return set_cuda_error(e);
    note_launch();
    return FDC_OK;
}

}  // namespace fdc
