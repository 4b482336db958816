// Split-KV pass for bf16 caches (head_dim 128) on the 5th-generation tensor cores (tcgen05 + TMEM).
// This file is the whole kernel and its launcher, for pairs of up to 64 query rows; it is compiled by the translation
// units that include it with FDC_TC_NGRP = 1 and 2 (the number of groups the softmax warps work
// in, see softmax_segment), and for two groups once more with FDC_TC_TWO (pairs in two parts, fdc_tc_common.cuh), so that each
// build holds only its own inner loop and gets its own register allocation.
//
// Sec. 3.3: the queries of all parallel fields of a scene, times the GQA heads of a KV head,
// share ONE read of the KV rows.  The kernel is written in the transposed form, with the KV
// rows on the M side of the MMAs and the (few) query rows on the N side, so that the tensor
// work scales with the real number of queries and every TMEM lane / softmax thread owns a
// real KV row:
//     S^T = K Q^T      M = 128 KV rows (one "round" = two 64-row tiles of the visited-tile
//                      list), N = NP query rows (32/64), K = head_dim;  A = the K tiles
//                      as TMA left them in shared memory, B = Q^T staged once per segment
//     O^T += V^T P^T   M = head_dim, N = NP, K = 128 KV rows;  A = the V tiles (M-major), B =
//                      P^T written by the softmax threads (N-major), accumulator in TMEM
//     l   += P 1       M = 128 query columns, N = 16 columns of ones, K = 128 KV rows: the
//                      softmax denominators, from the same bf16 P^T as the line above
// One persistent CTA per SM, 20 warps:
//   warp 16      TMA producer of both rings (K stages and V stages: 128 rows, 128B swizzle, L2
//                evict-first); polls both rings' free barriers, never blocks on one of them
//   warp 17      issues S^T = K Q^T (one elected thread); allocates / frees TMEM.  S^T has four
//                buffers in TMEM, so K Q^T runs ahead of the softmax
//   warp 18      with fdc_set_fused_append, first writes the pass's new K/V rows that fall into
//                this CTA's tiles; then issues the column-sum multiplications (one elected thread)
//   warp 19      issues O^T += V^T P^T (one elected thread)
//   warps 0-15   softmax.  Thread = one KV row of the round (TMEM lane) x a quarter (one group) or
//                a half (two groups) of the query columns.  Eq. 1 is applied by select from the
//                branches' row bitmaps; prefix tiles skip it.  Beyond the prefix the same threads
//                clear the V rows that no branch may see (they can hold anything, NaN included,
//                and 0 * NaN must not reach the accumulator) before they hand P^T over.
// The softmax reference of a query column is set in the first round of a segment: inside the
// prefix from the score against the round's first row (visible to everybody), else from the
// column maximum (a column that sees no row yet borrows the round's highest maximum).  A score
// more than 2^16 above its reference leaves a note that all warps act on two or three rounds
// later (no barrier in the common path); a rise of more than 2^100 within those rounds is
// flagged.  Sums and accumulator use the same reference and the same rounded P^T, so the result
// is exact up to the rounding of P^T.
#if !defined(FDC_TC_NGRP) || !defined(FDC_TC_NPMAX)
#error "include from a translation unit that defines FDC_TC_NGRP (1 or 2), FDC_TC_NPMAX (32 or 64), FDC_TC_TWO (0 or 1), FDC_TC_KERNEL and FDC_TC_LAUNCH"
#endif
#include "fdc_tc_common.cuh"

namespace {

constexpr int RROWS = 2 * TILE;              // KV rows per round = M of S^T = K of O^T
constexpr int NGRP = FDC_TC_NGRP;            // groups the softmax warps work in (this build)
constexpr int NP_MAX = FDC_TC_NPMAX;         // padded query rows of the widest pair of the launches this build serves (32 or 64)
static_assert((NP_MAX == 64) == (NGRP == 2), "two groups exactly for 33 to 64 query rows");
constexpr int NSOFT = 16;                    // softmax warps: 4 row quadrants x 4 column parts
constexpr int NPART = NSOFT / 4;             // column parts
constexpr int W_PROD = NSOFT, W_QK = NSOFT + 1, W_AUX = NSOFT + 2, W_PV = NSOFT + 3;
constexpr int THREADS = (NSOFT + 4) * 32;
constexpr uint32_t TMEM_COLS = 512;          // S^T buffers [0,256): 4 x 64 columns | O^T [256,384) | sums [384,512)
constexpr uint32_t TM_O = 256;
constexpr uint32_t TM_L = 384;                // column sums [384, 400): accumulator of the multiplication by ones (lane n: query column n)
constexpr int PANEL = RROWS * 128;           // 128 rows x 128 bytes (64 bf16 columns)
constexpr int ONES_BYTES = 2048;             // B operand of the column-sum multiplication: 16 x 16 bf16 ones (the footprint of its layout)
constexpr int STAGE = (D / 64) * PANEL;      // one K (or V) stage: 128 rows x head_dim
constexpr int MAXST = 4;                     // stages per ring at most
constexpr float RAISE_LOG2 = 16.f;
constexpr float UNSET = 1.0e30f;             // -reference of a column that has seen nothing yet
constexpr int MBUF = 512;                    // bitmap words of a scene kept in shared memory (max_active * W): one buffer

// Instruction descriptor of kind::f16: fp32 accumulate, bf16 A and B, M x N; mn_major = 1 makes
// BOTH operands MN-major (contiguous along M resp. N), 0 makes both K-major.
__device__ __forceinline__ uint32_t instr_desc(int m, int n, uint32_t mn_major)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (mn_major << 15) | (mn_major << 16) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(m >> 4) << 24);
}
// One MMA (cta_group::1, kind::f16).  The descriptors are given as (low, high) words: the address
// field sits in the low word, so stepping through an operand is 32-bit arithmetic for the issuing thread.
__device__ __forceinline__ void umma2(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t idesc,
                                      uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\tsetp.ne.b32 p, %6, 0;\n\tmov.b64 da, {%1, %2};\n\tmov.b64 db, {%3, %4};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %5, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Barrier of the softmax warps (a named barrier).  Every call site is reached by all sixteen warps
// the same number of times whatever happens: a warp whose bounded wait ran out goes on without
// waiting but still takes every one of these.
__device__ __forceinline__ void soft_sync() { asm volatile("bar.sync 1, %0;" ::"n"(NSOFT * 32) : "memory"); }

// The barrier inside the reference-raising path.  Whether a warp enters that path in a given round
// depends on data (a note left two or three rounds earlier), which a warp that no longer waits for anything
// may read too early; a named barrier there could then be waited at for ever.  So this one is an
// mbarrier with a bounded wait, one arrival per warp: the worst a straying warp can cause is that the
// others give up too (FDC_DEV_TIMEOUT).
static __device__ __noinline__ void raise_sync_slow(uint32_t bar, uint64_t tok, volatile int* abort_flag, int32_t* status)
{
    for (uint32_t i = 0; i < (1u << 18); ++i) {
        uint32_t ok;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(ok) : "r"(bar), "l"(tok) : "memory");
        if (ok) return;
        if ((i & 255u) == 255u && *abort_flag) return;
    }
    *abort_flag = 1;
    atomicOr(status, FDC_DEV_TIMEOUT);
}
__device__ __forceinline__ void raise_sync(uint32_t bar, volatile int* abort_flag, int32_t* status)
{
    __syncwarp();
    uint64_t tok = 0;
    if ((threadIdx.x & 31) == 0) asm volatile("mbarrier.arrive.shared::cta.b64 %0, [%1];" : "=l"(tok) : "r"(bar) : "memory");
    tok = __shfl_sync(0xffffffffu, tok, 0);
    raise_sync_slow(bar, tok, abort_flag, status);
}

// Monotone map float -> int (for integer max reductions).
__device__ __forceinline__ int ord_of(float x)
{
    const int i = __float_as_int(x);
    return i ^ ((i >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float ord_to(int i) { return __int_as_float(i ^ ((i >> 31) & 0x7fffffff)); }

// Small per-CTA state in static shared memory.  The raise path finds its barrier from the address of
// the abort flag (it is handed that address anyway).
struct __align__(8) CtaFlags {
    uint64_t raise_bar;              // mbarrier of the reference-raising path (raise_sync)
    int abort_flag;                  // a bounded wait ran out somewhere in the CTA
    int v_steps[4];
};
constexpr uint32_t RAISE_BAR_BEFORE_ABORT_FLAG = 8;
static_assert(offsetof(CtaFlags, abort_flag) - offsetof(CtaFlags, raise_bar) == RAISE_BAR_BEFORE_ABORT_FLAG, "layout");

// Everything a role needs to find its barriers and buffers.
struct Ctx : Split {
    // mbarriers: one base address, fixed offsets (kept as functions so that a single register serves them all)
    uint32_t bar0;
    __device__ __forceinline__ uint32_t k_full() const { return bar0; }
    __device__ __forceinline__ uint32_t k_empty() const { return bar0 + 8 * MAXST; }
    __device__ __forceinline__ uint32_t v_full() const { return bar0 + 16 * MAXST; }
    __device__ __forceinline__ uint32_t v_empty() const { return bar0 + 24 * MAXST; }
    __device__ __forceinline__ uint32_t s_full() const { return bar0 + 32 * MAXST; }
    __device__ __forceinline__ uint32_t s_free() const { return bar0 + 32 * MAXST + 32; }
    __device__ __forceinline__ uint32_t p_full() const { return bar0 + 32 * MAXST + 64; }
    __device__ __forceinline__ uint32_t pv_done() const { return bar0 + 32 * MAXST + 80; }
    __device__ __forceinline__ uint32_t q_ready() const { return bar0 + 32 * MAXST + 96; }
    __device__ __forceinline__ uint32_t o_free() const { return bar0 + 32 * MAXST + 104; }
    __device__ __forceinline__ uint32_t app_done() const { return bar0 + 32 * MAXST + 112; }
    __device__ __forceinline__ uint32_t peer_done() const { return bar0 + 32 * MAXST + 120; }
    int ns, s_stride;                // S^T buffers in TMEM (4 of 64 columns) and their distance
    uint32_t tmem;
    unsigned char *kring, *vring, *qs, *ps, *ones;
    float *mneg, *alpha, *lred;      // [128] -reference per column, [128] rescale factors, [4][128] partial sums
    int *cmax, *flags;               // [128] column maxima (ordered ints), [4] flags of the raise path and the merge
    int* rflag;                      // [8] rflag[g & 7] == g: round g met a score far above its reference
    uint64_t* smask;                 // [2][mbuf] the current segment's scene bitmaps (when mstaged)
    int mbuf;                        // words per buffer
    uint64_t* sunion;                // [2][UW] their OR over the scene's active branches (when mstaged and W <= UW)
    int mstaged;
    volatile int* abortp;
    volatile int* v_steps;           // [2][2] per P^T buffer and tile of the round: the 16-row steps to multiply (bit k: rows 16k..)
    int nk, nv, q_panel, p_buf, npb; // ring depths, bytes per 64-column panel of Q^T, bytes per P^T buffer, P^T buffers (2)
};

// Row bitmap (Eq. 1) of branch b of the segment's scene.  While the K/V stream saturates the
// memory system a global read costs microseconds, so the softmax warps copy the scene's bitmaps
// to shared memory at the start of a segment whenever they fit.
__device__ __forceinline__ const uint64_t* mask_row(const AttnParams& p, const Ctx& cx, uint32_t seg, int s, int b)
{
    return cx.mstaged ? cx.smask + (seg & 1) * cx.mbuf + (size_t)b * p.W : p.mask + ((size_t)s * p.max_active + b) * p.W;
}
// 16-byte asynchronous copy global -> shared (zero fill when !valid); completes with cp_async_wait_all.
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
// One elected thread: S^T[g mod ns] = K(stage) Q^T for every round g.  A score buffer is free again
// once the softmax threads have read round g - ns (s_free); with four buffers K Q^T runs well ahead of
// the softmax, so a K stage is released soon after it landed and the K ring stays in flight.
// The whole warp goes round this loop (and those of the other two issuing warps) and one elected thread issues: a
// round's issue is on the path from its K rows to its weights, and with the loops inside "lane 0" it took longer (us a
// layer, lane 0 / elected: 8 scenes x 4 heads, 64 rows, prefix 8192: 61.5 / 59.1; 16 scenes, 24 rows, prefix 4096: 53.3 / 52.2).
__device__ __forceinline__ void qk_loop(const AttnParams& p, const Ctx& cx, long long lo, long long hi)
{
    const uint64_t q_desc = smem_desc(smem_u32(cx.qs), 16, 1024);
    const uint64_t k_desc0 = smem_desc(smem_u32(cx.kring), 16, 1024);
    const uint32_t q_lo = (uint32_t)q_desc, q_hi = (uint32_t)(q_desc >> 32), k_lo0 = (uint32_t)k_desc0, k_hi = (uint32_t)(k_desc0 >> 32);
    const uint32_t qp16 = (uint32_t)(cx.q_panel >> 4);
    int s = 0;
    uint32_t g = 0, seg = 0;
    int st = 0;
    uint32_t kph = 0;                               // ring position and phase of the K stage of round g
    long long u = lo;
    bool ok = true;
    while (u < hi && ok) {
        const Segment sg = decode_segment(u, hi, cx.pre, p.hkv, s);
        const int nr = (sg.j1 - sg.j0 + 1) >> 1;
        const int M = cx.nact[sg.s] * p.group;
        const int NP = (NP_MAX == 32 || M <= 32) ? 32 : 64;
        const uint32_t idesc_qk = instr_desc(RROWS, NP, 0);
        bool good = ok && mbar_wait_warp(cx.q_ready(), seg & 1, cx.abortp, p.status);
        for (int t = 0; t < nr && good; ++t, ++g) {
            good = mbar_wait(cx.k_full() + 8 * st, kph, cx.abortp, p.status);
            const uint32_t sb = g & (cx.ns - 1);                  // score buffer of the round
            if (good && g >= (uint32_t)cx.ns) good = mbar_wait(cx.s_free() + 8 * sb, ((g / cx.ns) - 1) & 1, cx.abortp, p.status);
            good = __all_sync(0xffffffffu, good);
            if (!good) break;
            tc_fence_after();
            if (elect_one()) {
                const uint32_t kd = k_lo0 + (uint32_t)((st * STAGE) >> 4);
                const uint32_t d = cx.tmem + sb * cx.s_stride;
#pragma unroll
                for (int ks = 0; ks < D / 16; ++ks)
                    umma2(d, kd + (uint32_t)(((ks >> 2) * PANEL + (ks & 3) * 32) >> 4), k_hi, q_lo + (ks >> 2) * qp16 + (uint32_t)(((ks & 3) * 32) >> 4), q_hi,
                          idesc_qk, ks > 0);
                umma_commit(cx.k_empty() + 8 * st);
                umma_commit(cx.s_full() + 8 * sb);
            }
            __syncwarp();
            if (++st == cx.nk) {
                st = 0;
                kph ^= 1;
            }
        }
        ok = good;
        ++seg;
        u = sg.next_u;
    }
}

// The auxiliary warp: with fdc_set_fused_append it writes the pass's new K/V rows that fall into
// this CTA's tiles, then lets the producer go on to the tiles beyond the prefix; after that one
// of its threads issues the column-sum multiplications.
__device__ __forceinline__ void aux_loop(const AttnParams& p, const Ctx& cx, long long lo, long long hi, int lane)
{
    if (p.app_row) {
        append_rows<4>(const_cast<char*>(reinterpret_cast<const char*>(p.k)), const_cast<char*>(reinterpret_cast<const char*>(p.v)),
                    p.stride_scene * 2, p.stride_head * 2, p.stride_row * 2, p.app_row, reinterpret_cast<const char*>(p.app_k),
                    reinterpret_cast<const char*>(p.app_v), p.tiles, p.ntile_max, p.max_active, p.hkv, p.rows, p.P, cx.pre, cx.nact, lo, hi,
                    p.status);
        if (lane == 0) mbar_arrive(cx.app_done());
    }
    // The column sums of P^T (the softmax denominators), taken by the tensor core beside every
    // O^T += V^T P^T: P (128 query columns as rows, read from the same P^T buffer, which is laid out
    // the same way for either operand) times 16 columns of ones, so that TMEM lane n of the accumulator
    // holds sum_k P^T[k][n] of exactly the values that are multiplied with V.  For fewer than 128 query
    // rows the multiplication reads on past the P^T buffer (shared memory of this CTA all the same):
    // those rows of the result are never looked at, and a row depends on nothing but its own inputs.
    // Issued from this warp so that the thread that issues the V multiplications is not slowed down;
    // the same 16-row steps are left out, and both threads commit to the pv_done barrier.
    const uint64_t ones_desc = smem_desc(smem_u32(cx.ones), PANEL, 1024);
    const uint64_t p_desc0 = smem_desc(smem_u32(cx.ps), PANEL, 1024);
    const uint32_t ones_lo = (uint32_t)ones_desc, ones_hi = (uint32_t)(ones_desc >> 32), p_lo0 = (uint32_t)p_desc0, p_hi = (uint32_t)(p_desc0 >> 32);
    const uint32_t tm_l = cx.tmem + TM_L;
    int s = 0;
    uint32_t g = 0, seg = 0;
    long long u = lo;
    bool ok = true;
    while (u < hi && ok) {
        const Segment sg = decode_segment(u, hi, cx.pre, p.hkv, s);
        const uint32_t idesc_sum = instr_desc(128, 16, 1);
        const int ntile = sg.j1 - sg.j0;
        bool good = ok;
        for (int t = 0; 2 * t < ntile && good; ++t, ++g) {
            good = mbar_wait(cx.p_full() + 8 * (g & 1), (g >> 1) & 1, cx.abortp, p.status);
            if (good && t == 0 && seg > 0) good = mbar_wait(cx.o_free(), (seg - 1) & 1, cx.abortp, p.status);
            good = __all_sync(0xffffffffu, good);
            if (!good) break;
            const uint32_t steps = (uint32_t)cx.v_steps[(g & 1) * 2] | ((uint32_t)cx.v_steps[(g & 1) * 2 + 1] << 4);
            tc_fence_after();
            if (elect_one()) {
                const uint32_t pd = p_lo0 + (uint32_t)((((g & 1) & (cx.npb - 1)) * cx.p_buf) >> 4);
                uint32_t acc = t > 0 ? 1u : 0u;
#pragma unroll 1
                for (int kk = 0; kk < 8; ++kk)
                    if ((steps >> kk) & 1u) {
                        umma2(tm_l, pd + kk * 128, p_hi, ones_lo, ones_hi, idesc_sum, acc);
                        acc = 1u;
                    }
                umma_commit(cx.pv_done() + 8 * (g & 1));
            }
            __syncwarp();
        }
        ok = good;
        ++seg;
        u = sg.next_u;
    }
}

// One elected thread: O^T += V^T(stage) P^T[g & 1] for every round g, once the stage has landed and
// the softmax warps have delivered P^T (and, beyond the prefix, cleared the stage's unseen rows).
// The multiplication runs in steps of 16 KV rows; the softmax warps say which steps hold a visible
// row (all of them inside the prefix), the others are left out.
__device__ __forceinline__ void pv_loop(const AttnParams& p, const Ctx& cx, long long lo, long long hi)
{
    const uint64_t v_desc0 = smem_desc(smem_u32(cx.vring), PANEL, 1024);
    const uint64_t p_desc0 = smem_desc(smem_u32(cx.ps), PANEL, 1024);
    const uint32_t v_lo0 = (uint32_t)v_desc0, v_hi = (uint32_t)(v_desc0 >> 32), p_lo0 = (uint32_t)p_desc0, p_hi = (uint32_t)(p_desc0 >> 32);
    const uint32_t tm_o = cx.tmem + TM_O;
    int s = 0;
    uint32_t g = 0, seg = 0;
    int st = 0;
    uint32_t vph = 0;
    long long u = lo;
    bool ok = true;
    while (u < hi && ok) {
        const Segment sg = decode_segment(u, hi, cx.pre, p.hkv, s);
        const int M = cx.nact[sg.s] * p.group;
        const int NP = (NP_MAX == 32 || M <= 32) ? 32 : 64;
        const uint32_t idesc_pv = instr_desc(D, NP, 1);
        const int ntile = sg.j1 - sg.j0;
        bool good = ok;
        for (int t = 0; 2 * t < ntile && good; ++t, ++g) {
            good = mbar_wait(cx.v_full() + 8 * st, vph, cx.abortp, p.status);
            if (good) good = mbar_wait(cx.p_full() + 8 * (g & 1), (g >> 1) & 1, cx.abortp, p.status);
            if (good && t == 0 && seg > 0) good = mbar_wait(cx.o_free(), (seg - 1) & 1, cx.abortp, p.status);
            good = __all_sync(0xffffffffu, good);
            if (!good) break;
            const uint32_t steps = (uint32_t)cx.v_steps[(g & 1) * 2] | ((uint32_t)cx.v_steps[(g & 1) * 2 + 1] << 4);
            tc_fence_after();
            if (elect_one()) {
                const uint32_t vd = v_lo0 + (uint32_t)((st * STAGE) >> 4);
                const uint32_t pd = p_lo0 + (uint32_t)((((g & 1) & (cx.npb - 1)) * cx.p_buf) >> 4);
                if (steps == 0xffu) {
#pragma unroll
                    for (int kk = 0; kk < 8; ++kk) umma2(tm_o, vd + kk * 128, v_hi, pd + kk * 128, p_hi, idesc_pv, (t > 0 || kk > 0) ? 1u : 0u);
                } else {
                    // a one-tile round has 64 KV rows; beyond the prefix, steps without a visible row are left out
                    // (rows that nobody may see can hold NaN, and 0 * NaN must not reach the accumulator)
                    uint32_t acc = t > 0 ? 1u : 0u;
#pragma unroll 1
                    for (int kk = 0; kk < 8; ++kk)
                        if ((steps >> kk) & 1u) {
                            umma2(tm_o, vd + kk * 128, v_hi, pd + kk * 128, p_hi, idesc_pv, acc);
                            acc = 1u;
                        }
                }
                umma_commit(cx.v_empty() + 8 * st);
                umma_commit(cx.pv_done() + 8 * (g & 1));
            }
            __syncwarp();
            if (++st == cx.nv) {
                st = 0;
                vph ^= 1;
            }
        }
        ok = good;
        ++seg;
        u = sg.next_u;
    }
}

// Visibility (Eq. 1) of one KV row for the nph (<= 32) query columns starting at col0: bit i <=>
// column col0 + i may see the row.  `row` (0..63) is the thread's row inside tile `tile`.  Columns
// b * G .. b * G + G - 1 belong to branch b; every thread reads the bitmap words of the two or three
// branches its columns belong to (the same words for the whole warp: one broadcast read each).
// When the prefix is a whole number of tiles a tile's 64 rows are one word of the bitmap; otherwise
// they straddle two (tile_rowmask).  Only tiles beyond the prefix come here.
__device__ __forceinline__ uint32_t row_visibility(const uint64_t* mask0, int W, int P, int tile, int row, int A, int G, int b_lo, int col0, int nph)
{
    uint32_t vis = 0u;
    const bool aligned = (P & (TILE - 1)) == 0;
    const int w = tile - P / TILE;
    int c = b_lo * G - col0;                       // first column of branch b relative to col0 (<= 0 for the first one)
#pragma unroll 1
    for (int b = b_lo; b < A && c < nph; ++b, c += G) {
        const uint64_t word = aligned ? (w < W ? mask0[(size_t)b * W + w] : 0ull) : tile_rowmask(mask0 + (size_t)b * W, W, P, tile);
        const int lo = c < 0 ? 0 : c, hi = c + G > nph ? nph : c + G;
        const uint32_t span = (hi - lo >= 32 ? 0xffffffffu : ((1u << (hi - lo)) - 1u)) << lo;
        if ((word >> row) & 1ull) vis |= span;
    }
    return vis;
}

// Asynchronous copies of the next segment's queries into Q^T and of its scene's bitmaps into
// the other bitmap buffer (softmax threads; completed with cp_async_wait_all in the prologue).
// (All arguments by value: a reference to the caller's context would force it into local memory.)
__device__ __noinline__ void prefetch_next_segment(const uint4* qg, const uint64_t* mask, int max_active, int W, int hq, int G, int hkv,
                                                   const int* pre, const int* nact, unsigned char* qs, int q_panel,
                                                   uint64_t* smask_dst, long long next_u, long long hi, int s_cur)
{
    const int tid = threadIdx.x;
    int s2 = s_cur;
    const Segment nx = decode_segment(next_u, hi, pre, hkv, s2);
    const int M2 = nact[nx.s] * G;
    const int NP2 = (NP_MAX == 32 || M2 <= 32) ? 32 : 64;
    for (int idx = tid; idx < NP2 * (D / 8); idx += NSOFT * 32) {
        const int n = idx / (D / 8), ch = idx - n * (D / 8);
        const bool valid = n < M2;
        const int bb = valid ? n / G : 0, hg = valid ? n - bb * G : 0;
        cp_async16(qs + (ch >> 3) * q_panel + n * 128 + (((ch & 7) ^ (n & 7)) << 4),
                   qg + ((((size_t)nx.s * max_active + bb) * hq + (size_t)nx.g * G + hg) * D) / 8 + ch, valid);
    }
    if (smask_dst) {
        const uint64_t* src = mask + (size_t)nx.s * max_active * W;
        for (int idx = tid; idx < max_active * W; idx += NSOFT * 32) cp_async8(smask_dst + idx, src + idx);
    }
}

// The first pair's bitmaps and queries when the kernel runs ahead of the dependency wait (softmax
// threads; out of line, arguments by value).  The bitmaps are complete and are copied right away.
// The queries may still be written by the kernel ahead: their lines are only requested into L2
// (which stays coherent), the wait is taken, and then they are read and laid out as Q^T.
__device__ __noinline__ void stage_first_pair_early(const uint4* qg, const uint64_t* mask, int max_active, int W, int hq, int G, int s, int g, int M,
                                                    unsigned char* qs, int q_panel, uint64_t* smask_dst)
{
    const int tid = threadIdx.x;
    const int NP = (NP_MAX == 32 || M <= 32) ? 32 : 64;
    if (smask_dst) {
        const uint64_t* src = mask + (size_t)s * max_active * W;
        for (int idx = tid; idx < max_active * W; idx += NSOFT * 32) smask_dst[idx] = src[idx];
    }
    for (int idx = tid * 8; idx < M * (D / 8); idx += NSOFT * 32 * 8) {      // one request per 128-byte line
        const int n = idx / (D / 8), ch = idx - n * (D / 8);
        const int bb = n / G, hg = n - bb * G;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(qg + ((((size_t)s * max_active + bb) * hq + (size_t)g * G + hg) * D) / 8 + ch));
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int idx = tid; idx < NP * (D / 8); idx += NSOFT * 32) {
        const int n = idx / (D / 8), ch = idx - n * (D / 8);
        const bool valid = n < M;
        const int bb = valid ? n / G : 0, hg = valid ? n - bb * G : 0;
        cp_async16(qs + (ch >> 3) * q_panel + n * 128 + (((ch & 7) ^ (n & 7)) << 4),
                   qg + ((((size_t)s * max_active + bb) * hq + (size_t)g * G + hg) * D) / 8 + ch, valid);
    }
}

// Merge of the partials of one (scene, KV head) pair by the CTA that delivered the last one
// (all softmax threads).  Every thread owns four accumulator columns of one query row and merges
// the parts' (m, l, O) for them in ONE pass, three parts per turn with all loads ahead of the
// arithmetic (a turn costs one trip to L2; the running maximum is carried like in the online
// softmax, so more parts need no second pass):
//     m = max_c m_c,  l = sum_c l_c 2^(m_c - m),  O = sum_c O_c 2^(m_c - m) / l.
// Out of line, arguments by value.
__device__ __noinline__ void merge_pair(const float* ws_ml, const float* ws_o, __nv_bfloat16* out, int pair, int mmax, int M, int G, int s, int g,
                                        int max_active, int hq, int c_first, int c_last)
{
    constexpr int MB = 3;                          // parts per turn
    const int tid = threadIdx.x;
    __threadfence();
    for (int idx = tid; idx < M * (D / 4); idx += NSOFT * 32) {
        const int m = idx / (D / 4), c4 = idx - m * (D / 4);
        const float2* ml = reinterpret_cast<const float2*>(ws_ml + ((size_t)pair * mmax + m) * 2);
        const float4* po = reinterpret_cast<const float4*>(ws_o + ((size_t)pair * mmax + m) * D) + c4;
        const size_t cs = (size_t)mmax, os = (size_t)mmax * (D / 4);      // strides between CTAs' entries
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        float mx = -INFINITY, lt = 0.f;
        for (int c0 = c_first; c0 <= c_last; c0 += MB) {
            float2 v[MB];
            float4 o[MB];
#pragma unroll
            for (int j = 0; j < MB; ++j) {
                const bool on = c0 + j <= c_last;
                v[j] = on ? __ldcg(ml + (size_t)(c0 + j) * cs) : make_float2(-INFINITY, 0.f);
                o[j] = on ? __ldcg(po + (size_t)(c0 + j) * os) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            float nm = mx;
#pragma unroll
            for (int j = 0; j < MB; ++j) nm = fmaxf(nm, v[j].x);
            const float sc = mx == nm ? 1.f : fast_exp2(mx - nm);           // (-inf) - (-inf) must not be formed
            lt *= sc;
            acc.x *= sc;
            acc.y *= sc;
            acc.z *= sc;
            acc.w *= sc;
#pragma unroll
            for (int j = 0; j < MB; ++j) {
                const float w = v[j].x == -INFINITY ? 0.f : fast_exp2(v[j].x - nm);   // a part that saw nothing
                lt = fmaf(v[j].y, w, lt);
                acc.x = fmaf(o[j].x, w, acc.x);
                acc.y = fmaf(o[j].y, w, acc.y);
                acc.z = fmaf(o[j].z, w, acc.z);
                acc.w = fmaf(o[j].w, w, acc.w);
            }
            mx = nm;
        }
        const float inv = 1.f / lt;
        const int b = m / G, hg = m - b * G;
        uint2 pk;
        pk.x = pack2(acc.x * inv, acc.y * inv);
        pk.y = pack2(acc.z * inv, acc.w * inv);
        *reinterpret_cast<uint2*>(out + (((size_t)s * max_active + b) * hq + (size_t)g * G + hg) * D + c4 * 4) = pk;
    }
}

// The rare path of the softmax, kept out of line so that the per-round loop stays small: the
// first round of a segment, or two (two groups: three) rounds after some score exceeded its column's reference by
// more than 2^16.  Column maxima of the round are gathered (shuffle transpose-reduce per warp,
// one shared-memory slot per row quadrant), references that are unset or too low are replaced,
// alpha[n] = 2^(old - new) is published, and the column sums (TMEM) and the accumulator O^T are
// rescaled where a reference moved.  Called by all softmax threads.  Returns 1 when a bounded
// wait ran out.  All arguments by value.
struct RaiseArgs {
    float* mneg;                 // column state in shared memory: mneg[128], alpha[128], lred[512], cmax[128], flags[4]
    volatile int* abortp;
    int32_t* status;
    uint32_t s_addr, o_addr;     // TMEM addresses of this thread's first score / accumulator column
    int np;                      // query columns of the pair, padded (32 / 64)
    uint32_t pv_bar, pv_parity;  // completion of the previous round's O^T += V^T P^T
    uint32_t vis;                // Eq. 1 bits of this thread's columns
    float c;
    int col0, nph;               // this thread's columns
    int live;                    // 1: the thread's KV row exists; 0: it does not (second half of a one-tile round); -1: the round
                                 // belongs to the other group of softmax warps, this one only takes part in the barriers
    int rescale_o, dead;
};
__device__ __noinline__ int raise_references(const RaiseArgs a)
{
    const int np = a.np;
    float* alpha = a.mneg + 128;
    int* wmax = reinterpret_cast<int*>(a.mneg + 256);      // [4][128]: maxima per row quadrant (shares the lred block)
    int* flags = reinterpret_cast<int*>(a.mneg + 768) + 128;
    const int tid = threadIdx.x, lane = threadIdx.x & 31, q4 = (threadIdx.x >> 5) & 3;
    bool dead = a.dead != 0;
    for (int ch = 0; ch < (a.live < 0 ? 0 : a.nph / 8); ++ch) {
        float mine = -INFINITY;                              // lane i < 8 ends up with the maximum of column ch * 8 + i
        if (a.live > 0) {
            uint32_t sv[8];
            tmem_ld<8>(a.s_addr + ch * 8, sv);
            tmem_wait_ld();
            float v[8];
            const uint32_t vb = a.vis >> (ch * 8);
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = ((vb >> i) & 1) ? __uint_as_float(sv[i]) * a.c : -INFINITY;
            // lanes whose index differs in bits >= 8 hold rows of the same columns: plain max
#pragma unroll
            for (int o = 16; o >= 8; o >>= 1)
#pragma unroll
                for (int i = 0; i < 8; ++i) v[i] = fmaxf(v[i], __shfl_xor_sync(0xffffffffu, v[i], o));
            // transpose-reduce: at distance k a lane keeps the half of the columns that matches its bit k
#pragma unroll
            for (int k = 4; k >= 1; k >>= 1) {
                const bool up = (lane & k) != 0;
#pragma unroll
                for (int i = 0; i < k; ++i) {
                    const float recv = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + k], k);
                    v[i] = fmaxf(up ? v[i + k] : v[i], recv);
                }
            }
            mine = v[0];
        }
        if (lane < 8) wmax[q4 * 128 + a.col0 + ch * 8 + lane] = ord_of(mine);
    }
    if (tid == 0) flags[0] = 0;
    raise_sync(smem_u32(const_cast<int*>(a.abortp)) - RAISE_BAR_BEFORE_ABORT_FLAG, a.abortp, a.status);
    if (tid < ((np + 31) & ~31)) {                         // whole warps (the shuffles below need all lanes)
        // highest column maximum of the round (every warp of these threads computes it for itself)
        int gm = INT_MIN;
        for (int n = lane; n < np; n += 32)
            gm = max(gm, max(max(wmax[n], wmax[128 + n]), max(wmax[256 + n], wmax[384 + n])));
#pragma unroll
        for (int o = 16; o; o >>= 1) gm = max(gm, __shfl_xor_sync(0xffffffffu, gm, o));
        if (tid < np) {
            const int m01 = max(wmax[tid], wmax[128 + tid]), m23 = max(wmax[256 + tid], wmax[384 + tid]);
            const float mx = ord_to(max(m01, m23));
            const float old = a.mneg[tid];                     // -reference, or UNSET
            float al = 1.f;
            if (old == UNSET) {
                // a column that sees no row yet borrows the round's highest reference: it will rarely have
                // to be raised later, and lower scores only make its terms smaller (far from underflow)
                const float ref = mx != -INFINITY ? mx : ord_to(gm);
                if (ref != -INFINITY) a.mneg[tid] = -ref;
            } else if (mx > RAISE_LOG2 - old) {
                al = fast_exp2(-old - mx);
                a.mneg[tid] = -mx;
                flags[0] = 1;
            }
            alpha[tid] = al;
        }
    }
    raise_sync(smem_u32(const_cast<int*>(a.abortp)) - RAISE_BAR_BEFORE_ABORT_FLAG, a.abortp, a.status);
    if (flags[0]) {                                        // a reference moved: rescale the accumulators (column sums and O^T)
        if (a.rescale_o) {
            if (!dead && !mbar_wait(a.pv_bar, a.pv_parity, a.abortp, a.status)) dead = true;   // no MMA may be writing O^T
            dead = __any_sync(0xffffffffu, dead);
            tc_fence_after();
            if (!dead) {
                for (int ch = 0; ch < a.nph / 8; ++ch) {
                    uint32_t ov[8];
                    tmem_ld<8>(a.o_addr + ch * 8, ov);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 8; ++i) ov[i] = __float_as_uint(__uint_as_float(ov[i]) * alpha[a.col0 + ch * 8 + i]);
                    tmem_st<8>(a.o_addr + ch * 8, ov);
                }
                if (a.col0 == 0) {                          // the column sums: TMEM lane n belongs to query column n
                    const uint32_t l_addr = a.o_addr - TM_O + TM_L;
                    uint32_t lv[8];
                    tmem_ld<8>(l_addr, lv);
                    tmem_wait_ld();
                    const float al = alpha[threadIdx.x & 127];
#pragma unroll
                    for (int i = 0; i < 8; ++i) lv[i] = __float_as_uint(__uint_as_float(lv[i]) * al);
                    tmem_st<8>(l_addr, lv);
                }
            }
        }
        tmem_wait_st();
    }
    return dead ? 1 : 0;
}

// The softmax warps' work on one segment; nphj = a quarter of the pair's padded query columns NP (8,
// 16 or 32).  Columns are handled eight at a time in real loops with the references read from
// shared memory, so that the same small loop serves every width.
//
// NGRP = 2 (launches whose widest pair has 33 to 64 query rows; measured: 3 to 6 % faster there, 1 %
// slower with fewer rows): the sixteen warps work as TWO GROUPS of eight on alternate rounds (group =
// round & 1: the round's score buffer and P^T buffer are then that group's own): a thread handles
// one KV row x NP / 2 columns of every other round, and while one group sits in the latency chain
// around a round (barrier tests, fences, arrivals) the other one is in its arithmetic.  Every warp
// still walks through all rounds of the segment, so both groups meet at the same places: the
// segment's set-up and end, its first round (references), its last round (next queries), and a
// raise of the references, which both decide on from a note that is three rounds old (by then it
// is final for either group without a wait of its own).
// NGRP = 1: all sixteen warps on every round, a thread handles one KV row x NP / 4 columns.
__device__ __forceinline__ void softmax_segment(const AttnParams& p, const Ctx& cx, const Segment& sg, const int nph, const uint32_t seg,
                                                const long long hi, int& prefetched, uint32_t& g, int& vst, uint32_t& vph, bool& dead, const int warp, const int lane)
{
    const int np = NPART * nph;                   // the pair's padded query columns
    const int tid = threadIdx.x;                  // 0..NSOFT * 32 - 1
    const int q4 = warp & 3, part = warp >> 2;
    const int krow = q4 * 32 + lane;              // KV row of the round = TMEM lane of S^T; head_dim index for O^T
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
    constexpr int ngrp = NGRP;                    // groups of softmax warps (two: warp >> 3 is the group, it works on the rounds of that parity)
    const int nphr = nph * ngrp, nchr = nphr >> 3;              // (round mapping: a group = 4 row quadrants x 4 / ngrp column parts)
    const int col0r = (ngrp == 2 ? (part & 1) : part) * nphr;
    const float c = p.scale_log2;
    const int A = cx.nact[sg.s];
    const int M = A * p.group;
    const int G = p.group;
    const int b_lo = col0r / G;                   // branch of this thread's first query column
    auto wait_u = [&](uint32_t bar, uint32_t parity) {    // warp-uniform outcome
        if (dead || __all_sync(0xffffffffu, mbar_try(bar, parity))) return;          // usually satisfied already
        if (!mbar_wait_slow(bar, parity, cx.abortp, p.status)) dead = true;
        dead = __any_sync(0xffffffffu, dead);
    };
    // ---- Q^T (B operand of S^T = K Q^T): row n = query row, K-major, 128B swizzle, rows >= M zero
    const bool published = prefetched == 2;       // Q^T, the bitmaps and their OR were completed and announced at the end of the previous segment
    {
        if (prefetched) {
            // queries and bitmaps were copied asynchronously during the previous segment's last round
            if (!published) cp_async_wait_all();
            prefetched = 0;
        } else {
            // all global reads first (one latency), then the stores
            const uint4* qg = reinterpret_cast<const uint4*>(p.q);
            constexpr int QPT = NP_MAX * (D / 8) / (NSOFT * 32);   // 16-byte chunks per thread for the widest pair of this build
            uint4 qv[QPT];
#pragma unroll
            for (int i = 0; i < QPT; ++i) {
                const int idx = tid + i * (NSOFT * 32);
                const int n = idx / (D / 8), ch = idx - n * (D / 8);
                qv[i] = make_uint4(0u, 0u, 0u, 0u);
                if (n < M) {
                    const int b = n / G, hg = n - b * G;
                    qv[i] = qg[((((size_t)sg.s * p.max_active + b) * p.hq + (size_t)sg.g * G + hg) * D) / 8 + ch];
                }
            }
            uint64_t mv[MBUF / (NSOFT * 32)];
            const int nw = cx.mstaged ? p.max_active * p.W : 0;
#pragma unroll
            for (int i = 0; i < MBUF / (NSOFT * 32); ++i) {
                const int idx = tid + i * (NSOFT * 32);
                mv[i] = idx < nw ? p.mask[(size_t)sg.s * p.max_active * p.W + idx] : 0ull;
            }
#pragma unroll
            for (int i = 0; i < QPT; ++i) {
                const int idx = tid + i * (NSOFT * 32);
                const int n = idx / (D / 8), ch = idx - n * (D / 8);
                if (n < np) *reinterpret_cast<uint4*>(cx.qs + (ch >> 3) * cx.q_panel + n * 128 + (((ch & 7) ^ (n & 7)) << 4)) = qv[i];
            }
#pragma unroll
            for (int i = 0; i < MBUF / (NSOFT * 32); ++i) {
                const int idx = tid + i * (NSOFT * 32);
                if (idx < nw) cx.smask[(seg & 1) * cx.mbuf + idx] = mv[i];
            }
        }
        if (cx.mstaged && p.W <= UW && !published) {
            // OR of the scene's bitmaps: the rows that some branch may see (the others are cleared in V)
            soft_sync();                              // everybody's share of the bitmaps is in place
            if (tid < p.W) {
                const uint64_t* mb = cx.smask + (seg & 1) * cx.mbuf + tid;
                uint64_t un = 0ull;
                for (int b = 0; b < A; ++b) un |= mb[(size_t)b * p.W];
                cx.sunion[(seg & 1) * UW + tid] = un;
            }
        }
        if (tid < np) cx.mneg[tid] = UNSET;
        if (!published) {
            fence_async_smem();
            __syncwarp();
            if (!dead && lane == 0) mbar_arrive(cx.q_ready());
        }
        soft_sync();
    }

    const int ntile = sg.j1 - sg.j0;
    int t = 0;                                    // round within the segment
    for (int jb = 0; jb < ntile; jb += 32) {
        const int jn = ntile - jb < 32 ? ntile - jb : 32;
#if FDC_TC_TWO
        const int my_tile = lane < jn ? p.tiles[(size_t)sg.s * p.ntile_max + tile_entry(sg, jb + lane)] : 0;
#else                                             // (the same thing; by way of tile_entry the build for 32 rows spills)
        const int my_tile = lane < jn ? p.tiles[(size_t)sg.s * p.ntile_max + sg.j0 + jb + lane] : 0;
#endif
        for (int k = 0; k < jn; k += 2, ++g, ++t) {
            const int nt = jn - k < 2 ? 1 : 2;
            const uint32_t b = g & 1;
            const int ti = q4 >> 1;                                   // which tile of the round this warp's rows are in
            const int tile = __shfl_sync(0xffffffffu, my_tile, (k + ti) & 31);
            const bool mine = ngrp == 1 || ((g ^ (uint32_t)(warp >> 3)) & 1u) == 0u;   // this warp's group works on the round (warps 0..7: even rounds)
            const bool live = mine && ti < nt && !dead;               // rows 64..127 of a one-tile round hold nothing
            const bool masked = live && tile * TILE + TILE > p.P;
            // Eq. 1 for this thread's KV row: bit i of vis <=> column col0r + i may see the row
            const uint32_t vis = masked ? row_visibility(mask_row(p, cx, seg, sg.s, 0), p.W, p.P, tile, (q4 & 1) * 32 + lane, A, G, b_lo, col0r, nphr) : ~0u;
            const uint32_t sb = g & (cx.ns - 1);                      // score buffer of the round
            const bool last_round = jb + k + 2 >= ntile && sg.next_u < hi;
            if (mine || last_round) {
                wait_u(cx.s_full() + 8 * sb, (g / cx.ns) & 1);
                tc_fence_after();
            }
            if (last_round) {
                // last round: every S^T = K Q^T of this segment has completed, so Q^T may be overwritten.
                // The next segment's queries (and its scene's bitmaps, into the other buffer) are copied
                // asynchronously; the latency hides behind this round, the drain and the partial write.
                prefetch_next_segment(reinterpret_cast<const uint4*>(p.q), p.mask, p.max_active, p.W, p.hq, G, p.hkv, cx.pre, cx.nact, cx.qs,
                                      cx.q_panel, cx.mstaged ? cx.smask + ((seg + 1) & 1) * cx.mbuf : nullptr, sg.next_u, hi, sg.s);
                prefetched = 1;
            }
            // The P^T buffer is still being read until the PV that used it last (two rounds ago) has completed.  Past this wait every softmax
            // warp has also finished round g - 2 (one group), so what that round left in rflag is the same
            // for all.  With two groups only the round's own group waits; what both groups know without
            // any further wait is that round g - 3 is over for everybody (the owners of round g through
            // this wait, the others through theirs a round ago), so there a pending raise is looked for
            // three rounds after the note.  (No warp ever waits for a barrier of the other group's rounds
            // in mid-segment: a parity wait tells only two consecutive phases apart, and nothing would keep
            // that barrier from moving on twice.)
            if (mine) {
                wait_u(cx.pv_done() + 8 * b, ((g >> 1) & 1) ^ 1);
            }
            const uint32_t s_addr = cx.tmem + lane_base + sb * cx.s_stride + col0r;
            // References are set in the first round of a segment.  Later a score more than 2^16 above its
            // reference only leaves a note (no barrier in the common path): p stays far from overflow, and
            // two (two groups: three) rounds later, when all warps are known to see the note, the references are raised.
            if (t == 0 && __shfl_sync(0xffffffffu, my_tile, k & 31) * TILE + TILE <= p.P) {
                // First round of a segment inside the prefix: every column takes its score against the
                // round's first KV row (visible to all) as reference.  That row's own term is then exactly
                // 1, so no column sum can vanish; higher scores are handled by the lazy raise as usual.
                if (mine && q4 == 0 && !dead) {                       // the warps (of the round's group) that hold TMEM lane 0
#pragma unroll 1
                    for (int ch = 0; ch < nchr; ++ch) {
                        uint32_t sv[8];
                        tmem_ld<8>(s_addr + ch * 8, sv);
                        tmem_wait_ld();
                        if (lane == 0) {
#pragma unroll
                            for (int i = 0; i < 8; ++i) cx.mneg[col0r + ch * 8 + i] = -(__uint_as_float(sv[i]) * c);
                        }
                    }
                }
                soft_sync();
            } else if (t == 0 || (NGRP == 1 ? (g >= 2 && cx.rflag[(g - 2) & 7] == (int)(g - 2)) : (t >= 3 && cx.rflag[(g - 3) & 7] == (int)(g - 3)))) {
                RaiseArgs ra;
                ra.mneg = cx.mneg;
                ra.abortp = cx.abortp;
                ra.status = p.status;
                ra.s_addr = s_addr;
                ra.o_addr = cx.tmem + lane_base + TM_O + col0r;
                ra.np = np;
                ra.pv_bar = cx.pv_done() + 8 * ((g - 1) & 1);
                ra.pv_parity = ((g - 1) >> 1) & 1;
                ra.vis = vis;
                ra.c = c;
                ra.col0 = col0r;
                ra.nph = nphr;
                ra.live = mine ? (live ? 1 : 0) : -1;
                ra.rescale_o = mine && t > 0;
                ra.dead = dead;
                dead = raise_references(ra) != 0;
            }
            if (!mine) {                                              // the other group's round
                if (++vst == cx.nv) {
                    vst = 0;
                    vph ^= 1;
                }
                continue;
            }
            if (live) {
                unsigned char* prow = cx.ps + (b & (cx.npb - 1)) * cx.p_buf + krow * 128;
                float emax = 0.f;
#pragma unroll 1
                for (int ch = 0; ch < nchr; ++ch) {
                    uint32_t sv[8];
                    tmem_ld<8>(s_addr + ch * 8, sv);
                    const float4 m0 = *reinterpret_cast<const float4*>(cx.mneg + col0r + ch * 8);
                    const float4 m1 = *reinterpret_cast<const float4*>(cx.mneg + col0r + ch * 8 + 4);
                    const float mn[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
                    tmem_wait_ld();
                    if (masked) {                                      // uniform branch: prefix rounds skip the selects
                        const uint32_t vb = vis >> (ch * 8);
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            if (!((vb >> i) & 1)) sv[i] = 0xff800000u;
                    }
                    float e[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        e[i] = fast_exp2(fmaf(__uint_as_float(sv[i]), c, mn[i]));
                        emax = fmaxf(emax, e[i]);
                    }
                    // P^T goes to the tensor core as bf16.  The column sums (the softmax denominators) are taken by
                    // the tensor core too, from the SAME rounded values (a multiplication of P^T by ones beside
                    // every O^T += V^T P^T), so numerator and denominator stay consistent: the rounding cancels
                    // where a few terms dominate.
                    uint32_t pk[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) pk[j] = pack2(e[2 * j], e[2 * j + 1]);
                    const int cidx = (col0r >> 3) + ch;                // 16-byte chunk of the P^T row
                    *reinterpret_cast<uint4*>(prow + (cidx >> 3) * PANEL + (((cidx & 7) ^ (krow & 7)) << 4)) =
                        make_uint4(pk[0], pk[1], pk[2], pk[3]);
                }
                if (emax > 65536.f) {                                  // 2^16 above the reference: note it for round g + 2
                    cx.rflag[g & 7] = (int)g;
                    if (!(emax < 1.0e30f)) atomicOr(p.status, FDC_DEV_SCORE_RANGE);     // beyond 2^100 (or inf / nan)
                }
            }
            // ---- this round's V stage.  Beyond the prefix, rows that no branch of the scene may see can hold
            // anything (NaN, Inf: slots that were never written), and although their P^T entries are
            // exactly 0, 0 * NaN must not reach the accumulator.  The multiplication runs in steps of 16
            // KV rows: a step without any visible row is left out, and in the other steps the unseen
            // rows are cleared here, every thread a quarter of its own row, once the stage has landed.
            uint32_t st4 = live ? 0xfu : 0u;                           // steps of this warp's tile to multiply
            if (masked) {                                              // (uniform over the warp)
                const uint64_t* un = (cx.mstaged && p.W <= UW) ? cx.sunion + (seg & 1) * UW : nullptr;
                const int w = tile - p.P / TILE;
                const uint64_t seen = (un && (p.P & (TILE - 1)) == 0) ? (w < p.W ? un[w] : 0ull)
                                                                       : tile_seen_rows(un, mask_row(p, cx, seg, sg.s, 0), p.W, p.P, A, tile);
                wait_u(cx.v_full() + 8 * vst, vph);
                const int row = (q4 & 1) * 32 + lane;
                const bool none = seen == 0ull;                        // (such a tile should not be listed: clear and multiply all of it)
                const uint32_t step_seen = (uint32_t)(seen >> (row & 48)) & 0xffffu;
                if (!dead && (none || (step_seen != 0u && !((seen >> row) & 1ull)))) {
                    // the column parts of the group share the row's 256 bytes (two panels of 128): a quarter each, or a half
                    if constexpr (NGRP == 1) {
                        const uint32_t va = smem_u32(cx.vring) + (uint32_t)vst * STAGE + (uint32_t)(part >> 1) * PANEL +
                                            (uint32_t)(ti * TILE + row) * 128 + (uint32_t)(part & 1) * 64;
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(va + (uint32_t)((i + lane) & 3) * 16), "r"(0u) : "memory");
                    } else {
                        const uint32_t va = smem_u32(cx.vring) + (uint32_t)vst * STAGE + (uint32_t)(part & 1) * PANEL + (uint32_t)(ti * TILE + row) * 128;
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(va + (uint32_t)((i + lane) & 7) * 16), "r"(0u) : "memory");
                    }
                }
                st4 = 0u;
#pragma unroll
                for (int i = 0; i < 4; ++i) st4 |= (none || ((seen >> (16 * i)) & 0xffffull)) ? (1u << i) : 0u;
                // the whole tiles of the prefix come first in a tile list (entry j = tile j): the producer relies on it
                if (col0r == 0 && (q4 & 1) == 0 && lane == 0 && tile_entry(sg, jb + k + ti) < p.P / TILE) atomicOr(p.status, FDC_DEV_TILE_LIST);
            }
            if (col0r == 0 && (q4 & 1) == 0 && lane == 0) cx.v_steps[b * 2 + ti] = (int)st4;
            if (++vst == cx.nv) {
                vst = 0;
                vph ^= 1;
            }
            // every thread orders its own TMEM reads and shared-memory writes, then one lane per warp signals
            tc_fence_before();
            fence_async_smem();
            __syncwarp();
            if (!dead && lane == 0) {
                mbar_arrive(cx.s_free() + 8 * sb);                       // the scores have been read: K Q^T may reuse the buffer
                mbar_arrive(cx.p_full() + 8 * b);
            }
        }
    }
    if (prefetched == 1) {
        // The next pair's queries are announced before this pair is finished off, so that its K Q^T runs
        // on (into the score buffers) while the last multiplications drain and the result is written.
        cp_async_wait_all();
        if (cx.mstaged && p.W <= UW) {
            soft_sync();
            int s2 = sg.s;
            const Segment nx = decode_segment(sg.next_u, hi, cx.pre, p.hkv, s2);
            if (tid < p.W) {
                const uint64_t* mb = cx.smask + ((seg + 1) & 1) * cx.mbuf + tid;
                uint64_t un = 0ull;
                const int A2 = cx.nact[nx.s];
                for (int b = 0; b < A2; ++b) un |= mb[(size_t)b * p.W];
                cx.sunion[((seg + 1) & 1) * UW + tid] = un;
            }
        }
        fence_async_smem();
        __syncwarp();
        if (!dead && lane == 0) mbar_arrive(cx.q_ready());
        prefetched = 2;
    }
    // ---- end of segment: the accumulator is final once the last PV has completed
    // (joint mapping from here on: sixteen warps = 4 row quadrants x 4 column parts)
    const int nch = nph >> 3, col0 = part * nph;
    const uint32_t o_addr = cx.tmem + lane_base + TM_O + col0;
    // A parity wait only tells two consecutive phases of a barrier apart, so a warp may wait for a
    // round's completion only when it knows the round two before to be complete.  The group whose
    // round the last one was not has not looked at that round's barrier for a while: it first waits
    // for the round before (its own, or the one it knows the predecessor of), which brings it close
    // enough.
    const uint32_t last = g - 1;
    if (ngrp == 2 && t > 1) wait_u(cx.pv_done() + 8 * ((last - 1) & 1), ((last - 1) >> 1) & 1);
    wait_u(cx.pv_done() + 8 * (last & 1), (last >> 1) & 1);
    tc_fence_after();
    // column sums: TMEM lane n of the accumulator of the multiplication by ones
    if (part == 0) {
        uint32_t lv[8];
        tmem_ld<8>(cx.tmem + lane_base + TM_L, lv);
        tmem_wait_ld();
        cx.lred[krow] = __uint_as_float(lv[0]);
    } else {
        cx.lred[part * 128 + krow] = 0.f;
    }
    soft_sync();
    const int pair = sg.s * p.hkv + sg.g;
    const int slot = blockIdx.x + pair;
    const bool whole = sg.j0 == 0 && sg.j1 == sg.nt;       // this CTA saw every tile of the pair
    if (TWO && half_of_pair(cx, sg, p.hkv) >= 0) return;   // (one part a CTA: the run's only segment; finish_in_two)
    if (p.pair_cnt && whole) {
        // no other partial exists: normalise and write the output directly
        if (tid < np) cx.alpha[tid] = 1.f / ((cx.lred[tid] + cx.lred[128 + tid]) + (cx.lred[256 + tid] + cx.lred[384 + tid]));
        soft_sync();
        if (!dead) {
            __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(p.out);
#pragma unroll 1
            for (int ch = 0; ch < nch; ++ch) {
                uint32_t ov[8];
                tmem_ld<8>(o_addr + ch * 8, ov);
                tmem_wait_ld();
                int b = (col0 + ch * 8) / G, hg = (col0 + ch * 8) - b * G;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int n = col0 + ch * 8 + i;
                    if (n < M)
                        out[(((size_t)sg.s * p.max_active + b) * p.hq + (size_t)sg.g * G + hg) * D + krow] =
                            __float2bfloat16_rn(__uint_as_float(ov[i]) * cx.alpha[n]);
                    if (++hg == G) {
                        hg = 0;
                        ++b;
                    }
                }
            }
        }
    } else {
        if (!dead) {
            if (tid < M) {
                const float lt = (cx.lred[tid] + cx.lred[128 + tid]) + (cx.lred[256 + tid] + cx.lred[384 + tid]);
                const float mn = cx.mneg[tid];
                *reinterpret_cast<float2*>(p.ws_ml + ((size_t)slot * p.mmax + tid) * 2) = make_float2(mn == UNSET ? -INFINITY : -mn, lt);
            }
            // O^T: lane = head_dim index, column = query row; partials are stored [query row][head_dim]
            float* wo = p.ws_o + (size_t)slot * p.mmax * D + krow;
#pragma unroll 1
            for (int ch = 0; ch < nch; ++ch) {
                uint32_t ov[8];
                tmem_ld<8>(o_addr + ch * 8, ov);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (col0 + ch * 8 + i < M) wo[(size_t)(col0 + ch * 8 + i) * D] = __uint_as_float(ov[i]);
            }
        }
        if (p.pair_cnt) {
            // the CTA that delivers the last partial of a pair merges them all (no second kernel)
            __threadfence();
            soft_sync();
            if (tid == 0) {
                int c_first, c_last;
                pair_ctas(p, cx, sg.s, sg.g, c_first, c_last);
                const int expected = c_last - c_first + 1;               // every CTA in between owns tiles of the pair
                const int old = dead ? -1 : atomicAdd(&p.pair_cnt[pair], 1);
                cx.flags[1] = old == expected - 1;
                cx.flags[2] = c_first;
                cx.flags[3] = c_last;
                if (old == expected - 1) p.pair_cnt[pair] = 0;          // ready for the next call
            }
            soft_sync();
            if (cx.flags[1])
                merge_pair(p.ws_ml, p.ws_o, reinterpret_cast<__nv_bfloat16*>(p.out), pair, p.mmax, M, G, sg.s, sg.g, p.max_active, p.hq,
                           cx.flags[2], cx.flags[3]);
        }
    }
    soft_sync();                     // column state and Q^T are free again
    tc_fence_before();
    __syncwarp();
    if (!dead && lane == 0) mbar_arrive(cx.o_free());
}

// The end of a CTA that has one part of a pair in two (half_of_pair; all softmax warps; the partial sums are in lred).  Half 0 finishes the pair's query columns of
// column parts 0 and 1, half 1 those of 2 and 3, each with what the other CTA hands over through the workspace.
__device__ __forceinline__ void finish_in_two(const AttnParams& p, const Ctx& cx, const Segment& sg, const int nph, const int half, const bool dead, const int warp, const int lane)
{
    const int tid = threadIdx.x, q4 = warp & 3, part = warp >> 2, krow = q4 * 32 + lane;
    const int nch = nph >> 3, col0 = part * nph, G = p.group, M = cx.nact[sg.s] * G;
    const uint32_t o_addr = cx.tmem + ((uint32_t)(q4 * 32) << 16) + TM_O + col0;
    const size_t slot = blockIdx.x + sg.s * p.hkv + sg.g, peer = half ? slot - 1 : slot + 1;
    const bool mine = part >> 1 == half;
    float m = -INFINITY, l = 0.f;                          // (thread = query column)
    if (tid < M) {
        const float mn = cx.mneg[tid];
        m = mn == UNSET ? -INFINITY : -mn;
        l = (cx.lred[tid] + cx.lred[128 + tid]) + (cx.lred[256 + tid] + cx.lred[384 + tid]);
        if (!dead) *reinterpret_cast<float2*>(p.ws_ml + (slot * p.mmax + tid) * 2) = make_float2(m, l);
    }
    if (!mine && !dead) {
        // O^T: lane = head_dim index, column = query row; partials are stored [query row][head_dim]
        float* wo = p.ws_o + slot * p.mmax * D + krow;
#pragma unroll 1
        for (int ch = 0; ch < nch; ++ch) {
            uint32_t ov[8];
            tmem_ld<8>(o_addr + ch * 8, ov);
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (col0 + ch * 8 + i < M) wo[(size_t)(col0 + ch * 8 + i) * D] = __uint_as_float(ov[i]);
        }
    }
    __threadfence();
    soft_sync();
    if (tid == 0 && !dead) arrive_at_peer(cx.peer_done());
    const bool ok = !dead && wait_for_peer(cx.peer_done(), cx.abortp, p.status);         // (else: flagged, no output)
    // the other CTA's values of this thread's columns, all on their way before the first is used
    constexpr int PER = NP_MAX / NPART;
    float z[PER];
    const float* po = p.ws_o + peer * p.mmax * D + krow;
    if (mine && ok)
#pragma unroll
        for (int i = 0; i < PER; ++i) z[i] = i < nph && col0 + i < M ? __ldcg(po + (size_t)(col0 + i) * D) : 0.f;
    if (tid < M && ok) {
        const float2 v = __ldcg(reinterpret_cast<const float2*>(p.ws_ml + (peer * p.mmax + tid) * 2));
        const float nm = fmaxf(m, v.x), ms = nm == -INFINITY ? 0.f : nm, a = fast_exp2(m - ms), w = fast_exp2(v.x - ms);      // (a part that saw nothing: 0)
        const float inv = 1.f / fmaf(v.y, w, l * a);
        cx.alpha[tid] = a * inv;
        cx.lred[tid] = w * inv;
    }
    soft_sync();
    if (mine && ok) {
        __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(p.out);
#pragma unroll
        for (int ch = 0; ch < PER / 8; ++ch)
            if (ch < nch) {
                uint32_t ov[8];
                tmem_ld<8>(o_addr + ch * 8, ov);
                tmem_wait_ld();
                int b = (col0 + ch * 8) / G, hg = (col0 + ch * 8) - b * G;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int n = col0 + ch * 8 + i;
                    if (n < M)
                        out[(((size_t)sg.s * p.max_active + b) * p.hq + (size_t)sg.g * G + hg) * D + krow] =
                            __float2bfloat16_rn(fmaf(z[ch * 8 + i], cx.lred[n], __uint_as_float(ov[i]) * cx.alpha[n]));
                    if (++hg == G) {
                        hg = 0;
                        ++b;
                    }
                }
            }
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
    constexpr int np_max = NP_MAX, npb = 2;
    cx.q_panel = np_max * 128;
    cx.p_buf = ((np_max + 63) / 64) * PANEL;
    // (register allocation: with this one value folded into the address arithmetic the two wider builds
    // spill; kept in a register they do not, or hardly)
    if (NP_MAX > 32) asm volatile("" : "+r"(cx.p_buf));
    cx.npb = npb;
    cx.kring = smem;
    cx.vring = cx.kring + (size_t)nk * STAGE;
    cx.ps = cx.vring + (size_t)nv * STAGE;
    cx.qs = cx.ps + npb * cx.p_buf;
    cx.ones = cx.qs + (D / 64) * cx.q_panel;
    uint64_t* bars = reinterpret_cast<uint64_t*>(cx.ones + ONES_BYTES);
    cx.bar0 = smem_u32(bars);
    cx.ns = 4;
    cx.s_stride = 64;
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 5 * MAXST + 16);
    cx.mneg = reinterpret_cast<float*>(tmem_holder + 4);
    cx.alpha = cx.mneg + 128;
    cx.lred = cx.alpha + 128;
    cx.cmax = reinterpret_cast<int*>(cx.lred + 512);
    cx.flags = cx.cmax + 128;
    cx.rflag = cx.flags + 4;
    cx.pre = cx.rflag + 8;
    cx.nact = cx.pre + p.batch + 1;
    cx.prev = cx.nact + p.batch;
    cx.smask = reinterpret_cast<uint64_t*>(((uintptr_t)(cx.prev + p.batch + 1) + 15) & ~(uintptr_t)15);
    cx.mbuf = MBUF;
    cx.sunion = cx.smask + 2 * cx.mbuf;
    cx.mstaged = p.max_active * p.W <= cx.mbuf;
    __shared__ CtaFlags cta_flags;
    cx.abortp = &cta_flags.abort_flag;
    cx.v_steps = cta_flags.v_steps;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        cta_flags.abort_flag = 0;
    }
    if (threadIdx.x < 8) cx.rflag[threadIdx.x] = -1;
    if (threadIdx.x < ONES_BYTES / 4 && !split_only) {
        reinterpret_cast<uint32_t*>(cx.ones)[threadIdx.x] = 0x3F803F80u;          // bf16 1.0 twice
        fence_async_smem();
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
        for (int i = 0; i < 4; ++i) {
            mbar_init(cx.s_full() + 8 * i, 1);
            mbar_init(cx.s_free() + 8 * i, NSOFT / NGRP);      // the warps of the round's group
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(cx.p_full() + 8 * i, NSOFT / NGRP);
            mbar_init(cx.pv_done() + 8 * i, 2);              // the V multiplications and the column sums
        }
        mbar_init(cx.q_ready(), NSOFT);
        mbar_init(cx.o_free(), NSOFT);
        mbar_init(cx.app_done(), 1);
        if (TWO) mbar_init(cx.peer_done(), 1);
        mbar_init(smem_u32(&cta_flags.raise_bar), NSOFT);
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
        producer_loop<2>(p, cx, &tm_k, &tm_v, lo, hi, lane);
    } else if (warp == W_AUX) {
        aux_loop(p, cx, lo, hi, lane);
    } else if (warp == W_PV) {
        pv_loop(p, cx, lo, hi);
    } else if (warp == W_QK) {
        qk_loop(p, cx, lo, hi);
    } else {
        int s = 0;
        uint32_t g = 0, seg = 0;
        int vst = 0;                              // V ring stage and phase of round g
        uint32_t vph = 0;
        long long u = lo;
        bool dead = false;                        // a bounded wait ran out somewhere in the CTA
        int prefetched = 0;                       // the segment's queries and bitmaps are already on their way
        if (p.early) {
            // ahead of the dependency wait: the first pair's bitmaps; its queries follow right after the wait
            int s0 = 0;
            const Segment sg = decode_segment(lo, hi, cx.pre, p.hkv, s0);
            stage_first_pair_early(reinterpret_cast<const uint4*>(p.q), p.mask, p.max_active, p.W, p.hq, p.group, sg.s, sg.g,
                                   cx.nact[sg.s] * p.group, cx.qs, cx.q_panel, cx.mstaged ? cx.smask : nullptr);
            prefetched = 1;
        }
        while (u < hi) {
            const Segment sg = decode_segment(u, hi, cx.pre, p.hkv, s);
            const int M = cx.nact[sg.s] * p.group;
            softmax_segment(p, cx, sg, ((NP_MAX == 32 || M <= 32) ? 32 : 64) / NPART, seg, hi, prefetched, g, vst, vph, dead, warp, lane);
            ++seg;
            u = sg.next_u;
        }
        if (TWO) {
            s = 0;
            const Segment sg = decode_segment(lo, hi, cx.pre, p.hkv, s);
            const int half = half_of_pair(cx, sg, p.hkv);
            if (half >= 0) finish_in_two(p, cx, sg, ((NP_MAX == 32 || cx.nact[sg.s] * p.group <= 32) ? 32 : 64) / NPART, half, dead, warp, lane);
        }
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

// bf16, head_dim 128, at most 64 query rows per (scene, KV head); FDC_ERR_SHAPE otherwise (the
// caller then takes another kernel).  split_only: the launch only computes the work split of the
// pass into p.split_memo (an ordinary launch; no rings, no TMEM).  This build of the kernel
// serves the launches whose widest pair has 33 to 64 query rows (two groups) or all others (one).
int FDC_TC_LAUNCH(const AttnParams& p, int head_dim, cudaStream_t st, int split_only)
{
    if (head_dim != D || p.mmax > 64) return FDC_ERR_SHAPE;
    const int np_max = p.mmax <= 32 ? 32 : 64;
    const int p_buf = ((np_max + 63) / 64) * PANEL;
    if (np_max != NP_MAX) return FDC_ERR_SHAPE;   // another build's launches
    const int npb = 2;
    static SmemLimit limit;
    int rc = FDC_OK;
    const size_t fixed = 1024 + (size_t)npb * p_buf + (size_t)(D / 64) * np_max * 128 + ONES_BYTES + 8 * (5 * MAXST + 16) + 16 +
                         4 * (128 + 128 + 512 + 128 + 12) + sizeof(int) * (3 * p.batch + 2) + 8 * (2 * MBUF + 2 * UW + 2) + 64;
    int stages = (int)((227 * 1024 - 256 - fixed) / STAGE);
    if (stages > 2 * MAXST) stages = 2 * MAXST;
    if (stages < 4) return FDC_ERR_SHAPE;
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
    {
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
    }
    note_launch();
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? FDC_OK : set_cuda_error(e);
}

}  // namespace fdc
