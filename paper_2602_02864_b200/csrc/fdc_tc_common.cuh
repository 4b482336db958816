// What the two tcgen05 kernels share (fdc_attn_tc_kernel.cuh: KV rows on the M side of the multiplications;
// fdc_attn_tc_rows_kernel.cuh: query rows): wrappers of the tensor-core instructions, the work split over the CTAs, the TMA
// producer of the K and V rings and the fused append.  Included once per translation unit.
#pragma once

#include <cudaTypedefs.h>

#include <climits>

#include "fdc_attn_common.cuh"

using namespace fdc;

namespace {

constexpr int D = 128;                       // head_dim handled by these kernels
constexpr int TILE = FDC_TILE_ROWS;          // rows per entry of the visited-tile list
#if !defined(FDC_TC_TWO)
#error "FDC_TC_TWO: 1 for the build that launches whose pairs are cut in two parts are given (pairs_in_two_parts), else 0"
#endif
constexpr bool TWO = FDC_TC_TWO != 0;
constexpr int UW = 64;                       // words of a scene's union bitmap kept in shared memory (when W <= UW)
constexpr int MIN_TILES = 8;                 // tiles per CTA below which fewer CTAs are used (small problems)
constexpr int MIN_UNITS = MIN_TILES * W_PREFIX;   // the same as a weighted length
static_assert(MIN_UNITS >= 2 * W_MASKED, "every part of a pair must contain the start of at least one tile");

// ---------------------------------------------------------------- tcgen05 wrappers
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Shared-memory matrix descriptor (128-byte swizzle, descriptor version 1): start address,
// leading-dimension byte offset, stride-dimension byte offset, all in units of 16 bytes.
// K-major operand: SBO = distance of 8-row groups.  MN-major operand: LBO = distance of
// 64-element groups along M/N, SBO = distance of 8-row groups along K.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo_bytes, uint32_t sbo_bytes)
{
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32) | (1ull << 46) | (2ull << 61);
}
// True in one thread of the (converged) warp.  A region entered by this predicate issues the multiplications faster than
// one behind "lane == 0" (measured: about 60 cycles each against 110).
__device__ __forceinline__ bool elect_one()
{
    uint32_t r;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
    return r != 0;
}
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

#define FDC_R8(v, o) "=r"(v[o + 0]), "=r"(v[o + 1]), "=r"(v[o + 2]), "=r"(v[o + 3]), "=r"(v[o + 4]), "=r"(v[o + 5]), "=r"(v[o + 6]), "=r"(v[o + 7])
#define FDC_I8(v, o) "r"(v[o + 0]), "r"(v[o + 1]), "r"(v[o + 2]), "r"(v[o + 3]), "r"(v[o + 4]), "r"(v[o + 5]), "r"(v[o + 6]), "r"(v[o + 7])
// N consecutive fp32 columns of this thread's TMEM lane (N = 8, 16 or 32).
template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&v)[N])
{
    static_assert(N == 8 || N == 16 || N == 32, "column count");
    if constexpr (N == 32) {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,"
            "%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
            : FDC_R8(v, 0), FDC_R8(v, 8), FDC_R8(v, 16), FDC_R8(v, 24)
            : "r"(taddr)
            : "memory");
    } else if constexpr (N == 16) {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                     : FDC_R8(v, 0), FDC_R8(v, 8)
                     : "r"(taddr)
                     : "memory");
    } else {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];" : FDC_R8(v, 0) : "r"(taddr) : "memory");
    }
}
template <int N>
__device__ __forceinline__ void tmem_st(uint32_t taddr, const uint32_t (&v)[N])
{
    static_assert(N == 8 || N == 16 || N == 32, "column count");
    if constexpr (N == 32) {
        asm volatile(
            "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,"
            "%24,%25,%26,%27,%28,%29,%30,%31};"
            ::FDC_I8(v, 0), FDC_I8(v, 8), FDC_I8(v, 16), FDC_I8(v, 24), "r"(taddr)
            : "memory");
    } else if constexpr (N == 16) {
        asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15};"
                     ::FDC_I8(v, 0), FDC_I8(v, 8), "r"(taddr)
                     : "memory");
    } else {
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};" ::FDC_I8(v, 0), "r"(taddr) : "memory");
    }
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack2(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
// Asynchronous copy global -> shared; completes with cp_async_wait_all.
__device__ __forceinline__ void cp_async8(void* dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all()
{
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// A CTA's view of the pass and of the work split.
struct Split {
    int *pre, *nact;                 // [batch + 1] tile prefix sums, [batch] active branches per scene
    int* prev;                       // [batch + 1] prefix sums over scenes (per KV head) of parts (tpart > 0) or weighted lengths; or nullptr
    int n_cta;                       // CTAs that take part: at most the grid, at least MIN_UNITS tiles each
    int tpart;                       // > 0: every CTA owns one part (at most tpart tiles) of one pair
    int npre;                        // tiles wholly inside the prefix
    long long vtot;                  // total weighted length
};

// ---- weighted work split ---------------------------------------------------------------------
// CTAs get equal shares of a WEIGHTED length, not of the tile count: a tile beyond the prefix
// costs W_MASKED / W_PREFIX prefix tiles and the end of every pair costs W_PAIR / W_PREFIX.  Tile j of a pair starts at
// weighted offset vt(j); a pair of nt tiles is vt(nt) + W_PAIR long.  A CTA owns the tiles whose
// start falls into its share, so shares always cut the unit sequence into consecutive runs.
__device__ __forceinline__ int vt_of(const Split& cx, int nt, int j)
{
    return weighted_tiles(cx.npre < nt ? cx.npre : nt, j);
}
// First tile of a pair of nt tiles whose weighted start is >= r (nt if there is none).
__device__ __forceinline__ int tile_of_vt(const Split& cx, int nt, int r)
{
    const int np = cx.npre < nt ? cx.npre : nt;
    const int j = r <= np * W_PREFIX ? (r + W_PREFIX - 1) / W_PREFIX : np + (r - np * W_PREFIX + W_MASKED - 1) / W_MASKED;
    return j > nt ? nt : j;
}
// Spread parts (the builds for pairs in two parts).  Where a pair is cut for one part per CTA and every part gets at least SPREAD tiles beyond the prefix, a part
// has its share of the prefix AND its share of what lies beyond (the units of such a pair are counted part by part): all parts begin with tiles that
// can be requested ahead of the dependency wait and that cover the append, which the tiles beyond the prefix wait for (a part of those alone idled for
// 4.4 us), and they are equal whatever the two kinds of tile cost.  With fewer of them, and with many parts, a part's few masked tiles and two
// roundings cost more than that (us a pass, one scene, prefix 18250, 126 rows beyond it, 18 parts of a pair: 606 without, 627 spread).
// (In static shared memory: registers held for it cost the kernels that sit at their limit spills, and local memory is far away beside 217 KB of shared
// memory: up to 11 % on passes with short parts.)
constexpr int SPREAD = 4;
__device__ __forceinline__ bool spread_parts(int nt, int np, int k) { return k > 1 && nt - np >= SPREAD * k; }
struct Spread {
    int na, a0, b0;                  // na >= 0: this CTA's part is spread (tiles of the prefix, the first of them, the first beyond)
};
__device__ __forceinline__ Spread& spread_of_cta()
{
    __shared__ Spread x;
    return x;
}
// List entry of the segment's tile t, and how many of its tiles are whole tiles of the prefix (they come first).
__device__ __forceinline__ int tile_entry(const Segment& sg, int t)
{
    if (!TWO) return sg.j0 + t;
    const Spread& x = spread_of_cta();
    return x.na < 0 ? sg.j0 + t : (t < x.na ? x.a0 + t : x.b0 + t - x.na);
}
__device__ __forceinline__ int prefix_tiles(const Segment& sg, int npre)
{
    const int na = TWO ? spread_of_cta().na : -1;
    return na >= 0 ? na : (npre <= sg.j0 ? 0 : (npre < sg.j1 ? npre : sg.j1) - sg.j0);
}
// First unit whose weighted start is >= x.
__device__ __forceinline__ long long unit_of_virt(const AttnParams& p, const Split& cx, long long x)
{
    if (x >= cx.vtot) return (long long)cx.pre[p.batch] * p.hkv;
    int lo = 0, hi = p.batch;                      // largest s with prev[s] * hkv <= x
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if ((long long)cx.prev[mid] * p.hkv <= x) lo = mid;
        else hi = mid;
    }
    int s = lo;
    while (cx.prev[s + 1] == cx.prev[s]) ++s;     // scenes without tiles have no length
    const int V = cx.prev[s + 1] - cx.prev[s], nt = cx.pre[s + 1] - cx.pre[s];
    const long long y = x - (long long)cx.prev[s] * p.hkv;
    const int g = (int)(y / V), r = (int)(y - (long long)g * V);
    return (long long)cx.pre[s] * p.hkv + (long long)g * nt + tile_of_vt(cx, nt, r);
}
// CTAs that hold the first and the last tile of pair (s, g).
__device__ __forceinline__ void pair_ctas(const AttnParams& p, const Split& cx, int s, int g, int& c_first, int& c_last)
{
    const int nt = cx.pre[s + 1] - cx.pre[s];
    if (cx.tpart) {                                // one part per CTA: the pair's parts are consecutive CTAs
        const int k = cx.prev[s + 1] - cx.prev[s];
        c_first = cx.prev[s] * p.hkv + g * k;
        c_last = c_first + k - 1;
    } else if (!cx.prev) {
        const long long u0 = (long long)cx.pre[s] * p.hkv + (long long)g * nt, U = (long long)cx.pre[p.batch] * p.hkv;
        c_first = unit_cta(u0, U, cx.n_cta);
        c_last = unit_cta(u0 + nt - 1, U, cx.n_cta);
    } else {
        const long long v0 = (long long)cx.prev[s] * p.hkv + (long long)g * (cx.prev[s + 1] - cx.prev[s]);
        c_first = (int)((v0 * cx.n_cta) / cx.vtot);
        c_last = (int)(((v0 + vt_of(cx, nt, nt - 1)) * cx.n_cta) / cx.vtot);
    }
}

// The CTA's run of units.
// The layers of one forward pass see the same per-scene counts, so the work split is made once
// per pass (a launch of this kernel with split_only set) and kept in the memo, with the counts it
// was computed from.  The memo's loads and those of the counts are all issued before the first
// use, so that they share one trip to memory; when they may be read ahead of the dependency wait
// issue() is called there, and the trip hides behind the set-up.
template <int THREADS>
struct SplitFinder {
    static constexpr int MEMO_MAGIC = 0x5D180000 | (TWO ? 0x02000000 : 0) | (W_PREFIX << 12) | (W_MASKED << 8) | W_PAIR;
    const int32_t* mrd;
    int4 mh0, mh1, mh2, me, msp;
    int m_na, m_nt, m_prev;
    int na[4], nt[4];

    __device__ __forceinline__ SplitFinder(const AttnParams& p, int split_only) : mrd((p.split_memo && !split_only) ? p.split_memo : nullptr)
    {
        mh0 = mh1 = mh2 = me = msp = make_int4(0, 0, 0, 0);
        m_na = m_nt = -1;
        m_prev = 0;
    }
    __device__ __forceinline__ void issue(const AttnParams& p)
    {
        if (mrd) {
            mh0 = __ldcg(reinterpret_cast<const int4*>(mrd));
            mh1 = __ldcg(reinterpret_cast<const int4*>(mrd) + 1);
            mh2 = __ldcg(reinterpret_cast<const int4*>(mrd) + 2);
            me = __ldcg(reinterpret_cast<const int4*>(mrd + FDC_MEMO_ENTRIES) + blockIdx.x);
            if (TWO && threadIdx.x == 0) msp = __ldcg(reinterpret_cast<const int4*>(mrd + FDC_MEMO_SPREAD) + blockIdx.x);
            if ((int)threadIdx.x < p.batch) {
                m_na = __ldcg(mrd + 16 + threadIdx.x);
                m_nt = __ldcg(mrd + 16 + FDC_MEMO_BATCH + threadIdx.x);
            }
            if ((int)threadIdx.x <= p.batch) m_prev = __ldcg(mrd + 16 + 2 * FDC_MEMO_BATCH + threadIdx.x);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int i = threadIdx.x + j * THREADS;
            na[j] = i < p.batch ? p.n_active[i] : 0;
            nt[j] = i < p.batch ? p.ntiles[i] : 0;
        }
    }
    // Fills cx and returns whether this CTA has units (all threads; lo, hi: its run).
    __device__ __forceinline__ bool find(const AttnParams& p, Split& cx, const int split_only, long long& lo, long long& hi)
    {
        bool active = true;
        lo = hi = 0;
        // the raw tile counts wait in prev[] for the scan
        {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int i = threadIdx.x + j * THREADS;
                if (i < p.batch) {
                    cx.nact[i] = na[j];
                    cx.prev[i] = nt[j];
                }
            }
            for (int i = threadIdx.x + 4 * THREADS; i < p.batch; i += THREADS) {
                cx.nact[i] = p.n_active[i];
                cx.prev[i] = p.ntiles[i];
            }
        }
        __syncthreads();
        const long long total = scan_ntiles(cx.prev, p.batch, cx.pre);
        const long long U = total * p.hkv;
        if (U == 0) active = false;
        cx.tpart = 0;
        cx.n_cta = p.n_cta;
        cx.vtot = 0;
        cx.npre = p.P / TILE;
        bool hit = false;
        if (mrd) {
            int same = mh0.x == MEMO_MAGIC && mh0.y == (int)p.seq && mh0.z == p.hkv && mh0.w == p.n_cta && mh1.x == p.P && mh1.y == p.batch;
            if ((int)threadIdx.x < p.batch) same = same && m_na == cx.nact[threadIdx.x] && m_nt == cx.pre[threadIdx.x + 1] - cx.pre[threadIdx.x];
            hit = __syncthreads_and(same) != 0;
        }
        if (hit) {
            // same counts as the launch before: its split stands
            cx.tpart = mh1.z;
            cx.n_cta = mh1.w;
            cx.vtot = ((long long)mh2.y << 32) | (uint32_t)mh2.x;
            if ((int)threadIdx.x <= p.batch) cx.prev[threadIdx.x] = m_prev;
            if (TWO && threadIdx.x == 0) spread_of_cta() = Spread{msp.x, msp.y, msp.z};
            __syncthreads();
            lo = ((long long)me.y << 32) | (uint32_t)me.x;
            hi = ((long long)me.w << 32) | (uint32_t)me.z;
        } else if (!active) {
        } else if (p.pair_cnt) {
            // This kernel also merges the partial results of a pair.  Ending one pair and starting the
            // next inside a CTA costs as much as streaming a dozen tiles (drain, partial write, merge,
            // new queries), so while there are no more pairs than CTAs every CTA gets ONE part of ONE
            // pair: pairs are cut into the fewest equal parts of at most tpart (weighted) tiles, tpart the smallest
            // size (at least MIN_UNITS) for which the parts do not outnumber the CTAs.  With more pairs
            // than CTAs, CTAs get equal shares of a weighted length (see above).
            cx.npre = p.P / TILE;
            __shared__ int split_tpart, split_max, split_pairs;
            if (threadIdx.x == 0) {
                split_tpart = 0x7fffffff;
                split_max = 0;
                split_pairs = 0;
            }
            __syncthreads();
            {
                int nsc = 0, mx = 0;
                for (int i = threadIdx.x; i < p.batch; i += THREADS) {
                    const int nt = cx.pre[i + 1] - cx.pre[i];
                    nsc += nt > 0;
                    mx = nt > mx ? nt : mx;
                }
                if (nsc) {
                    atomicAdd(&split_pairs, nsc);
                    atomicMax(&split_max, mx);
                }
            }
            __syncthreads();
            const bool one_part = (long long)split_pairs * p.hkv <= p.n_cta;
            if (one_part) {
                // every thread tries sizes of its own; the smallest that fits wins
                const uint32_t vmax = (uint32_t)vt_of(cx, split_max, split_max);
                const uint32_t tl = vmax < (uint32_t)MIN_UNITS ? vmax : (uint32_t)MIN_UNITS;
                const uint32_t budget = (uint32_t)(p.n_cta / p.hkv);          // parts per KV head
                for (uint32_t T = tl + threadIdx.x; T <= vmax && T < (uint32_t)split_tpart; T += THREADS) {
                    uint32_t cnt = 0;
                    for (int i = 0; i < p.batch; ++i) {
                        const int nt = cx.pre[i + 1] - cx.pre[i];
                        cnt += ((uint32_t)vt_of(cx, nt, nt) + T - 1) / T;
                    }
                    if (cnt <= budget) {
                        atomicMin(&split_tpart, (int)T);
                        break;
                    }
                }
            } else if (threadIdx.x == 0) {
                split_tpart = 0;
            }
            __syncthreads();
            if (one_part && threadIdx.x == 0) {
                long long tot = 0;
                for (int i = 0; i < p.batch; ++i) {
                    const int nt = cx.pre[i + 1] - cx.pre[i];
                    if (nt > 0) tot += vt_of(cx, nt, nt) + W_PAIR;
                }
                if (equal_shares(tot * p.hkv, split_tpart, p.n_cta, p.mmax)) split_tpart = 0;
            }
            __syncthreads();
            if (threadIdx.x < 32) {
                const uint32_t T = (uint32_t)split_tpart;
                int carry = 0;
                for (int b0 = 0; b0 < p.batch; b0 += 32) {
                    const int i = b0 + threadIdx.x;
                    int x = 0;
                    if (i < p.batch) {
                        const int nt = cx.pre[i + 1] - cx.pre[i];
                        x = T ? (int)(((uint32_t)vt_of(cx, nt, nt) + T - 1) / T) : (nt > 0 ? vt_of(cx, nt, nt) + W_PAIR : 0);
                    }
                    int inc = x;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(0xffffffffu, inc, o);
                        if ((int)threadIdx.x >= o) inc += y;
                    }
                    if (i < p.batch) cx.prev[i] = carry + inc - x;
                    carry += __shfl_sync(0xffffffffu, inc, 31);
                }
                if (threadIdx.x == 0) cx.prev[p.batch] = carry;
            }
            __syncthreads();
            cx.tpart = split_tpart;
            if (cx.tpart) {
                const int c = blockIdx.x;
                cx.n_cta = cx.prev[p.batch] * p.hkv;
                if (c < cx.n_cta) {
                    int sl = 0, sh = p.batch;              // largest s with prev[s] * hkv <= c
                    while (sh - sl > 1) {
                        const int mid = (sl + sh) >> 1;
                        if (cx.prev[mid] * p.hkv <= c) sl = mid;
                        else sh = mid;
                    }
                    while (cx.prev[sl + 1] == cx.prev[sl]) ++sl;          // scenes without tiles have no parts
                    const int k = cx.prev[sl + 1] - cx.prev[sl], nt = cx.pre[sl + 1] - cx.pre[sl];
                    const uint32_t idx = (uint32_t)(c - cx.prev[sl] * p.hkv), g = idx / (uint32_t)k, i = idx - g * (uint32_t)k;
                    const uint32_t V = (uint32_t)vt_of(cx, nt, nt);       // part i: tiles whose weighted start lies in [i V / k, (i + 1) V / k)
                    int j0 = tile_of_vt(cx, nt, (int)((i * V + k - 1) / (uint32_t)k));
                    int j1 = tile_of_vt(cx, nt, (int)(((i + 1) * V + k - 1) / (uint32_t)k));
                    const int np = cx.npre < nt ? cx.npre : nt;
                    if (TWO && spread_parts(nt, np, k)) {
                        j0 = np * (int)i / k + (nt - np) * (int)i / k;
                        j1 = np * ((int)i + 1) / k + (nt - np) * ((int)i + 1) / k;
                    }
                    lo = (long long)cx.pre[sl] * p.hkv + (long long)g * nt + j0;
                    hi = lo + (j1 - j0);
                }
            } else {
                const long long want = (U + MIN_TILES - 1) / MIN_TILES;      // small problems use fewer CTAs
                if (want < cx.n_cta) cx.n_cta = (int)want;
                cx.vtot = (long long)cx.prev[p.batch] * p.hkv;
                lo = unit_of_virt(p, cx, cta_first_unit(blockIdx.x, cx.vtot, cx.n_cta));
                hi = unit_of_virt(p, cx, cta_first_unit(blockIdx.x + 1, cx.vtot, cx.n_cta));
            }
        } else {
            cx.prev = nullptr;
            lo = cta_first_unit(blockIdx.x, U, cx.n_cta);
            hi = cta_first_unit(blockIdx.x + 1, U, cx.n_cta);
        }
        if (lo >= hi || (int)blockIdx.x >= cx.n_cta) active = false;
        if (TWO && !hit) {
            if (threadIdx.x == 0) {
                Spread& x = spread_of_cta();
                x = Spread{-1, 0, 0};
                if (active && cx.tpart && p.W >= 2 * SPREAD - 1) {       // (else no pair has that many tiles beyond the prefix)
                    int s = 0;
                    const Segment sg = decode_segment(lo, hi, cx.pre, p.hkv, s);
                    const int np = cx.npre < sg.nt ? cx.npre : sg.nt, k = cx.prev[s + 1] - cx.prev[s];
                    if (spread_parts(sg.nt, np, k)) {
                        const int i = (int)blockIdx.x - (cx.prev[s] * p.hkv + sg.g * k);
                        x.a0 = np * i / k;
                        x.na = np * (i + 1) / k - x.a0;
                        x.b0 = np + (sg.nt - np) * i / k;
                    }
                }
            }
            __syncthreads();
        }
        if (split_only) {
            // this launch only computes the split and leaves it to the attention launches of the pass
            int32_t* mwr = p.split_memo;
            if (threadIdx.x == 0)
                reinterpret_cast<int4*>(mwr + FDC_MEMO_ENTRIES)[blockIdx.x] =
                    active ? make_int4((int)(uint32_t)lo, (int)(lo >> 32), (int)(uint32_t)hi, (int)(hi >> 32)) : make_int4(0, 0, 0, 0);
            if (TWO && threadIdx.x == 0)
                reinterpret_cast<int4*>(mwr + FDC_MEMO_SPREAD)[blockIdx.x] = make_int4(spread_of_cta().na, spread_of_cta().a0, spread_of_cta().b0, 0);
            if (blockIdx.x == 0) {
                if (threadIdx.x == 0) {
                    reinterpret_cast<int4*>(mwr)[0] = make_int4(MEMO_MAGIC, (int)p.seq, p.hkv, p.n_cta);
                    reinterpret_cast<int4*>(mwr)[1] = make_int4(p.P, p.batch, cx.tpart, cx.n_cta);
                    reinterpret_cast<int4*>(mwr)[2] = make_int4((int)(uint32_t)cx.vtot, (int)(cx.vtot >> 32), 0, 0);
                }
                if ((int)threadIdx.x < p.batch) {
                    mwr[16 + threadIdx.x] = cx.nact[threadIdx.x];
                    mwr[16 + FDC_MEMO_BATCH + threadIdx.x] = cx.pre[threadIdx.x + 1] - cx.pre[threadIdx.x];
                }
                if ((int)threadIdx.x <= p.batch) mwr[16 + 2 * FDC_MEMO_BATCH + threadIdx.x] = U > 0 ? cx.prev[threadIdx.x] : 0;
            }
        }
        if (split_only) active = false;
        return active;
    }
};

// ---- pairs in two parts -----------------------------------------------------------------------
// The launch's CTAs come in clusters of two, so the two CTAs of a pair that is cut in two (consecutive, the first one even) are on the chip
// together and may wait for one another: each hands the other one half of its partial result through the workspace, finishes the other half itself
// and no CTA merges alone.  Every thread of the launch arrives at the cluster's barrier when its block's barriers stand, and waits there ahead of its role; and
// again at the very end, so that no block leaves while the other one may still signal it.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// One arrival at the other block's barrier at the same place; everything the thread has written or seen written is known to who sees it.
__device__ __forceinline__ void arrive_at_peer(uint32_t bar)
{
    asm volatile(
        "{\n\t.reg .b32 r, a;\n\tmov.u32 r, %cluster_ctarank;\n\txor.b32 r, r, 1;\n\tmapa.shared::cluster.u32 a, %0, r;\n\t"
        "mbarrier.arrive.release.cluster.shared::cluster.b64 _, [a];\n\t}" ::"r"(bar)
        : "memory");
}
// (bounded like every in-kernel wait; the outcome is the warp's)
__device__ __forceinline__ bool wait_for_peer(uint32_t bar, volatile int* abort_flag, int32_t* status)
{
    bool ok = mbar_wait_warp(bar, 0, abort_flag, status);
    asm volatile("fence.acq_rel.cluster;" ::: "memory");
    return ok;
}
// This CTA's place in a pair cut in two: 0 or 1; -1: not such a pair, or not in one cluster.
__device__ __forceinline__ int half_of_pair(const Split& cx, const Segment& sg, int hkv)
{
    if (!cx.tpart || cx.prev[sg.s + 1] - cx.prev[sg.s] != 2) return -1;
    const int c_first = cx.prev[sg.s] * hkv + sg.g * 2;
    return (c_first & 1) ? -1 : (int)blockIdx.x - c_first;
}

// Position of one ring's producer in the CTA's unit sequence.
struct Cursor {
    long long u;                 // first unit of the current segment
    Segment sg;
    int s, jb, jn, k, my_tile;   // scene hint; batch of up to 32 tile ids (one per lane; jb: the segment's tiles ahead of it) and the position inside it
    uint32_t g;                  // round
    int st;                      // ring stage of round g
    uint32_t ph;                 // ring phase of round g
    int live;
};
__device__ __forceinline__ void cursor_batch(Cursor& c, const AttnParams& p, int lane)
{
    const int n = c.sg.j1 - c.sg.j0;
    c.jn = n - c.jb < 32 ? n - c.jb : 32;
    // entry j of a tile list is tile j for every whole tile of the prefix: no need to read those
    const int j = tile_entry(c.sg, c.jb + lane);
    c.my_tile = lane < c.jn ? (j < p.P / TILE ? j : p.tiles[(size_t)c.sg.s * p.ntile_max + j]) : 0;
    c.k = 0;
}
__device__ __forceinline__ void cursor_open(Cursor& c, const AttnParams& p, const Split& cx, long long hi, int lane)
{
    c.live = c.u < hi;
    if (!c.live) return;
    c.sg = decode_segment(c.u, hi, cx.pre, p.hkv, c.s);
    c.jb = 0;
    cursor_batch(c, p, lane);
}
template <int TPS>
__device__ __forceinline__ void cursor_next(Cursor& c, const AttnParams& p, const Split& cx, long long hi, int nst, int lane)
{
    c.k += TPS;
    ++c.g;
    if (++c.st == nst) {
        c.st = 0;
        c.ph ^= 1;
    }
    if (c.k < c.jn) return;
    c.jb += 32;
    if (c.jb < c.sg.j1 - c.sg.j0) {
        cursor_batch(c, p, lane);
    } else {
        c.u = c.sg.next_u;
        cursor_open(c, p, cx, hi, lane);
    }
}
// Does the stage at the cursor reach beyond the prefix?  (whole warp; tile ids ascend)
template <int TPS>
__device__ __forceinline__ bool cursor_beyond_prefix(const Cursor& c, int P)
{
    const int nt = c.jn - c.k < TPS ? 1 : TPS;
    return __shfl_sync(0xffffffffu, c.my_tile, (c.k + nt - 1) & 31) * TILE + TILE > P;
}
// The stage at the cursor: TPS tiles (one or two), rows 0-63 and 64-127 of both 64-column panels.
template <int TPS>
__device__ __forceinline__ void cursor_issue(const Cursor& c, const CUtensorMap* tm, unsigned char* ring, uint32_t full, uint64_t pol, int lane)
{
    constexpr int PANEL = TPS * TILE * 128, STAGE = (D / 64) * PANEL;
    const int nt = c.jn - c.k < TPS ? 1 : TPS;
    const int t0 = __shfl_sync(0xffffffffu, c.my_tile, c.k);
    const int t1 = TPS == 2 ? __shfl_sync(0xffffffffu, c.my_tile, (c.k + 1) & 31) : 0;
    if (lane == 0) {
        const uint32_t dst = smem_u32(ring + (size_t)c.st * STAGE);
        mbar_expect_tx(full + 8 * c.st, nt * (STAGE / TPS));
#pragma unroll
        for (int h = 0; h < D / 64; ++h) {
            tma_load_4d_hint(dst + h * PANEL, tm, full + 8 * c.st, h * 64, t0 * TILE, c.sg.g, c.sg.s, pol);
            if (TPS == 2 && nt == 2) tma_load_4d_hint(dst + h * PANEL + TILE * 128, tm, full + 8 * c.st, h * 64, t1 * TILE, c.sg.g, c.sg.s, pol);
        }
    }
}

// One TMA producer warp for both rings: whichever of the next K stage and the next V stage is
// free gets its round's tiles; the warp never blocks on one ring while the other could be fed.
template <int TPS, class Ctx>
__device__ __forceinline__ void producer_loop(const AttnParams& p, const Ctx& cx, const CUtensorMap* tm_k, const CUtensorMap* tm_v,
                                              long long lo, long long hi, int lane)
{
    const uint64_t pol = l2_evict_first_policy();     // every KV row is read once per call
    Cursor ck, cv;
    ck.u = lo;
    ck.s = 0;
    ck.g = 0;
    ck.st = 0;
    ck.ph = 0;
    cursor_open(ck, p, cx, hi, lane);
    cv = ck;
    int ok = 1;
    uint32_t idle = 0;
    int app_ok = p.app_row == nullptr;               // rows appended by this kernel are in place (tiles beyond the prefix may be loaded)
    int waited = !p.early;                           // the kernel ahead in the stream has completed (griddepcontrol.wait was taken)
    int q_hold = p.early;                            // after the wait, the first pair's queries go ahead of further K/V requests
    while ((ck.live || cv.live) && ok) {
        if (!app_ok && waited) {
            const int done = lane == 0 ? (int)mbar_try(cx.app_done(), 0) : 0;
            app_ok = __shfl_sync(0xffffffffu, done, 0);
        }
        // Rows beyond the prefix may have been written by the kernel ahead (fdc_kv_append) or are written
        // by this one (fused append): their tiles wait for both.  Prefix rows never change during decode.
        if (q_hold && waited) {
            // The queries are requested right after the wait; whatever this SM requests before them
            // arrives before them.  The stages requested ahead of the wait keep the first rounds fed.
            const int done = lane == 0 ? (int)mbar_try(cx.q_ready(), 0) : 0;
            q_hold = !__shfl_sync(0xffffffffu, done, 0);
        }
        const bool hold_all = q_hold && waited;
        const bool hold_k = hold_all || (!(app_ok && waited) && ck.live && cursor_beyond_prefix<TPS>(ck, p.P));
        const bool hold_v = hold_all || (!(app_ok && waited) && cv.live && cursor_beyond_prefix<TPS>(cv, p.P));
        int rk = 0, rv = 0;
        if (lane == 0) {
            rk = ck.live && !hold_k && mbar_try(cx.k_empty() + 8 * ck.st, ck.ph ^ 1);
            rv = cv.live && !hold_v && mbar_try(cx.v_empty() + 8 * cv.st, cv.ph ^ 1);
        }
        rk = __shfl_sync(0xffffffffu, rk, 0);
        rv = __shfl_sync(0xffffffffu, rv, 0);
        if (rk) {
            cursor_issue<TPS>(ck, tm_k, cx.kring, cx.k_full(), pol, lane);
            cursor_next<TPS>(ck, p, cx, hi, cx.nk, lane);
        }
        if (rv) {
            cursor_issue<TPS>(cv, tm_v, cx.vring, cx.v_full(), pol, lane);
            cursor_next<TPS>(cv, p, cx, hi, cx.nv, lane);
        }
        if (rk | rv) {
            idle = 0;
        } else if (!waited) {
            // nothing more can be requested ahead of the kernel before this one: wait for it to complete
            asm volatile("griddepcontrol.wait;" ::: "memory");
            waited = 1;
        } else if (((++idle) & 63u) == 0u) {
            // bounded: no stage became free for a long time, or another role gave up
            if (idle >= SPIN_LIMIT) {
                if (lane == 0) {
                    *cx.abortp = 1;
                    atomicOr(p.status, FDC_DEV_TIMEOUT);
                }
                ok = 0;
            } else if (*cx.abortp) {
                ok = 0;
            } else {
                __nanosleep(32);
            }
        }
    }
    if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");     // (a run wholly inside the prefix that fitted the rings)
    if (!ok && lane == 0) {
        // give the copies already in flight a bounded chance to land before the CTA ends
        for (int r = 0; r < 2; ++r) {
            const uint32_t g = r ? cv.g : ck.g, nst = r ? cx.nv : cx.nk, full = r ? cx.v_full() : cx.k_full();
            const uint32_t first = g > nst ? g - nst : 0;
            for (uint32_t k = first; k < g; ++k) {
                const uint32_t bar = full + 8 * (k % nst), ph = (k / nst) & 1;
                for (uint32_t i = 0; i < (1u << 16) && !mbar_try(bar, ph); ++i) __nanosleep(64);
            }
        }
    }
}

// Fused append (one warp; out of line, all arguments by value).  The new K/V vectors of this pass
// (Sec. 3.3: every emitted token's K/V is written once, at the row its slot reserves) whose rows
// lie in KV tiles that this CTA owns are written here, before the CTA loads those tiles: every
// tile of a (scene, KV head) pair belongs to exactly one CTA, so every vector is written exactly
// once and no CTA depends on another.  Lanes 0-15 copy the 16 chunks of a K row, lanes 16-31
// those of the V row.  Rows outside [P, rows) are skipped and flagged.  The writes are made
// visible to the TMA loads (asynchronous proxy) of this CTA before the caller signals them.
template <int TURN>
__device__ __noinline__ void append_rows(char* kc, char* vc, long long stride_scene_b, long long stride_head_b, long long stride_row_b,
                                         const int32_t* app_row, const char* app_k, const char* app_v, const int32_t* tiles,
                                         int ntile_max, int max_active, int hkv, int rows, int P, const int* pre, const int* nact,
                                         long long lo, long long hi, int32_t* status)
{
    const int lane = threadIdx.x & 31;
    const int chunk = (lane & 15) * 16;
    const char* src_base = lane < 16 ? app_k : app_v;
    char* dst_base = lane < 16 ? kc : vc;
    int s = 0;
    long long u = lo;
    while (u < hi) {
        const Segment sg = decode_segment(u, hi, pre, hkv, s);
        const int A = nact[sg.s];
        int j0 = sg.j0, j1 = sg.j1;
        if (TWO) {                                     // (a new row is in no whole tile of the prefix)
            const int n = sg.j1 - sg.j0, na = prefix_tiles(sg, P / TILE);
            j0 = na < n ? tile_entry(sg, na) : 0;
            j1 = na < n ? tile_entry(sg, n - 1) + 1 : 1;
        }
        const int t_first = tiles[(size_t)sg.s * ntile_max + j0], t_last = tiles[(size_t)sg.s * ntile_max + j1 - 1];
        for (int b0 = 0; b0 < A; b0 += 32) {
            const int b = b0 + lane;
            const int r = b < A ? app_row[(size_t)sg.s * max_active + b] : P;
            const bool in_range = r >= P && r < rows;
            if (!in_range && sg.g == 0 && sg.j0 == 0) atomicOr(status, FDC_DEV_ROW_RANGE);      // once per scene
            const int t = r / TILE;
            unsigned m = __ballot_sync(0xffffffffu, b < A && in_range && t >= t_first && t <= t_last);
            while (m) {
                // up to TURN rows per turn, all loads before the first store (the tiles beyond the prefix wait for this)
                uint4 val[TURN];
                long long dst[TURN];
#pragma unroll
                for (int i = 0; i < TURN; ++i) {
                    dst[i] = -1;
                    if (m) {
                        const int bi = __ffs(m) - 1;
                        m &= m - 1;
                        const int ri = __shfl_sync(0xffffffffu, r, bi);
                        const size_t slot = (size_t)sg.s * max_active + b0 + bi;
                        val[i] = *reinterpret_cast<const uint4*>(src_base + (slot * hkv + sg.g) * (D * 2) + chunk);
                        dst[i] = (long long)sg.s * stride_scene_b + (long long)sg.g * stride_head_b + (long long)ri * stride_row_b + chunk;
                    }
                }
#pragma unroll
                for (int i = 0; i < TURN; ++i)
                    if (dst[i] >= 0) *reinterpret_cast<uint4*>(dst_base + dst[i]) = val[i];
            }
        }
        u = sg.next_u;
    }
    __threadfence();
    asm volatile("fence.proxy.async;" ::: "memory");
    __syncwarp();
}

// Rows of a KV tile beyond the prefix that some branch of the scene may see (the OR of the
// branches' bitmaps; prefix rows of a tile that straddles the end of the prefix included).  `un` is
// that OR as the softmax warps prepared it per pair (the usual case), else nullptr and the bitmaps
// themselves are combined here (templates too long for the shared-memory copy).
__device__ __noinline__ uint64_t tile_seen_rows(const uint64_t* un, const uint64_t* mask0, int W, int P, int A, int tile)
{
    if (un) return tile_rowmask(un, W, P, tile);
    // (whole warp: the lanes share the branches and combine)
    const int lane = threadIdx.x & 31;
    uint64_t um = 0ull;
    for (int b = lane; b < A; b += 32) um |= tile_rowmask(mask0 + (size_t)b * W, W, P, tile);
    const uint32_t ul = __reduce_or_sync(0xffffffffu, (uint32_t)um);
    const uint32_t uh = __reduce_or_sync(0xffffffffu, (uint32_t)(um >> 32));
    return ((uint64_t)uh << 32) | ul;
}

}  // namespace
