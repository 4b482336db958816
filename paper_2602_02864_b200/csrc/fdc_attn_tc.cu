// The tcgen05 split-KV kernel, build for launches whose widest pair has up to 32 query rows (one
// group of softmax warps), and the entry points that choose between the builds.
#define FDC_TC_NGRP 1
#define FDC_TC_NPMAX 32
#define FDC_TC_TWO 0
#define FDC_TC_KERNEL attn_tc_kernel
#define FDC_TC_LAUNCH launch_tc_np32
#include "fdc_attn_tc_kernel.cuh"

namespace fdc {

int launch_tc_np64(const AttnParams& p, int head_dim, cudaStream_t st, int split_only);        // fdc_attn_tc_g2.cu
int launch_tc_rows(const AttnParams& p, int head_dim, cudaStream_t st, int split_only);        // fdc_attn_tc_rows.cu
int launch_tc_np64_two(const AttnParams& p, int head_dim, cudaStream_t st, int split_only);    // fdc_attn_tc_g2_two.cu
int launch_tc_rows_two(const AttnParams& p, int head_dim, cudaStream_t st, int split_only);    // fdc_attn_tc_rows_two.cu

// Launches whose pairs come in two parts each, one per CTA, as long as no scene has ended, go to builds of their own (parts that are spread over the
// pair's list, and that hand each other half of their results): with more than 32 query rows, from 32 tiles a pair on, while all tiles of a
// template, listed at once, still make one part per CTA (equal_shares, as the kernels split them), and where a template as a whole gains by it.
//
// That is where the tiles beyond the prefix are at least half of the list's length, so that the plain builds' second part has nothing that it could
// load ahead of the append, or where a merge by one CTA is long (120 query rows and more).  CTAs that start two by two cost 1 us a launch (blocks that wait for a
// place for both), which passes with few fields at work, as most templates have them at one end, do not win back.  Whole templates, plain build / these (the time of every 8th or 16th
// pass, fan, diamond, wide and free, fields of equal and of drawn lengths, 50 to 74 pairs, prefix 512 to 16384): half and more beyond 1.054 (181 templates, the
// worst 0.984), 120 rows and more otherwise 1.028 (81, 0.990), 65 to 119 rows 1.009 (195, 0.974, 18 of them below 0.985), 33 to 64 rows 0.999 (190,
// 0.957, 42 below 0.985; 8 scenes, 16 fields x 4 heads, prefix 8192: widest passes 1.02, later ones 0.98).  Within these lines single passes lie between 0.90 (most scenes
// ended) and 1.2.  Up to 100 tiles per CTA (row form) and 200: longer lists in one part per CTA (70 to 74 pairs) gain 1.008 (72 templates, prefix 12288 to 24576, 120 rows and
// more), single passes 0.95 to 1.045.
//
// us a layer, without / with: 64 pairs, 128 rows, 48 tiles 38.6 / 34.0; 64 rows, prefix 1024, 32 tiles 32.6 / 27.1.  With
// 16 tiles a pair that start costs more than this gains (64 pairs, 35 rows 21.7 / 23.7), with equal shares nothing is
// handed over (128 rows, 208 tiles, 32 of them beyond the prefix 93.4 / 95.9; 231 tiles, 96 beyond 117.3 / 128.1), and up to 32 rows are merged as fast by the
// CTA that comes last (64 pairs, 24 rows, prefix 4096 34.4 / 34.8; 28 rows, 2048 23.3 / 24.2).
bool pairs_in_two_parts(int64_t pairs, int mmax, int P, int ntile_max, int n_cta)
{
    if (mmax <= 32 || n_cta % 2 || 2 * pairs > n_cta || 3 * pairs <= n_cta || ntile_max < 32) return false;
    const int length = weighted_tiles(P / FDC_TILE_ROWS, ntile_max);
    if (mmax < 120 && 2 * W_PREFIX * (P / FDC_TILE_ROWS) > length) return false;
    if (ntile_max * pairs >= (mmax > 64 ? 100 : 200) * (int64_t)n_cta) return false;
    return !equal_shares(pairs * (length + W_PAIR), (length + 1) / 2, n_cta, mmax);
}

// More than 64 query rows go to the row form.  Measured on both sides of the line (us a layer, transposed / row
// form): 128 rows, 8 scenes, prefix 1024 / 4096 / 32768: 56.6 / 40.7, 90.8 / 61.1, 336 / 212; 84 rows, 8 scenes, prefix
// 4096: 49.8 / 37.8; 126 rows, 4 scenes, prefix 2000: 42.3 / 36.3; 64 rows, 8 scenes, prefix 8192: 61.8 / 62.6; 24 rows, 16
// scenes, prefix 4096: 53.3 / 59.5; 16 rows, 64 scenes, prefix 16384: 629 / 732.
static int launch_tc(const AttnParams& p, int head_dim, cudaStream_t st, int split_only)
{
    if (p.pair_cnt && pairs_in_two_parts((int64_t)p.batch * p.hkv, p.mmax, p.P, p.ntile_max, p.n_cta)) {
        const int rc = p.mmax > 64 ? launch_tc_rows_two(p, head_dim, st, split_only) : launch_tc_np64_two(p, head_dim, st, split_only);
        if (rc != FDC_ERR_SHAPE) return rc;
    }
    if (p.mmax > 64) return launch_tc_rows(p, head_dim, st, split_only);
    if (p.mmax > 32) return launch_tc_np64(p, head_dim, st, split_only);
    return launch_tc_np32(p, head_dim, st, split_only);
}

int launch_attn_tc(const AttnParams& p, int head_dim, cudaStream_t st) { return launch_tc(p, head_dim, st, 0); }
int launch_attn_tc_split(const AttnParams& p, int head_dim, cudaStream_t st) { return launch_tc(p, head_dim, st, 1); }

}  // namespace fdc
