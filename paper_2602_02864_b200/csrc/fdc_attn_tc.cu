// The tcgen05 split-KV kernel, build for launches whose widest pair has up to 32 query rows (one
// group of softmax warps), and the entry points that choose between the builds.
#define FDC_TC_NGRP 1
#define FDC_TC_NPMAX 32
#define FDC_TC_KERNEL attn_tc_kernel
#define FDC_TC_LAUNCH launch_tc_np32
#include "fdc_attn_tc_kernel.cuh"

namespace fdc {

int launch_tc_np64(const AttnParams& p, int head_dim, cudaStream_t st, int split_only);    // fdc_attn_tc_g2.cu
int launch_tc_rows(const AttnParams& p, int head_dim, cudaStream_t st, int split_only);    // fdc_attn_tc_rows.cu

// More than 64 query rows go to the row form.  Measured on both sides of the line (us a layer, transposed / row
// form): 128 rows, 8 scenes, prefix 1024 / 4096 / 32768: 56.6 / 40.7, 90.8 / 61.1, 336 / 212; 84 rows, 8 scenes, prefix
// 4096: 49.8 / 37.8; 126 rows, 4 scenes, prefix 2000: 42.3 / 36.3; 64 rows, 8 scenes, prefix 8192: 61.8 / 62.6; 24 rows, 16
// scenes, prefix 4096: 53.3 / 59.5; 16 rows, 64 scenes, prefix 16384: 629 / 732.
static int launch_tc(const AttnParams& p, int head_dim, cudaStream_t st, int split_only)
{
    if (p.mmax > 64) return launch_tc_rows(p, head_dim, st, split_only);
    if (p.mmax > 32) return launch_tc_np64(p, head_dim, st, split_only);
    return launch_tc_np32(p, head_dim, st, split_only);
}

int launch_attn_tc(const AttnParams& p, int head_dim, cudaStream_t st) { return launch_tc(p, head_dim, st, 0); }
int launch_attn_tc_split(const AttnParams& p, int head_dim, cudaStream_t st) { return launch_tc(p, head_dim, st, 1); }

}  // namespace fdc
