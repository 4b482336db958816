// The tcgen05 split-KV kernel for 33 to 64 query rows, build for launches whose pairs come in two parts each.
#define FDC_TC_NGRP 2
#define FDC_TC_NPMAX 64
#define FDC_TC_TWO 1
#define FDC_TC_KERNEL attn_tc_kernel_g2_two
#define FDC_TC_LAUNCH launch_tc_np64_two
#include "fdc_attn_tc_kernel.cuh"
