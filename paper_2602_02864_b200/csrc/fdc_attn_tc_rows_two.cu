// The row form, build for launches whose pairs come in two parts each.
#define FDC_TC_TWO 1
#define FDC_TC_KERNEL attn_tc_rows_kernel_two
#define FDC_TC_LAUNCH launch_tc_rows_two
#include "fdc_attn_tc_rows_kernel.cuh"
