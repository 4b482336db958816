// The row form of the tcgen05 kernel (65 to 128 query rows).
#define FDC_TC_TWO 0
#define FDC_TC_KERNEL attn_tc_rows_kernel
#define FDC_TC_LAUNCH launch_tc_rows
#include "fdc_attn_tc_rows_kernel.cuh"
