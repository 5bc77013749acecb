// Pass kernels of the pair-of-FP32 operator for log2 sizes 5, 6 (launched from
// tbc_df.cu; one unit per group so that they compile in parallel).
#include "df64.cuh"
#include "tbc_apply.cuh"

TBC_PASS_KERNELS(, df, 5)
TBC_B1_KERNEL(, df, 5)
TBC_PASS_KERNELS(, df, 6)
TBC_B1_KERNEL(, df, 6)
