// Double-float line-resident plane kernels, one size group.
#include "plane_lines.cuh"

WDF_LINES_UNIT(lines_df_a, df64, 24,30,32)
