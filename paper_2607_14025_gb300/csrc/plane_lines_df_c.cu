// Double-float line-resident plane kernels, one size group.
#include "plane_lines.cuh"

WDF_LINES_UNIT(lines_df_c, df64, 48,50,54)
