// Double-float line-resident plane kernels, one size group.
#include "plane_lines.cuh"

WDF_LINES_UNIT(lines_df_b, df64, 36,40,45)
