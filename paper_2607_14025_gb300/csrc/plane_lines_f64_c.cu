// FP64 line-resident plane kernels, one size group.
#include "plane_lines.cuh"

WDF_LINES_UNIT(lines_f64_c, double, 60,64,72)
