// FP64 line-resident plane kernels, one size group.
#include "plane_lines.cuh"

WDF_LINES_UNIT(lines_f64_b, double, 45,48,50,54)
