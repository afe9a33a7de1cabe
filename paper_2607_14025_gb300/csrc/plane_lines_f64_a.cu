// FP64 line-resident plane kernels, one size group.
#include "plane_lines.cuh"

WDF_LINES_UNIT(lines_f64_a, double, 24,30,32,36,40)
