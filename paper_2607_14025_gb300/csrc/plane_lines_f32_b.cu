// FP32 line-resident plane kernels, one size group.
#include "plane_lines.cuh"

WDF_LINES_UNIT(lines_f32_b, float, 50,54,60,64)
