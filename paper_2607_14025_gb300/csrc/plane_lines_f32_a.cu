// FP32 line-resident plane kernels, one size group.
#include "plane_lines.cuh"

WDF_LINES_UNIT(lines_f32_a, float, 24,30,32,36,40,45,48)
