// FP32 line-resident plane kernels, one size group.
#include "plane_lines.cuh"

WDF_LINES_UNIT(lines_f32_c, float, 72,75,80,96)
