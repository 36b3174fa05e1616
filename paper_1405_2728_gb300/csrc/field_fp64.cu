// Field kernels and their launchers instantiated for one precision:
// double fields, convolution in block fixed point (MM_FP64).
#include "field_launch.cuh"

MM_DEFINE_FIELD_ENTRIES(fp64, double, fx)
