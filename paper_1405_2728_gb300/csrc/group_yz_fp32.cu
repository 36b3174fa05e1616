// The grouped batch's y-z kernel (MM_FP32).
#include "batch_kernels.cuh"

const void *mm_group_yz_fp32() { return (const void *)k_yz_group<float, false>; }
