// The grouped batch's x kernels (MM_FP32).
#include "batch_kernels.cuh"

const void *mm_group_xfwd_fp32() { return (const void *)k_xfwd_group<float>; }
const void *mm_group_xinv_fp32() { return (const void *)k_xinv_group<float>; }
