// The grouped batch's x kernels (MM_FP64).
#include "batch_kernels.cuh"

const void *mm_group_xfwd_fp64() { return (const void *)k_xfwd_group<double>; }
const void *mm_group_xinv_fp64() { return (const void *)k_xinv_group<double>; }
