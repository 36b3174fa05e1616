// The grouped batch's y-z kernel (MM_FP64).
#include "batch_kernels.cuh"

const void *mm_group_yz_fp64() { return (const void *)k_yz_group<double, false>; }
const void *mm_group_yz_sep_fp64() { return (const void *)k_yz_group<double, true>; }
