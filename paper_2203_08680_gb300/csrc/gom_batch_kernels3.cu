// gom_batch_kernels3.cu -- the batched kernel with registers for three blocks of
// 256 threads per SM (per-lane variants only).
#include "gom_batch_kernels.cuh"

const void *gom_batch_kernel3() { return (const void *)k_batch<3>; }
