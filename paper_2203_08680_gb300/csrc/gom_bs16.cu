// gom_bs16.cu -- the bit-sliced kernels for elements of at most 16 variables.
#include "gom_bs_kernels.cuh"
#include "gom_kernels.cuh"

const void *gom_run_bs16(int r, int ub, bool learn) { return run_bs_kernel<16>(r, ub, learn); }
const void *gom_mix_bs16(int r, int ub, bool learn) { return mix_bs_kernel<16>(r, ub, learn); }
