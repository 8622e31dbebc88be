// gom_bs8.cu -- the bit-sliced kernels for elements of at most 8 variables.
#include "gom_bs_kernels.cuh"
#include "gom_kernels.cuh"

const void *gom_run_bs8(int r, int ub, bool learn) { return run_bs_kernel<8>(r, ub, learn); }
const void *gom_mix_bs8(int r, int ub, bool learn) { return mix_bs_kernel<8>(r, ub, learn); }
