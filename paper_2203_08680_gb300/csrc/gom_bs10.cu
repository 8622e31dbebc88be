// gom_bs10.cu -- the bit-sliced kernels for elements of at most 10 variables.
#include "gom_bs_kernels.cuh"
#include "gom_kernels.cuh"

const void *gom_run_bs10(int r, int ub, bool learn) { return run_bs_kernel<10>(r, ub, learn); }
const void *gom_mix_bs10(int r, int ub, bool learn) { return mix_bs_kernel<10>(r, ub, learn); }
