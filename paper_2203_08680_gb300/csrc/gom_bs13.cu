// gom_bs13.cu -- the bit-sliced kernels for elements of at most 13 variables.
#include "gom_bs_kernels.cuh"
#include "gom_kernels.cuh"

const void *gom_run_bs13(int r, int ub, bool learn) { return run_bs_kernel<13>(r, ub, learn); }
const void *gom_mix_bs13(int r, int ub, bool learn) { return mix_bs_kernel<13>(r, ub, learn); }
