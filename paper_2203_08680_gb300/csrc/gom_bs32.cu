// gom_bs32.cu -- the bit-sliced kernels for elements of at most 32 variables.
#include "gom_bs_kernels.cuh"
#include "gom_kernels.cuh"

const void *gom_run_bs32(int r, int ub, bool learn) { return run_bs_kernel<32>(r, ub, learn); }
const void *gom_mix_bs32(int r, int ub, bool learn) { return mix_bs_kernel<32>(r, ub, learn); }
