// gom_bs8.cu -- the bit-sliced kernels for elements of at most 8 variables.
#include "gom_bs_kernels.cuh"
#include "gom_kernels.cuh"

const void *gom_run_bs8(int r, bool learn) { return learn ? run_bs_kernel<8, true>(r) : run_bs_kernel<8, false>(r); }
const void *gom_mix_bs8(int r, bool learn) { return learn ? mix_bs_kernel<8, true>(r) : mix_bs_kernel<8, false>(r); }
