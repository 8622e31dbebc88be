// gom_bs16.cu -- the bit-sliced kernels for elements of at most 16 variables.
#include "gom_bs_kernels.cuh"
#include "gom_kernels.cuh"

const void *gom_run_bs16(int r, bool learn) { return learn ? run_bs_kernel<16, true>(r) : run_bs_kernel<16, false>(r); }
const void *gom_mix_bs16(int r, bool learn) { return learn ? mix_bs_kernel<16, true>(r) : mix_bs_kernel<16, false>(r); }
