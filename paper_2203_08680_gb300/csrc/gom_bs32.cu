// gom_bs32.cu -- the bit-sliced kernels for elements of at most 32 variables.
#include "gom_bs_kernels.cuh"
#include "gom_kernels.cuh"

const void *gom_run_bs32(int r, bool learn) { return learn ? run_bs_kernel<32, true>(r) : run_bs_kernel<32, false>(r); }
const void *gom_mix_bs32(int r, bool learn) { return learn ? mix_bs_kernel<32, true>(r) : mix_bs_kernel<32, false>(r); }
