// gom_batch_kernels.cu -- the batched kernel with registers for two blocks of
// 256 threads per SM (the bit-sliced phases among its variants), its selection
// and the collection of the instances' results.
#include "gom_batch_kernels.cuh"

const void *gom_batch_kernel3();

const void *gom_batch_kernel(int minb) { return minb >= 3 ? gom_batch_kernel3() : (const void *)k_batch<2>; }

// After a batched call: each instance's generation count and error word.
__global__ void k_batch_collect(const GomParams *Ps, GomBatchInst *inst, int B)
{
    for (int b = (int)gthread(); b < B; b += (int)gthreads()) {
        const GomDevState *st = Ps[b].st;
        inst[b].gens_run = (int32_t)(st->g - st->call_g0);
        inst[b].err = st->err;
    }
}

