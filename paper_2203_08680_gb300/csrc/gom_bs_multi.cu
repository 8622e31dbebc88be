// gom_bs_multi.cu -- the persistent kernels of the bit-sliced mixing by element
// classes (gom_bs_multi.cuh).
#include "gom_bs_multi.cuh"
#include "gom_kernels.cuh"

namespace {

// One block of eight warps per SM: what the 32-variable class's regions leave of
// its shared memory, and twice the warps for a large element's edges than two
// blocks of four (tree of bound 128, 100x100 torus, p = 1,024: 542 -> 476 us a
// generation).
template <int R, int UB>
__global__ void __launch_bounds__(kMsThreads, 1) k_run_multi(GomParams P, int G, int64_t target)
{
    extern __shared__ __align__(16) uint32_t s_dyn[];
    __shared__ unsigned long long s_cnt[4];
    bs_multi_generations<R, UB>(P, whole_grid(), P.bar, G, target, reinterpret_cast<unsigned long long *>(s_dyn),
                                s_dyn + 64 * P.W, reinterpret_cast<long long *>(s_dyn), s_cnt);
}

} // namespace

const void *gom_run_multi_kernel(int ub) { return ub == 8 ? (const void *)k_run_multi<16, 8> : (const void *)k_run_multi<20, 16>; }

int gom_bs_multi_words(int max_s, int wv, int warps, int edges)
{
    return bs_multi_words(max_s < 32 ? max_s : 32, wv, warps, max_s > 32, edges);
}
