// gom_batch_kernels.cuh -- the batched kernel: many independent instances in one
// cooperative launch, each on the per-lane or the bit-sliced phase.  Included
// by one translation unit per register budget, so that they compile in parallel.
#pragma once

#include <climits>
#include <cuda_runtime.h>

#include "gom_bs_multi.cuh"
#include "gom_device.cuh"
#include "gom_internal.h"
#include "gom_kernels.cuh"
#include "gom_lane.cuh"

// One kernel variant of the batched path, compiled as its own function so
// that each variant gets its own register allocation, without Forced Improvement's
// call in the generation loop: batches refuse it, and the registers kept across
// that call made the four instances of 5,000 to 20,000 vertices, p = 128, two
// blocks of eight warps a SM, 5 % slower (1,038 -> 1,006 us a generation).
template <int WPI, typename MaskT, typename AccT>
__device__ __noinline__ void batch_variant(const GomParams &P, const VGrid V, GomBarrier *bar, int G, int64_t target,
                                           const RunShared &S)
{
    run_generations<WPI, MaskT, AccT, false, false>(P, V, bar, G, target, S);
}

// The bit-sliced variant of the batched path: the instance's generations on
// the bit-sliced phase (gom_bs.cuh), its warps' regions of P.bs_words words
// after the fitness accumulators.
template <int SB, int R, int UB>
__device__ __noinline__ void batch_variant_bs(const GomParams &P, const VGrid V, GomBarrier *bar, int G,
                                              int64_t target, const RunShared &S)
{
    const GomParams Q = P; // a private copy: in shared memory every store to it might change a parameter
    bs_generations<SB, R, UB, false, false>(Q, V, bar, G, target, reinterpret_cast<unsigned long long *>(S.dyn),
                             S.dyn, S.f, S.cnt, nullptr);
}

template <int R, int UB>
__device__ __noinline__ void batch_variant_multi(const GomParams &P, const VGrid V, GomBarrier *bar, int G,
                                                 int64_t target, const RunShared &S)
{
    const GomParams Q = P;
    bs_multi_generations<R, UB, false>(Q, V, bar, G, target, reinterpret_cast<unsigned long long *>(S.dyn), S.dyn, S.f,
                                     S.cnt);
}

// Batched path: many independent instances in one cooperative launch.  Each
// instance owns a range of blocks and runs its own generations on them, with
// its own barrier counter and its own stop decision, exactly as its
// persistent kernel would; instances never wait for one another.  Ps[b] is
// instance b's parameter block (one-slice staging), inst[b] its blocks,
// kernel variant, target and generation count (at most G).  The dynamic shared memory holds the block's
// fitness accumulators (f_words 32-bit words, 32 W of the widest instance)
// and then the warps' staging slices.
// MINB: resident blocks of 256 threads the register budget is cut for (2: 128
// registers, the per-lane functions spill 30 to 160 bytes, the bit-sliced ones
// 460 to 940; 3: 80 registers and more warps per SM, 260 to 460 bytes).
template <int MINB>
__global__ void __launch_bounds__(kMixThreads, MINB)
    k_batch(const GomParams *Ps, const GomBatchInst *inst, GomBarrier *bars, int B, int G, int f_words)
{
    extern __shared__ __align__(16) uint32_t s_dyn[];
    __shared__ GomParams sP;
    __shared__ unsigned long long s_cnt[4];
    __shared__ int s_b;
    if (threadIdx.x == 0) {
        // the instance of this block: the last b with blk0 <= blockIdx.x
        int lo = 0, hi = B - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (inst[mid].blk0 <= (int)blockIdx.x)
                lo = mid;
            else
                hi = mid - 1;
        }
        s_b = lo;
        sP = Ps[lo];
    }
    __syncthreads();
    const int b = s_b;
    const GomBatchInst I = inst[b];
    if ((int)blockIdx.x >= I.blk0 + I.nblk) return; // a block past every range (none by construction)
    const VGrid V{(int)blockIdx.x - I.blk0, I.nblk};
    const RunShared S{s_dyn + f_words, reinterpret_cast<long long *>(s_dyn), s_cnt, nullptr, nullptr};
    GomBarrier *bar = bars + b;
    G = min(G, I.gens);
    if (MINB == 2 && I.variant == kVarBits) { // the bit-sliced phase needs the larger register budget
        if constexpr (MINB == 2) {
            // fewer instances than the single-instance kernels have, the next wider planes for the rest
            const int cls = bs_class(sP.bs_S);
            if (I.bs_ub == 8)
                cls == 5    ? batch_variant_bs<5, 16, 8>(sP, V, bar, G, I.target, S)
                : cls == 7  ? batch_variant_bs<7, 16, 8>(sP, V, bar, G, I.target, S)
                : cls == 8  ? batch_variant_bs<8, 16, 8>(sP, V, bar, G, I.target, S)
                : cls == 10 ? batch_variant_bs<10, 16, 8>(sP, V, bar, G, I.target, S)
                : cls == 13 ? batch_variant_bs<13, 16, 8>(sP, V, bar, G, I.target, S)
                : cls == 16 ? batch_variant_bs<16, 16, 8>(sP, V, bar, G, I.target, S)
                            : batch_variant_bs<32, 16, 8>(sP, V, bar, G, I.target, S);
            else
                cls == 8    ? batch_variant_bs<8, 20, 16>(sP, V, bar, G, I.target, S)
                : cls == 16 ? batch_variant_bs<16, 20, 16>(sP, V, bar, G, I.target, S)
                            : batch_variant_bs<32, 20, 16>(sP, V, bar, G, I.target, S);
        }
    } else if (MINB == 2 && I.variant == kVarMulti) {
        if constexpr (MINB == 2) {
            if (I.bs_ub == 8)
                batch_variant_multi<16, 8>(sP, V, bar, G, I.target, S);
            else
                batch_variant_multi<20, 16>(sP, V, bar, G, I.target, S);
        }
    } else if (I.variant == kVarNarrow || I.variant == kVarBits) {
        if (I.wpi == 4)
            batch_variant<4, uint32_t, int32_t>(sP, V, bar, G, I.target, S);
        else if (I.wpi == 2)
            batch_variant<2, uint32_t, int32_t>(sP, V, bar, G, I.target, S);
        else
            batch_variant<1, uint32_t, int32_t>(sP, V, bar, G, I.target, S);
    } else if (I.variant == kVarHuge) {
        if (I.wpi == 2)
            batch_variant<2, Mask128, long long>(sP, V, bar, G, I.target, S);
        else
            batch_variant<1, Mask128, long long>(sP, V, bar, G, I.target, S);
    } else {
        if (I.wpi == 4)
            batch_variant<4, uint64_t, long long>(sP, V, bar, G, I.target, S);
        else if (I.wpi == 2)
            batch_variant<2, uint64_t, long long>(sP, V, bar, G, I.target, S);
        else
            batch_variant<1, uint64_t, long long>(sP, V, bar, G, I.target, S);
    }
}
