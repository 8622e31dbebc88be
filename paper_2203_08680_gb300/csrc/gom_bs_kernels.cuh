// gom_bs_kernels.cuh -- the kernels of the bit-sliced mixing path (gom_bs.cuh):
// the persistent generation kernel and the per-group mixing kernel of the
// per-generation graph, with the selection of their instances.  Included by
// one translation unit per element class.
#pragma once

#include <cuda_runtime.h>

#include "gom_bs.cuh"
#include "gom_internal.h"

namespace {

// Persistent path on the bit-sliced phase: up to G generations in one
// cooperative launch (bs_generations on the whole grid).  The dynamic shared
// memory holds the block's fitness accumulators, then the warps' regions (the
// k group keys of the order phase overlay them).
template <int SB, int R, int UB, bool LEARN>
__global__ void __launch_bounds__(kBsThreads, bs_blocks(SB)) k_run_bs(GomParams P, int G, int64_t target)
{
    extern __shared__ __align__(16) uint32_t s_dyn[];
    __shared__ unsigned long long s_cnt[4], s_fc[4];
    bs_generations<SB, R, UB, LEARN>(P, whole_grid(), P.bar, G, target, reinterpret_cast<unsigned long long *>(s_dyn),
                             s_dyn + 64 * P.W, reinterpret_cast<long long *>(s_dyn), s_cnt, s_fc);
}

// Per-launch path: the mixing of the group at position t (one launch per
// group in the per-generation CUDA graph).
template <int SB, int R, int UB, bool LEARN>
__global__ void __launch_bounds__(kBsThreads, bs_blocks(SB)) k_mix_bs(GomParams P, int t)
{
    extern __shared__ __align__(16) uint32_t s_dyn[];
    __shared__ unsigned long long s_cnt[4], s_fc[4];
    long long *s_f = reinterpret_cast<long long *>(s_dyn);
    if (P.st->done) return;
    fc_zero(s_fc);
    acc_zero(P, s_f, s_cnt);
    const BsMap M = bs_map<LEARN>(P, whole_grid(), s_dyn + 64 * P.W, P.bs_words);
    BsLane<FitShared> L;
    L.fit.v = bs_fit(P, s_dyn + 64 * P.W);
    bs_lane_zero(L, M.w);
    phase_mix_bs<SB, R, UB, LEARN>(P, M, t, P.order[t], P.st->g, [] { return true; }, L, s_f, s_fc);
    bs_finish_generation(P, L, s_f, s_cnt);
    acc_flush(P, s_f, s_cnt);
    if (LEARN) fc_flush(P, s_fc);
}

// The instance for R-bit sums of UB-bit weights (the learned filter's exist
// for 8-bit weights only), or null.
template <int SB>
const void *run_bs_kernel(int r, int ub, bool learn)
{
    if (learn)
        return ub != 8 ? nullptr : r == 12 ? (const void *)k_run_bs<SB, 12, 8, true> : (const void *)k_run_bs<SB, 16, 8, true>;
    return r == 12 ? (const void *)k_run_bs<SB, 12, 8, false>
         : ub == 8 ? (const void *)k_run_bs<SB, 16, 8, false>
         : r == 16 ? (const void *)k_run_bs<SB, 16, 12, false>
                   : (const void *)k_run_bs<SB, 20, 16, false>;
}

template <int SB>
const void *mix_bs_kernel(int r, int ub, bool learn)
{
    if (learn)
        return ub != 8 ? nullptr : r == 12 ? (const void *)k_mix_bs<SB, 12, 8, true> : (const void *)k_mix_bs<SB, 16, 8, true>;
    return r == 12 ? (const void *)k_mix_bs<SB, 12, 8, false>
         : ub == 8 ? (const void *)k_mix_bs<SB, 16, 8, false>
         : r == 16 ? (const void *)k_mix_bs<SB, 16, 12, false>
                   : (const void *)k_mix_bs<SB, 20, 16, false>;
}

} // namespace
