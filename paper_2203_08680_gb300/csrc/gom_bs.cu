// gom_bs.cu -- the bit-sliced mixing path's kernels by element class (their
// instances are in gom_bs5.cu to gom_bs32.cu, so that they compile in parallel) and the Forced Improvement kernels of the
// per-generation graph.
#include <climits>
#include <cuda_runtime.h>

#include "gom_bs.cuh"
#include "gom_internal.h"
#include "gom_kernels.cuh"

namespace {

// Forced Improvement on the per-launch path (one CUDA graph per
// generation): the elitist update of its start (one block), the start
// (flags, x_e, the set of individuals in FI), one launch per group, the end.
__global__ void __launch_bounds__(1024) k_fi_elite(GomParams P)
{
    if (P.st->done) return;
    int64_t best;
    int arg;
    block_argmax(P.f, P.p, &best, &arg);
    if (threadIdx.x == 0) {
        const bool newel = best > P.st->fe;
        if (newel) {
            P.st->fe = best;
            P.st->argmax = arg;
            P.st->improved = 1;
        }
        P.st->fi_newel = newel ? 1 : 0;
    }
}

__global__ void k_fi_start(GomParams P)
{
    if (P.st->done) return;
    fi_start(P, whole_grid(), P.st->fi_newel != 0, P.st->argmax >> 5, P.st->argmax & 31, blockIdx.x == 0);
}

template <int R>
__global__ void __launch_bounds__(kMixThreads, 2) k_fi_group(GomParams P, int t)
{
    __shared__ long long s_f[1024];
    __shared__ unsigned long long s_cnt[4];
    __shared__ uint32_t s_act[32];
    if (P.st->done) return;
    if (threadIdx.x < 32) {
        uint32_t done = 0;
        if ((int)threadIdx.x < P.W)
            for (int t2 = 0; t2 < t; ++t2) done |= P.fi.imp[(int64_t)t2 * P.W + threadIdx.x];
        s_act[threadIdx.x] = (int)threadIdx.x < P.W ? P.fi.act0[threadIdx.x] & ~done : 0u;
    }
    acc_zero(P, s_f, s_cnt);
    BsLane<FitRegs> L;
    bs_lane_zero(L, (threadIdx.x & 31) & (P.W - 1));
    unsigned cnt[3] = {0, 0, 0};
    fi_group<R>(P, whole_grid(), t, P.order[t], s_act, L, cnt, s_f);
    bs_flush(L, s_f);
    fi_count_flush(P, cnt);
    acc_flush(P, s_f, s_cnt);
}

__global__ void k_fi_finish(GomParams P)
{
    __shared__ uint32_t s_rep[32];
    if (P.st->done) return;
    if (threadIdx.x < 32) {
        uint32_t done = 0;
        if ((int)threadIdx.x < P.W)
            for (int t2 = 0; t2 < P.k; ++t2) done |= P.fi.imp[(int64_t)t2 * P.W + threadIdx.x];
        s_rep[threadIdx.x] = (int)threadIdx.x < P.W ? P.fi.act0[threadIdx.x] & ~done : 0u;
    }
    __syncthreads();
    fi_finish(P, whole_grid(), s_rep, P.st->fe, blockIdx.x == 0);
}

} // namespace

// One thread per element position: its outside edges, grouped by the near end
// a (segments of P.seg), then its inside edges.
__global__ void k_bs_edges(GomParams P, int2 *bdep)
{
    for (int64_t q = gthread(); q < P.m; q += gthreads()) {
        const int4 h0 = P.hdr[2 * q], h1 = P.hdr[2 * q + 1];
        const int f0 = h0.y, d0 = h0.z, s = h0.w & 0xFF, n_in = h0.w >> 8, n_out = h1.x;
        const auto pack = [](int a, int w) { // |w| < 2^16 where the path is available
            const uint32_t mag = (uint32_t)(w < 0 ? -w : w);
            return (int)((uint32_t)(32 * a) | mag << kEdgeWeight | (w < 0 ? 0x80000000u : 0u));
        };
        for (int a = 0; a < s; ++a)
            for (uint32_t x = P.seg[f0 + q + a]; x < P.seg[f0 + q + a + 1]; ++x) {
                const int2 e = P.dep[d0 + x];
                bdep[d0 + x] = make_int2(e.x * P.W, pack(a, e.y));
            }
        for (int x = n_out; x < n_out + n_in; ++x) {
            const int2 e = P.dep[d0 + x];
            bdep[d0 + x] = make_int2(32 * (e.x >> 8), pack(e.x & 0xFF, e.y));
        }
    }
}

const void *gom_fi_kernel(int which, int r)
{
    switch (which) {
    case 0: return (const void *)k_fi_elite;
    case 1: return (const void *)k_fi_start;
    case 2: return r <= 12 ? (const void *)k_fi_group<12> : (const void *)k_fi_group<16>;
    default: return (const void *)k_fi_finish;
    }
}

const void *gom_run_bs_kernel(int s, int r, int ub, bool learn)
{
    switch (bs_class(s)) {
    case 5: return gom_run_bs5(r, ub, learn);
    case 7: return gom_run_bs7(r, ub, learn);
    case 8: return gom_run_bs8(r, ub, learn);
    case 10: return gom_run_bs10(r, ub, learn);
    case 13: return gom_run_bs13(r, ub, learn);
    case 16: return gom_run_bs16(r, ub, learn);
    default: return gom_run_bs32(r, ub, learn);
    }
}

const void *gom_mix_bs_kernel(int s, int r, int ub, bool learn)
{
    switch (bs_class(s)) {
    case 5: return gom_mix_bs5(r, ub, learn);
    case 7: return gom_mix_bs7(r, ub, learn);
    case 8: return gom_mix_bs8(r, ub, learn);
    case 10: return gom_mix_bs10(r, ub, learn);
    case 13: return gom_mix_bs13(r, ub, learn);
    case 16: return gom_mix_bs16(r, ub, learn);
    default: return gom_mix_bs32(r, ub, learn);
    }
}

int gom_bs_warp_words(int s) { return bs_warp_words(s); }
