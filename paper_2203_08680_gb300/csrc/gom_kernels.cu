// gom_kernels.cu -- sm_103a kernels of parallel GOM for weighted Max-Cut.
//
// Population layout (bit-sliced, variable-major): O[v*W + w] holds variable v
// of individuals 32w .. 32w+31, one bit each.  W is a power of two; words and
// bits past the population size stay zero.  A warp therefore reads one
// variable of 32 individuals with a single broadcast load, and the writes of
// one GOM trial batch (32 individuals x one element) are whole words.
//
// Kernels of one generation (Alg. 3):
//   gen start  Clone (P <- O), copy of the new elitist, elitist flags
//   order      random order of the colour groups
//   mix        one phase per colour group: every (individual, element) trial
//              of the group -- donor, partial evaluation, accept, write
//   gen end    elitist update, counters, target check
// Two ways to run them: one kernel per phase in a per-generation CUDA graph
// (k_gen_start, k_order, k_mix, k_gen_end), or one persistent cooperative
// kernel (k_run) that runs many generations with grid barriers between the
// phases.  Plus initialisation, full evaluation and import/export kernels.
#include <climits>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "gom_device.cuh"
#include "gom_fi.cuh"
#include "gom_filter_dev.cuh"
#include "gom_internal.h"
#include "gom_kernels.cuh"
#include "gom_lane.cuh"
#include "gom_rows.cuh"


// ----------------------------------------------------------------------------
// InitializePopulation (Alg. 3): one Philox call gives 128 variables of one
// individual; a warp covers 32 individuals and turns each variable into one
// word with a ballot.
__global__ void k_init_pop(GomParams P)
{
    const int lane = threadIdx.x & 31;
    const int64_t warp = gthread() >> 5, nwarps = gthreads() >> 5;
    const int64_t nq = (P.n + 127) / 128;
    const int64_t items = nq * P.W;
    const uint32_t k0 = (uint32_t)P.seed, k1 = (uint32_t)(P.seed >> 32);
    for (int64_t it = warp; it < items; it += nwarps) {
        const int64_t q = it / P.W;
        const int w = (int)(it - q * P.W);
        const int i = 32 * w + lane;
        const bool valid = i < P.p;
        const uint4 r = philox10(make_uint4((uint32_t)q, (uint32_t)i, 0u, kTagInit), k0, k1);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const uint32_t word = pick(r, t);
            uint32_t mine = 0;
#pragma unroll
            for (int b = 0; b < 32; ++b) {
                const uint32_t mk = __ballot_sync(kFull, valid && ((word >> b) & 1u));
                if (lane == b) mine = mk;
            }
            const int64_t v = 128 * q + 32 * t + lane;
            if (v < P.n) P.O[v * P.W + w] = mine;
        }
    }
}

// Full evaluation (Sec. 6.2) of the population, added into out[p].
__global__ void __launch_bounds__(256, 2) k_fitness(GomParams P, int64_t *out)
{
    __shared__ long long s_f[1024], s_const;
    cut_sums(P.O, P.n, P.p, P.W, P.row_ptr, P.col, P.wgt, s_f, &s_const, out);
}

// Elitist of a fresh population: lowest index of maximal fitness.
__global__ void k_elite_init(GomParams P)
{
    int64_t best;
    int arg;
    block_argmax(P.f, P.p, &best, &arg);
    if (threadIdx.x == 0) {
        P.st->fe = best;
        P.st->best = best;
        P.st->argmax = arg;
        P.st->improved = 1;
        P.st->done = 0;
    }
    for (int w = threadIdx.x; w < 2 * P.W; w += blockDim.x) P.eqw[w] = kFull;
}

__global__ void k_begin_call(GomParams P, int64_t target)
{
    P.st->done = 0;
    P.st->target = target;
    P.st->call_g0 = P.st->g; // first generation of this call
}


// ----------------------------------------------------------------------------
// Kernels of the per-launch path (one CUDA graph per generation).

__global__ void k_gen_start(GomParams P)
{
    if (P.st->done) return;
    phase_gen_start(P, whole_grid(), P.st->improved, P.st->argmax, P.st->g, true);
}

__global__ void k_order(GomParams P)
{
    extern __shared__ unsigned long long s_key[];
    if (P.st->done) return;
    phase_order(P, whole_grid(), s_key, P.st->g);
}

template <int WPI, typename MaskT, typename AccT, bool LEARN>
__global__ void __launch_bounds__(kMixThreads, 3) k_mix(GomParams P, int t)
{
    extern __shared__ __align__(16) uint32_t s_dyn[];
    __shared__ long long s_f[1024];
    __shared__ unsigned long long s_cnt[4];
    if (P.st->done) return;
    acc_zero(P, s_f, s_cnt);
    unsigned n_dl = 0, n_acc = 0, n_imp = 0;
    if (sizeof(MaskT) == 16 && P.blk)
        phase_mix_block<WPI, MaskT, AccT>(P, whole_grid(), t, P.order[t], P.st->g, s_dyn, false, s_f, n_dl, n_acc,
                                          n_imp);
    else
        phase_mix<WPI, MaskT, AccT, LEARN>(P, whole_grid(), t, P.order[t], P.st->g,
                                    s_dyn + (threadIdx.x >> 5) * warp_words(P, false), false, false, s_f, n_dl, n_acc,
                                    n_imp);
    count_flush(s_cnt, n_dl, n_acc, n_imp);
    acc_flush(P, s_f, s_cnt);
}

// The learned filter's select phase on the per-generation graph path: the
// decisions (with `compact`, each warp's count of elements to run), the scan
// of the counts (one block) and the compacted list, each a node of its own,
// launched on the same grid for the first and the last.
__global__ void __launch_bounds__(256) k_filter_select(GomParams P, int compact)
{
    if (P.st->done) return;
    filter_select_decide(P, whole_grid(), P.st->g, compact != 0);
}

__global__ void __launch_bounds__(1024) k_filter_scan(GomParams P, int nwarps)
{
    if (P.st->done) return;
    filter_select_scan(P, nwarps);
}

__global__ void __launch_bounds__(256) k_filter_compact(GomParams P)
{
    if (P.st->done) return;
    filter_select_compact(P, whole_grid());
}

__global__ void __launch_bounds__(1024) k_gen_end(GomParams P)
{
    if (P.st->done) return;
    GenEnd e{P.st->fe, 0, P.st->argmax};
    phase_gen_end(P, P.st->target, P.st->g, e, true);
}

template <int WPI, typename MaskT, typename AccT, bool LEARN>
__global__ void __launch_bounds__(kRunThreads, 1) k_run(GomParams P, int G, int64_t target)
{
    extern __shared__ __align__(16) uint32_t s_dyn[];
    __shared__ long long s_f[1024];
    __shared__ unsigned long long s_cnt[4];
    __shared__ unsigned long long s_okey[kStageAllMaxK];
    __shared__ int s_order[kStageAllMaxK];
    const RunShared S{s_dyn, s_f, s_cnt, s_okey, s_order};
    run_generations<WPI, MaskT, AccT, LEARN>(P, whole_grid(), P.bar, G, target, S);
}

// Self-test of the grid barrier's bounded wait: `blocks` co-resident blocks
// meet at a barrier that expects `blocks + extra` arrivals; with extra > 0 no
// block is ever released and every block must give up after limit_ns.
__global__ void k_barrier_selftest(GomBarrier *bar, int *err, int extra, unsigned long long limit_ns)
{
    const unsigned expected = gridDim.x + (unsigned)extra;
    unsigned long long next = 0;
    if (threadIdx.x == 0) next = barrier_first(&bar->count, expected);
    grid_barrier(&bar->count, err, expected, next, limit_ns);
}

template <bool LEARN>
const void *mix_kernel(int wpi, int variant)
{
    if (variant == kVarNarrow)
        return wpi == 4 ? (const void *)k_mix<4, uint32_t, int32_t, LEARN>
             : wpi == 2 ? (const void *)k_mix<2, uint32_t, int32_t, LEARN>
                        : (const void *)k_mix<1, uint32_t, int32_t, LEARN>;
    if (variant == kVarHuge) // no filter instances, at most two words per item
        return LEARN || wpi > 2 ? nullptr
             : wpi == 2         ? (const void *)k_mix<2, Mask128, long long, false>
                                : (const void *)k_mix<1, Mask128, long long, false>;
    return wpi == 4 ? (const void *)k_mix<4, uint64_t, long long, LEARN>
         : wpi == 2 ? (const void *)k_mix<2, uint64_t, long long, LEARN>
                    : (const void *)k_mix<1, uint64_t, long long, LEARN>;
}

template <bool LEARN>
const void *run_kernel(int wpi, int variant)
{
    if (variant == kVarNarrow)
        return wpi == 4 ? (const void *)k_run<4, uint32_t, int32_t, LEARN>
             : wpi == 2 ? (const void *)k_run<2, uint32_t, int32_t, LEARN>
                        : (const void *)k_run<1, uint32_t, int32_t, LEARN>;
    if (variant == kVarHuge)
        return LEARN || wpi > 2 ? nullptr
             : wpi == 2         ? (const void *)k_run<2, Mask128, long long, false>
                                : (const void *)k_run<1, Mask128, long long, false>;
    return wpi == 4 ? (const void *)k_run<4, uint64_t, long long, LEARN>
         : wpi == 2 ? (const void *)k_run<2, uint64_t, long long, LEARN>
                    : (const void *)k_run<1, uint64_t, long long, LEARN>;
}

const void *gom_mix_kernel(int wpi, int variant, bool learn)
{
    return learn ? mix_kernel<true>(wpi, variant) : mix_kernel<false>(wpi, variant);
}

const void *gom_run_kernel(int wpi, int variant, bool learn)
{
    return learn ? run_kernel<true>(wpi, variant) : run_kernel<false>(wpi, variant);
}

// ----------------------------------------------------------------------------
// uint8 rows out[i*n + v] of the population.
__global__ void __launch_bounds__(kRowThreads) k_export_pop(GomParams P, uint8_t *out)
{
    __shared__ __align__(16) uint32_t sm[row_words(32)];
    unpack_rows(P.O, P.n, P.p, P.W, out, sm);
}

// The same, one byte a thread, for small populations (export_small).
__global__ void k_export_small(GomParams P, uint8_t *out)
{
    const int64_t total = (int64_t)P.p * P.n;
    for (int64_t idx = gthread(); idx < total; idx += gthreads()) {
        const int64_t i = idx / P.n, v = idx - i * P.n;
        out[idx] = (uint8_t)((P.O[v * P.W + (i >> 5)] >> (i & 31)) & 1u);
    }
}

__global__ void k_export_elite(GomParams P, uint8_t *out)
{
    const int improved = P.st->improved;
    const int aw = P.st->argmax >> 5, ab = P.st->argmax & 31;
    for (int64_t v = gthread(); v < P.n; v += gthreads())
        out[v] = improved ? (uint8_t)((P.O[v * P.W + aw] >> ab) & 1u) : P.xe[v];
}

// Packs uint8 rows in[i*n + v] into the bit-sliced O, copies the elitist, and
// sets the state of an import: the given elitist fitness and generation
// counter, the fitness array zeroed for the evaluation that follows.
__global__ void __launch_bounds__(kRowThreads, 4) k_import_pop(GomParams P, const uint8_t *in, const uint8_t *elite,
                                                            int64_t fe, int64_t g)
{
    __shared__ __align__(16) uint32_t sm[row_words(32)];
    pack_rows(in, P.n, P.p, P.W, P.O, sm);
    for (int64_t v = gthread(); v < P.n; v += gthreads()) P.xe[v] = elite[v] ? 1 : 0;
    if (blockIdx.x > 0) return;
    if (threadIdx.x == 0) {
        P.st->fe = fe;
        P.st->best = fe;
        P.st->argmax = 0;
        P.st->improved = 0;
        P.st->done = 0;
        P.st->g = (uint32_t)g;
        P.st->cnt[0] = P.st->cnt[1] = P.st->cnt[2] = P.st->cnt[3] = 0;
    }
    for (int w = threadIdx.x; w < 2 * P.W; w += blockDim.x) P.eqw[w] = kFull;
    for (int i = threadIdx.x; i < 32 * P.W; i += blockDim.x) P.f[i] = 0;
}
