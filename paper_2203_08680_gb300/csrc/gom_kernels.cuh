// gom_kernels.cuh -- declarations of the kernels in gom_kernels.cu for the
// host code that launches them and builds the per-generation CUDA graph.
#pragma once

#include <cuda_runtime.h>

#include "gom_internal.h"

__global__ void k_init_pop(GomParams P);
__global__ void k_fitness(GomParams P, int64_t *out);
__global__ void k_elite_init(GomParams P);
__global__ void k_begin_call(GomParams P, int64_t target);
__global__ void k_gen_start(GomParams P);
__global__ void k_order(GomParams P);
// The mixing kernel instance for WPI words per warp item (1, 2 or 4) and
// variant (kVarNarrow: 32-bit masks and deltas; kVarWide: 64-bit masks and
// deltas; kVarHuge: 128-bit masks and 64-bit deltas, WPI <= 2, no learned
// filter), with or without the learned filter's bookkeeping; a host-stub
// address usable as a graph-node function, or null for a combination that
// has no instance.
const void *gom_mix_kernel(int wpi, int variant, bool learn);
// The persistent generation kernel k_run<WPI, mask, delta, learn>(GomParams,
// int G, int64_t target), with the same instances (null where none).
const void *gom_run_kernel(int wpi, int variant, bool learn);
// The bit-sliced path (gom_bs.cu): the persistent generation kernel
// k_run_bs<class, R, UB, learn>(GomParams, int G, int64_t target) and the
// per-group mixing kernel k_mix_bs<class, R, UB, learn>(GomParams, int t) for
// elements of at most s <= 32 variables, weights of UB bits and sums of R bits
// (BsPlanes), with or without the learned filter's select phase and
// bookkeeping (8-bit weights only, else null), and the shared-memory words of
// one warp's region.
const void *gom_run_bs_kernel(int s, int r, int ub, bool learn);
const void *gom_mix_bs_kernel(int s, int r, int ub, bool learn);
int gom_bs_warp_words(int s);
// The bit-sliced path by element classes (gom_bs_multi.cu): its persistent
// kernel for elements of at most max_s <= 128 variables and weights of ub = 8
// (sums below 2^16) or 16 bits (2^20), and a block's dynamic shared-memory
// words after the fitness accumulators (edges: the most of an element above 32
// variables).
const void *gom_run_multi_kernel(int ub);
int gom_bs_multi_words(int max_s, int wv, int warps, int edges);
// Packs the dependency lists into the bit-sliced path's edge lists (P.bdep).
__global__ void k_bs_edges(GomParams P, int2 *bdep);
// The instances of one element class (5, 7, 8, 10, 13, 16 or 32 variables at most).
const void *gom_run_bs5(int r, int ub, bool learn);
const void *gom_mix_bs5(int r, int ub, bool learn);
const void *gom_run_bs7(int r, int ub, bool learn);
const void *gom_mix_bs7(int r, int ub, bool learn);
const void *gom_run_bs8(int r, int ub, bool learn);
const void *gom_mix_bs8(int r, int ub, bool learn);
const void *gom_run_bs10(int r, int ub, bool learn);
const void *gom_mix_bs10(int r, int ub, bool learn);
const void *gom_run_bs13(int r, int ub, bool learn);
const void *gom_mix_bs13(int r, int ub, bool learn);
const void *gom_run_bs16(int r, int ub, bool learn);
const void *gom_mix_bs16(int r, int ub, bool learn);
const void *gom_run_bs32(int r, int ub, bool learn);
const void *gom_mix_bs32(int r, int ub, bool learn);
// Forced Improvement on the per-launch path: which = 0 k_fi_elite(GomParams)
// (one block of 1024), 1 k_fi_start(GomParams), 2 k_fi_group<R>(GomParams,
// int t) (256 threads), 3 k_fi_finish(GomParams).
const void *gom_fi_kernel(int which, int r);
// Batched path: instances on block ranges of one cooperative launch.
// k_batch<MINB>(const GomParams *Ps, const GomBatchInst *inst, GomBarrier *bars, int B, int G, int f_words),
// registers cut for MINB (2 or 3) resident blocks of 256 threads.
const void *gom_batch_kernel(int minb);
__global__ void k_batch_collect(const GomParams *Ps, GomBatchInst *inst, int B);
__global__ void k_barrier_selftest(GomBarrier *bar, int *err, int extra, unsigned long long limit_ns);
__global__ void k_gen_end(GomParams P);
// The learned filter's select phase on the graph path: decisions (and with
// `compact` each warp's count of elements to run; 256 threads), the scan of
// the counts over `nwarps` warps (one block of up to 1024 threads), and the
// compacted list (the decision kernel's grid).
__global__ void k_filter_select(GomParams P, int compact);
__global__ void k_filter_scan(GomParams P, int nwarps);
__global__ void k_filter_compact(GomParams P);
__global__ void k_export_pop(GomParams P, uint8_t *out);
__global__ void k_export_small(GomParams P, uint8_t *out);
__global__ void k_export_elite(GomParams P, uint8_t *out);
__global__ void k_import_pop(GomParams P, const uint8_t *in, const uint8_t *elite, int64_t fe, int64_t g);
