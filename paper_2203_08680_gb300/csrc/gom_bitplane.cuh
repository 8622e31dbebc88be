// gom_bitplane.cuh -- bit-plane arithmetic shared by the bit-sliced mixing
// path and Forced Improvement: one 32-bit register holds one bit of 32
// individuals, so one logic instruction works on 32 trials.  Weighted sums
// of bit-planes by ripple-carry adders (the signed delta of a GOM step in one
// chain per edge), and the per-lane bit-sliced fitness accumulator with its
// flush into the block's fitness accumulators.  Anonymous namespace: each translation
// unit that includes it compiles its own copy.
#pragma once

#include <cuda_runtime.h>

#include "gom_internal.h"

namespace {

constexpr int kFitPlanes = 24;  // bits of the per-lane bit-sliced fitness accumulator
constexpr int kWeightBits = 8;  // |w| < 2^8 in Forced Improvement

// Transposes the NR x NR bit blocks of NR registers inside the lane (NR = 8:
// four blocks, one per byte column; 16: two; 32: one): bit NR c + r of x[a]
// on entry is bit NR c + a of x[r] on return.  log2(NR) steps; step j swaps
// the off-diagonal j x j blocks of each 2j x 2j block.  3 * 4 * 4 = 48
// instructions transpose 8 variables of 32 individuals in each of 32 lanes,
// where shuffle transposes across the warp took 15 for one word of 32
// individuals, used 20 of 32 rows, and kept the shuffle unit busy.
template <int NR, int J = NR / 2>
__device__ __forceinline__ void transpose_lane(uint32_t (&x)[NR])
{
    constexpr uint32_t m = J == 16 ? 0x0000FFFFu : J == 8 ? 0x00FF00FFu : J == 4 ? 0x0F0F0F0Fu : J == 2 ? 0x33333333u
                                                                                                    : 0x55555555u;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        if (r & J) continue;
        const uint32_t a = x[r], b = x[r + J];
        x[r] = (a & m) | ((b << J) & ~m);
        x[r + J] = ((a >> J) & m) | (b & ~m);
    }
    if constexpr (J > 1) transpose_lane<NR, J / 2>(x); // (a loop over J would stay a loop, with x in local memory)
}

// x & (bit t of u ? ~0 : 0), for a per-lane weight u.
__device__ __forceinline__ uint32_t bit_mask(uint32_t x, uint32_t u, int t) { return ((u >> t) & 1u) ? x : 0u; }

// D += u * pos - u * neg over NP bit-planes, two's complement (pos and neg
// disjoint; u < 2^UB).  A lane that subtracts adds the complement of u with a
// carry of one in: its planes are ~u below UB, all ones above (the sign
// extension), and a lane that adds has u below UB, zero above -- so plane t
// is (bit t of u ? pos : neg) below UB and neg above, and one ripple-carry
// chain serves both signs.  The caller keeps every partial sum inside
// [-2^(NP-1), 2^(NP-1)); the carry out of the top plane is dropped.
template <int NP, int UB>
__device__ __forceinline__ void add_signed(uint32_t (&D)[NP], uint32_t pos, uint32_t neg, uint32_t u)
{
    uint32_t carry = neg;
#pragma unroll
    for (int t = 0; t < NP; ++t) {
        const uint32_t in = t < UB ? (((u >> t) & 1u) ? pos : neg) : neg;
        const uint32_t a = D[t];
        D[t] = a ^ in ^ carry;
        carry = (a & in) | (a & carry) | (in & carry);
    }
}

// An edge of the bit-sliced path's lists (GomParams::bdep): x = the far end's
// word offset v W in O (an edge leaving the element) or its row 32 b (inside);
// y = the weight's sign in bit 31, |w| from bit kEdgeWeight on and the near
// end's row 32 a in the bits of kEdgeRowMask.
constexpr int kEdgeRowMask = 127 << 5; // a <= 127
constexpr int kEdgeWeight = 12;        // |w|: bits 12 .. 27

// D += the sum over four edges of |w| pos - |w| neg, as add_signed would: the
// edges in two pairs on UB + 2 planes each, the pairs' sum on UB + 3, and one
// chain over all NP planes; the four carries of one that complements need
// (neg) go into the four chains.  148 logic instructions for UB = 8, NP = 13,
// against 4 x 42 for four chains over all planes.  The logic pipe is the
// busier one: for 8-bit weights one edge of a pair selects by a multiplication
// (torus1000 20.4 -> 19.9 ms a pass, random 12-regular 13.2 -> 12.8; with more
// weight bits the extra instructions cost more, torus317 1.74 -> 1.83).
template <int NP, int UB>
__device__ __forceinline__ void add_signed4(uint32_t (&D)[NP], const uint32_t (&pos)[4], const uint32_t (&neg)[4],
                                            const int2 (&ed)[4])
{
    static_assert(NP >= UB + 3, "accumulator narrower than the sum of four edges");
    uint32_t A[2][UB + 2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t n0 = neg[2 * h], n1 = neg[2 * h + 1];
        uint32_t carry = n0;
#pragma unroll
        for (int t = 0; t < UB + 2; ++t) {
            uint32_t i0 = n0, i1 = n1;
            if (t < UB) {
                if (UB > 8) {
                    i0 = (ed[2 * h].y & (1 << (kEdgeWeight + t))) != 0 ? pos[2 * h] : n0;
                } else { // n0 + m (n0 - pos), m = -1 or 0: the select on the multiplier's pipe
                    const int m = (int)((uint32_t)ed[2 * h].y << (31 - kEdgeWeight - t)) >> 31;
                    i0 = (uint32_t)m * (n0 - pos[2 * h]) + n0;
                }
                i1 = (ed[2 * h + 1].y & (1 << (kEdgeWeight + t))) != 0 ? pos[2 * h + 1] : n1;
            }
            A[h][t] = i0 ^ i1 ^ carry;
            carry = (i0 & i1) | (i0 & carry) | (i1 & carry);
        }
    }
    uint32_t S[UB + 3];
    uint32_t carry = neg[1];
#pragma unroll
    for (int t = 0; t < UB + 3; ++t) {
        const uint32_t a = A[0][t < UB + 2 ? t : UB + 1], b = A[1][t < UB + 2 ? t : UB + 1];
        S[t] = a ^ b ^ carry;
        carry = (a & b) | (a & carry) | (b & carry);
    }
    carry = neg[3];
#pragma unroll
    for (int t = 0; t < NP; ++t) {
        const uint32_t a = D[t], b = S[t < UB + 3 ? t : UB + 2];
        D[t] = a ^ b ^ carry;
        carry = (a & b) | (a & carry) | (b & carry);
    }
}

// The bit-sliced fitness accumulator of a lane: kFitPlanes planes in
// registers, or in shared memory (plane t of the warp's lanes at word 32 t; the
// mixing needs the registers for its tables).
struct FitRegs {
    uint32_t v[kFitPlanes];
    __device__ __forceinline__ uint32_t get(int t) const { return v[t]; }
    __device__ __forceinline__ void set(int t, uint32_t x) { v[t] = x; }
};
struct FitShared {
    uint32_t *v;
    __device__ __forceinline__ uint32_t get(int t) const { return v[32 * t]; }
    __device__ __forceinline__ void set(int t, uint32_t x) { v[32 * t] = x; }
};

// Per-lane state of the bit-sliced path across the groups of a generation.
template <class Fit>
struct BsLane {
    Fit fit;         // accepted deltas of this lane's 32 individuals (word w), bit-sliced
    int w;
    int since_flush; // items added since the last flush (warp-uniform)
    unsigned n_dl, n_acc, n_imp;
};

template <class Fit>
__device__ __forceinline__ void bs_lane_zero(BsLane<Fit> &L, int w)
{
    L.w = w;
#pragma unroll
    for (int t = 0; t < kFitPlanes; ++t) L.fit.set(t, 0);
    L.since_flush = 0;
    L.n_dl = L.n_acc = L.n_imp = 0;
}

// The 32 numbers whose planes x[0 .. kFitPlanes) are, each added into f[b].
__device__ __forceinline__ void planes_add(uint32_t (&x)[32], long long *f)
{
    transpose_lane<32>(x);
#pragma unroll
    for (int b = 0; b < 32; ++b)
        if (x[b]) atomicAdd(reinterpret_cast<unsigned long long *>(&f[b]), (unsigned long long)x[b]);
}

// Adds the lane's accumulated deltas into the block's fitness accumulators
// s_f[32 w + b] (one shared atomic per individual with a non-zero sum) and
// clears them.  In Forced Improvement few individuals have any: bit by bit, and
// nothing for a lane without (a launch per group: 75x75 torus, p = 32, 15
// groups, 185 us a generation with a transpose in every lane, 154 so).
__device__ __forceinline__ void bs_flush(BsLane<FitRegs> &L, long long *s_f)
{
    uint32_t any = 0;
#pragma unroll
    for (int t = 0; t < kFitPlanes; ++t) any |= L.fit.v[t];
    while (any) {
        const int b = __ffs(any) - 1;
        any &= any - 1;
        unsigned v = 0;
#pragma unroll
        for (int t = 0; t < kFitPlanes; ++t) v |= ((L.fit.v[t] >> b) & 1u) << t;
        atomicAdd(reinterpret_cast<unsigned long long *>(&s_f[32 * L.w + b]), (unsigned long long)v);
    }
#pragma unroll
    for (int t = 0; t < kFitPlanes; ++t) L.fit.v[t] = 0;
    L.since_flush = 0;
}

__device__ __noinline__ void bs_flush_shared(uint32_t *v, long long *f)
{
    uint32_t x[32];
#pragma unroll
    for (int t = 0; t < 32; ++t) x[t] = t < kFitPlanes ? v[32 * t] : 0u;
    planes_add(x, f);
#pragma unroll
    for (int t = 0; t < kFitPlanes; ++t) v[32 * t] = 0;
}

__device__ __forceinline__ void bs_flush(BsLane<FitShared> &L, long long *s_f)
{
    bs_flush_shared(L.fit.v, s_f + 32 * L.w);
    L.since_flush = 0;
}

// Adds the accepted deltas (non-negative and below 2^R: planes 0 .. R - 1 of
// D, masked by acc) into the lane's fitness accumulator.
template <int R, class Fit>
__device__ __forceinline__ void fit_add(BsLane<Fit> &L, const uint32_t (&D)[R + 1], uint32_t acc)
{
    uint32_t carry = 0;
#pragma unroll
    for (int t = 0; t < R; ++t) {
        const uint32_t in = D[t] & acc, a = L.fit.get(t);
        L.fit.set(t, a ^ in ^ carry);
        carry = (a & in) | (a & carry) | (in & carry);
    }
#pragma unroll
    for (int t4 = R; t4 < kFitPlanes; t4 += 4) {
        if (!carry) return;
#pragma unroll
        for (int t = t4; t < t4 + 4 && t < kFitPlanes; ++t) {
            const uint32_t a = L.fit.get(t);
            L.fit.set(t, a ^ carry);
            carry &= a;
        }
    }
}

} // namespace
