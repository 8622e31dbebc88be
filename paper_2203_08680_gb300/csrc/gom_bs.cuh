// gom_bs.cuh -- the bit-sliced mixing path of parallel GOM for weighted Max-Cut:
// its device code, shared by its own kernels (gom_bs_kernels.cuh), those by
// element class (gom_bs_multi.cuh) and the batched kernel
// (gom_batch_kernels.cuh).  Anonymous namespace: each translation unit that
// includes it compiles its own copy.
//
// Same generations as the per-lane path of gom_lane.cuh (Alg. 3; every
// trial of Alg. 2 decided by the exact integer delta), with the partial
// evaluation, the acceptance and the fitness bookkeeping done on bit-planes:
// one 32-bit register holds one bit of 32 individuals, so one logic
// instruction works on 32 trials at once.
//
// A tile takes an item of E elements of the colour group.  A pair is one word
// (32 individuals) of one element; an element has Wv pairs.  Normally a tile
// is a warp, a lane owns one pair and E = 32 / Wv.  Where a colour group is too
// small to give every resident warp an item, 2 to 32 lanes share a pair (they
// repeat phase 0 and split the donor draws and the element's edges), and an
// element whose lanes pass one warp takes 2 or 4 warps of a block (BsMap).
// Per item:
//   phase 0  (lane = pair) the generation-start rows of P on F_j; the run
//            starts of P's patterns (bit d: pattern d differs from pattern
//            d - 1, cyclically); then, by a bit transpose inside the lane, the
//            pattern P_d of each of its 32 individuals, and by one backward
//            walk over them the pattern N_d of the next run start after d: one
//            table entry (P_d, N_d) per individual
//   phase 1  (lane = 4 individuals of a pair) the donor search of Sec. 4.2: one
//            Philox call gives 4 starts; one table entry per trial holds the
//            start's pattern and the pattern the search falls through to when
//            the start equals the parent.  So far everything comes from P: this
//            is bs_prepare, the rest bs_item.  (Lane = pair) the 32 entries come
//            back through the inverse transpose as bit-planes T1_a (the
//            starts' bits) and T2_a (the fall-through's), and the flip planes
//            F_a (bit b: individual b flips variable a) are a plane select;
//            the rare individuals whose own column is the run start the
//            search falls through to are resolved one by one
//   phase 2  (lane = pair) the partial evaluation (Sec. 2.2, Alg. 4) as
//            bit-plane arithmetic: an edge e that a trial toggles (t_e = F_a
//            for an edge leaving F_j, F_a ^ F_b inside) changes the cut by
//            +|w_e| if it was uncut and -|w_e| if it was cut (its cut plane
//            c_e taken with the weight's sign folded in), so
//              delta = sum_e |w_e| (t_e & ~c_e) - |w_e| (t_e & c_e),
//            four edges at a time in signed ripple-carry chains on as many
//            two's-complement planes as their partial sums need, R + 1 for the
//            total (each edge counted once); then the accept plane (Alg. 2:
//            delta > 0, or delta = 0 and not the elitist), counters by
//            popcount, the accepted flips XORed into the rows, and the
//            accepted deltas into a bit-sliced per-lane fitness accumulator,
//            flushed into the block's accumulators once per generation (or
//            before it could overflow).
// With the learned trial filter on, a select phase after the generation start
// (gom_filter_dev.cuh) decides which elements run and lists them in order, the
// groups run only the listed elements, and each item records its elements'
// history and training samples.
// What bounds it: instruction issue and the integer ALU.  Donor tables made and
// read inside the lane took a generation of the 1000x1000 torus (p = 256) from
// 2.27 to 1.31 ms against tables of packed patterns transposed across the warp
// with a run-start search per trial; one flat edge list per element and chains
// over four edges took it to 1.10 ms, instances with the rows known at compile
// time and selects shared with the multiply pipe to 0.98 ms (103 warp
// instructions per 32 trials, the ALU pipe busy 65 % of the cycles).
//
// Elements of one colour group share no variable and no edge (LMIG
// colouring), so the rows a pair reads and writes belong to it alone during
// the group.
//
// The path takes elements of at most 32 variables, |w| < 2^UB, and elements
// whose sum of |w| over their edges is below 2^R, the width of the bit-plane
// accumulators: (R, UB) = (12, 8), (16, 8), (16, 12) or (20, 16); the host
// selects it only then.  (The last two took a generation of the 317x317 torus
// with weights in [-1000, 1000], p = 100, from 700 us per lane to 182 us.)
#pragma once

#include <climits>
#include <cuda_runtime.h>

#include "gom_bitplane.cuh"
#include "gom_device.cuh"
#include "gom_fi.cuh"
#include "gom_filter_dev.cuh"
#include "gom_internal.h"

namespace {

// Brings the 128-byte line holding *ptr into L2 (a hint: no data returned).
__device__ __forceinline__ void prefetch_l2(const void *ptr)
{
    asm volatile("prefetch.global.L2 [%0];" ::"l"(ptr));
}

// First position at or after x, in cyclic order over [0, p), whose bit is set
// in the run starts rs[0..Wv); nz has bit w set iff rs[w] != 0 (so the next
// non-empty word is one bit scan away).  -1 if no bit is set.
__device__ __forceinline__ int next_run_start(const uint32_t *rs, uint32_t nz, int x)
{
    const int w = x >> 5;
    const uint32_t m = rs[w] & (0xFFFFFFFFu << (x & 31));
    if (m) return 32 * w + __ffs(m) - 1;
    const uint32_t later = nz & ~((2u << w) - 1u); // words after w
    const uint32_t any = later ? later : nz;        // else wrap round (word w's low bits included)
    if (!any) return -1;
    const int w2 = __ffs(any) - 1;
    return 32 * w2 + __ffs(rs[w2]) - 1;
}

// The kernels' element classes: instances for elements of at most SB = 5, 7, 8,
// 10, 13, 16 or 32 variables.  Up to 13 the rows are known at compile time (the
// neighbourhoods of degree 4, 6 and 7, 8 and 9, 12): a generation of torus1000,
// p = 256, takes 9 % less in the class of 5 than in that of 8, one of random
// 12-regular graphs 5 % less in the class of 13 than in that of 16.
__host__ __device__ constexpr int bs_class(int S)
{
    return S <= 5 ? 5 : S <= 7 ? 7 : S <= 8 ? 8 : S <= 10 ? 10 : S <= 13 ? 13 : S <= 16 ? 16 : 32;
}

// Rows of a class's shared arrays: the class's in the small ones, else those of
// the model's largest element.
__host__ __device__ constexpr int bs_rows(int S) { return S <= 13 ? bs_class(S) : S; }

// Variables of a pattern in the class's tables: entries of 2 bytes (P_d in the
// low byte, N_d in the high one), 4 bytes (halves) or 8 bytes (P_d, N_d) for
// 8, 16 or 32; a pair's 32 entries take twice as many words.
__host__ __device__ constexpr int bs_table(int S) { return S <= 8 ? 8 : S <= 16 ? 16 : 32; }
__host__ __device__ constexpr int bs_entry_words(int S) { return 2 * bs_table(S); }

// Shared-memory words of one warp's region (a tile of several warps uses its
// first warp's): the donor tables [32 pairs], the trials' entries [32 pairs]
// (their slots reused for the flip planes [S][32 pairs]), the rows of O on F_j
// [S][32 pairs], per pair the run starts, the patterns of the word's last
// individual and of its first run start, and the warp's fitness planes
// [kFitPlanes][32 lanes] (every warp of a tile its own).  Row arrays are
// variable-major: pair slot l reads word 32 a + l, free of bank conflicts for
// any a.
__host__ __device__ __forceinline__ int bs_warp_words(int S)
{
    return 64 * bs_entry_words(S) + 32 * bs_rows(S) + 96 + 32 * kFitPlanes;
}

// Blocks per SM the kernels' registers are cut for, by element class: what the
// regions leave of an SM's shared memory (34, 54 and 90 KB a block).  Measured
// for 8-bit weights (torus1000: 5 blocks of 96 registers 25.5 ms a pass, 6 of 80
// 25.1); the 20-bit sums of 5 to 8 variables spill about 210 bytes at 80.
constexpr int bs_blocks(int SB) { return SB <= 8 ? 6 : SB <= 16 ? 4 : 2; }

// This lane's fitness planes; `regions` is the block's first warp region.
__device__ __forceinline__ uint32_t *bs_fit(const GomParams &P, uint32_t *regions)
{
    return regions + ((threadIdx.x >> 5) + 1) * P.bs_words - 32 * kFitPlanes + (threadIdx.x & 31);
}

// This thread's place in its tile: lanes 2^lsh per pair, nwi warps per tile
// (more than one only for E = 1), the pair's slot, its element slot e and word
// w, `sub` the lane's number within the pair; in: the slot holds a pair of the
// tile's E elements.
struct BsMap {
    int lsh, nwi, E;
    int tile, ntiles; // of the (virtual) grid: consecutive tiles go to different blocks
    int slot, e, w, sub;
    bool in;
    uint32_t *sm;     // the tile's shared region
};

// The tile's map; `regions` is the block's first warp region, `words` a region's size.
template <bool LEARN>
__device__ __forceinline__ BsMap bs_map(const GomParams &P, const VGrid &V, uint32_t *regions, int words)
{
    BsMap M;
    const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
    M.lsh = LEARN ? 0 : P.bs_lsh; // the learned filter's bookkeeping takes one lane per pair
    M.nwi = LEARN ? 1 : P.bs_nwi;
    M.E = M.nwi > 1 ? 1 : (32 >> M.lsh) / P.Wv;
    const int tb = wib / M.nwi, tw = wib - tb * M.nwi;
    M.tile = tb * V.nblk + V.blk;
    M.ntiles = (int)(blockDim.x >> 5) / M.nwi * V.nblk;
    M.slot = (32 * tw + lane) >> M.lsh;
    M.e = M.slot / P.Wv;
    M.w = M.slot - M.e * P.Wv;
    M.sub = lane & ((1 << M.lsh) - 1);
    M.in = M.e < M.E;
    M.sm = regions + tb * M.nwi * words;
    return M;
}

// Waits for the tile's threads (every thread of the tile calls it): a warp, a
// whole block, or some of its warps on a named barrier.  The barrier numbers
// are constants: a number in a register makes the compiler reserve all 16 of a
// block, and an SM's 64 then hold four blocks.
__device__ __forceinline__ void tile_sync(const BsMap &M)
{
    const int n = 32 * M.nwi;
    if (M.nwi == 1) {
        __syncwarp();
    } else if (n == (int)blockDim.x) {
        __syncthreads();
    } else {
        switch ((int)(threadIdx.x >> 5) / M.nwi) { // at most four tiles of several warps in a block of eight
        case 0: asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory"); break;
        case 1: asm volatile("bar.sync 2, %0;" ::"r"(n) : "memory"); break;
        case 2: asm volatile("bar.sync 3, %0;" ::"r"(n) : "memory"); break;
        default: asm volatile("bar.sync 4, %0;" ::"r"(n) : "memory"); break;
        }
    }
}

// Learned filter bookkeeping after a bit-sliced item (warp-wide): each
// element's accepted, donor-less and improving trials (summed over its W
// lanes) into this generation's history, the block's item counters s_fc (run,
// useful, audited, audited and useful; one item per element on this path),
// and for the elements the sampling hash picks a training sample -- the
// features as the select phase saw them, label: the element was useful (an
// accepted trial, or with P.flt.label an improving one).
__device__ __noinline__ void bs_record(const GomParams &P, int q, bool ke, bool audited, uint32_t g, unsigned acc,
                                       unsigned dl, unsigned imp, unsigned long long *s_fc)
{
    const int lane = threadIdx.x & 31;
    const int Wv = P.Wv, E = 32 / Wv, first = lane - lane % Wv; // the element's first lane (one lane per pair here)
    unsigned ad = acc | dl << 16, sum_ad = 0, sum_imp = 0; // at most 1,024 each
    for (int x = 0; x < Wv; ++x) {
        sum_ad += __shfl_sync(kFull, ad, first + x);
        sum_imp += __shfl_sync(kFull, imp, first + x);
    }
    acc = sum_ad & 0xFFFFu;
    dl = sum_ad >> 16;
    imp = sum_imp;
    const bool useful = P.flt.label ? imp != 0 : acc != 0;
    if (ke && lane == first) {
        uint32_t *cur = P.flt.hist + (size_t)(g & 1) * 3 * (size_t)P.m;
        cur[q] = acc;
        cur[P.m + q] = dl;
        cur[2 * (size_t)P.m + q] = imp;
        atomicAdd(&s_fc[0], 1ull);
        if (useful) atomicAdd(&s_fc[1], 1ull);
        if (audited) atomicAdd(&s_fc[2], 1ull);
        if (audited && useful) atomicAdd(&s_fc[3], 1ull);
    }
    for (int e2 = 0; e2 < E; ++e2) {
        const int src = e2 * Wv;
        const int q2 = __shfl_sync(kFull, q, src);
        const bool ok = __shfl_sync(kFull, ke ? 1 : 0, src) != 0;
        const bool u2 = __shfl_sync(kFull, useful ? 1 : 0, src) != 0;
        if (ok && filter_sample(q2, g)) {
            float x[kFilterIn];
            filter_features(P, q2, g, x);
            filter_log_sample(P, x, u2);
        }
    }
    __syncwarp();
}

// Individual i of element j (its pairs from b2 on in the table), possibly the
// run start its own search falls through to: its start is drawn again, and if
// the next run start after it is not i, the result is false.  Otherwise the
// search goes on behind i, and *fl receives the donor's flips: the donor is
// i + 1 if its pattern differs from the parent's (xf, the pattern of the run
// before i, which holds the start), else the first run start after i + 1 --
// unless the element has no more than two run starts: then the run of i + 1
// reaches round to i, everyone but i equals the parent, and there is no donor.
template <int SB>
__device__ __noinline__ bool self_hit(uint32_t *fl, const uint32_t *tab, const uint32_t *rs, uint32_t nz, int b2, int j,
                                      int i, uint32_t g, int p, uint64_t seed)
{
    const uint4 r4 = philox10(make_uint4((uint32_t)j, (uint32_t)(i >> 2), g, kTagDonor), (uint32_t)seed,
                              (uint32_t)(seed >> 32));
    const uint32_t d = (uint32_t)(i + 1) + __umulhi(pick(r4, i & 3), (uint32_t)(p - 1));
    const int st = (int)min(d, d - (uint32_t)p);
    if (next_run_start(rs, nz, st + 1 == p ? 0 : st + 1) != i) return false;
    const auto entry = [&](int x, uint32_t *next) -> uint32_t {
        if constexpr (bs_table(SB) == 8) {
            const uint32_t en = reinterpret_cast<const uint16_t *>(tab)[32 * b2 + x];
            *next = en >> 8;
            return en & 0xFFu;
        } else {
            const int k3 = b2 + (x >> 5), at = 32 * k3 + ((x + k3) & 31);
            *next = bs_table(SB) == 16 ? tab[at] >> 16 : tab[1024 + at];
            return bs_table(SB) == 16 ? tab[at] & 0xFFFFu : tab[at];
        }
    };
    uint32_t unused, nn;
    const uint32_t xf = entry(i == 0 ? p - 1 : i - 1, &unused), pn = entry(i + 1 == p ? 0 : i + 1, &nn);
    int starts = 0;
    for (uint32_t m = nz; m; m &= m - 1) starts += __popc(rs[__ffs(m) - 1]);
    *fl = pn != xf ? pn ^ xf : starts == 2 ? 0u : nn ^ xf;
    return true;
}

// An item between its two parts: the lane's element and what the first part
// found in the generation-start population.
struct BsItem {
    int q, j, s, f0, d0, n_out, n_in;
    bool ke, audited;   // the lane's pair exists; the element runs as an audit of the learned filter
    uint32_t rs, nz;    // run starts of the pair, non-empty run-start words of the element
    uint32_t xp[16];    // P's rows (the widest class reads them again)
};

// First part of an item of a colour group: entries [k0, k1) (at most E) of the
// group's elements -- positions k0 .. k1 - 1, or the positions qlist[k0 .. k1)
// of a list (the learned filter's, or an element class's) -- with every word.  Donor tables and the trials' entries: all of it from P, which does
// not change during a generation, so a tile makes the first item of a group
// between its arrival at the barrier that opens the group and its wait there.
template <int SB, bool LEARN>
__device__ __forceinline__ void bs_prepare(const GomParams &P, const BsMap &M, const int32_t *qlist, int k0, int k1,
                                           uint32_t g, BsItem &I)
{
    const int lane = threadIdx.x & 31, slot = M.slot;
    const int W = P.W, Wv = P.Wv, p = P.p, S = SB <= 13 ? SB : min(P.bs_S, SB);
    const int e = M.e, w = M.w, b2 = e * Wv; // b2: the element's first slot
    const bool ke = M.in && k0 + e < k1;     // this lane's pair exists
    int q = k0 + e;
    I.audited = false;
    if (qlist && ke) {
        const int32_t en = qlist[k0 + e];
        q = en & 0x7FFFFFFF;
        I.audited = LEARN && en < 0;
    }
    I.q = q;
    I.ke = ke;
    constexpr int EW = bs_entry_words(SB), TB = bs_table(SB);
    uint32_t *tab = M.sm, *res = M.sm + 32 * EW;
    uint32_t *sRS = M.sm + 64 * EW + 32 * S, *sLst = sRS + 32, *sFst = sLst + 32;
    const int lim = p - 32 * w; // >= 1
    const uint32_t vm = lim >= 32 ? 0xFFFFFFFFu : (1u << lim) - 1u; // this word's individuals

    // ---- phase 0: P's rows, run starts, donor table
    int j = 0, s = 0, f0 = 0, d0 = 0, n_in = 0, n_out = 0;
    if (ke) {
        const int4 a = __ldg(P.hdr + 2 * q), b = __ldg(P.hdr + 2 * q + 1);
        j = a.x;
        f0 = a.y;
        d0 = a.z;
        s = a.w & 0xFF;
        n_in = a.w >> 8;
        n_out = b.x;
        // the element's edge list is read in phase 2: ask for its lines in L2
        // now (the Wv words of the element take every Wv-th line; the array
        // starts on a 256-byte boundary, so every line named here holds bytes
        // of it)
        const uintptr_t d_at = reinterpret_cast<uintptr_t>(P.bdep + d0), d_end = d_at + 8u * (uint32_t)(n_out + n_in);
        for (uintptr_t at = (d_at & ~uintptr_t(127)) + 128u * (uint32_t)w; at < d_end; at += 128u * (uint32_t)Wv)
            prefetch_l2(reinterpret_cast<const void *>(at));
    }
    I.j = j;
    I.s = s;
    I.f0 = f0;
    I.d0 = d0;
    I.n_in = n_in;
    I.n_out = n_out;
    uint32_t xp[SB];
#pragma unroll
    for (int a = 0; a < SB; ++a) xp[a] = 0;
#pragma unroll
    for (int a8 = 0; a8 < SB; a8 += 8) {
        if (a8 < S) {
            constexpr int C = SB < 8 ? SB : 8;
            int at[C];
#pragma unroll
            for (int c = 0; c < C; ++c) at[c] = a8 + c < SB && ke && a8 + c < s ? __ldg(P.fv + f0 + a8 + c) * W + w : -1;
#pragma unroll
            for (int c = 0; c < C; ++c)
                if (a8 + c < SB) xp[a8 + c < SB ? a8 + c : 0] = at[c] >= 0 ? P.P[at[c]] : 0u;
        }
    }
    if constexpr (SB <= 16) {
#pragma unroll
        for (int a = 0; a < SB; ++a) I.xp[a] = xp[a];
    }
    uint32_t rs = 0, nx, nz;
    {   // run starts of the element's patterns in word w: bit b set iff the
        // pattern of individual 32 w + b differs from the one before it
        // (cyclically: the word before's last individual); the pattern at the
        // word's first run start
        const int lastb = lim >= 32 ? 31 : lim - 1;
        uint32_t lst = 0;
#pragma unroll
        for (int a = 0; a < SB; ++a)
            if (a < S) lst |= ((xp[a] >> lastb) & 1u) << a;
        sLst[slot] = lst;
        tile_sync(M);
        const uint32_t prv = sLst[M.in ? b2 + (w == 0 ? Wv - 1 : w - 1) : slot];
#pragma unroll
        for (int a = 0; a < SB; ++a)
            if (a < S) rs |= xp[a] ^ __funnelshift_l(prv << (31 - a), xp[a], 1);
        rs = ke ? rs & vm : 0u;
        sRS[slot] = rs;
        const int fb = rs ? __ffs(rs) - 1 : 0;
        uint32_t fst = 0;
#pragma unroll
        for (int a = 0; a < SB; ++a)
            if (a < S) fst |= ((xp[a] >> fb) & 1u) << a;
        sFst[slot] = fst;
        tile_sync(M);
        // the element's words with a run start: bits b2 .. of the ballot over all slots
        const uint32_t nzb = __ballot_sync(kFull, lane < M.E * Wv && sRS[lane] != 0);
        nz = Wv == 32 ? nzb : (nzb >> b2) & ((1u << Wv) - 1u);
        // the first run start after word w (cyclically): its pattern carries into
        // the word's last individuals; without any run start every pattern is the same
        const uint32_t later = nz & ~((2u << w) - 1u); // words after w
        const uint32_t any = later ? later : nz;        // else wrap round
        nx = any ? sFst[b2 + __ffs(any) - 1] : fst;
        I.rs = rs;
        I.nz = nz;
    }
    {
        uint32_t x[TB];
#pragma unroll
        for (int a = 0; a < TB; ++a) x[a] = a < SB ? xp[a < SB ? a : 0] : 0u;
        transpose_lane<TB>(x); // block column c of x[r]: the pattern of individual 32 w + TB c + r
        if (TB < 32) nx <<= 32 - TB;
        if constexpr (TB == 8) {
#pragma unroll
            for (int c = 3; c >= 0; --c) {
                uint32_t ent[4]; // two entries each
#pragma unroll
                for (int r = 6; r >= 0; r -= 2) {
                    const uint32_t hi = __byte_perm(x[r + 1], nx, c | (c + 4) << 4);
                    if ((rs >> (8 * c + r + 1)) & 1u) nx = x[r + 1];
                    const uint32_t lo = __byte_perm(x[r], nx, c | (c + 4) << 4);
                    if ((rs >> (8 * c + r)) & 1u) nx = x[r];
                    ent[r / 2] = __byte_perm(lo, hi, 0x5410);
                }
                nx >>= 8;
                *reinterpret_cast<uint4 *>(tab + 16 * slot + 4 * c) = make_uint4(ent[0], ent[1], ent[2], ent[3]);
            }
        } else if constexpr (TB == 16) {
#pragma unroll
            for (int c = 1; c >= 0; --c) {
#pragma unroll
                for (int r = 15; r >= 0; --r) {
                    // word 32 slot + d rotated by the slot: 32 slots hit 32 banks
                    tab[32 * slot + ((16 * c + r + slot) & 31)] = __byte_perm(x[r], nx, c ? 0x7632 : 0x5410);
                    if ((rs >> (16 * c + r)) & 1u) nx = x[r];
                }
                nx >>= 16;
            }
        } else {
#pragma unroll
            for (int r = 31; r >= 0; --r) {
                const int at = 32 * slot + ((r + slot) & 31);
                tab[at] = x[r];
                tab[1024 + at] = nx;
                if ((rs >> r) & 1u) nx = x[r];
            }
        }
    }
    tile_sync(M);

    // ---- phase 1: donors, on the warp's own 32 / 2^lsh slots.  Call (slot k2,
    // c) covers individuals 32 w2 + 4c .. + 3; the starts of individuals past p
    // (in the last word's last call) stay below 32 Wv, inside the element's table
    const int own = 32 >> M.lsh, k0w = slot & ~(own - 1); // slots of a warp are aligned to their number
    const int info = ke ? w | b2 << 8 | 1 << 16 : 0;
#pragma unroll 1
    for (int r = 0; r < own; r += 4) {
        const int kl = r + (lane >> 3), c = lane & 7;
        const int src = (kl & (own - 1)) << M.lsh, k2 = k0w + kl;
        const int j2 = __shfl_sync(kFull, j, src), inf2 = __shfl_sync(kFull, info, src);
        if (kl < own && inf2) {
            const int w2 = inf2 & 0xFF, b2 = (inf2 >> 8) & 0xFF; // b2: that element's first slot
            const uint4 r4 = philox10_rk(make_uint4((uint32_t)j2, (uint32_t)(8 * w2 + c), g, kTagDonor), P.rk);
            const int i0 = 32 * w2 + 4 * c;
            uint32_t en[4], en2[4];
    #pragma unroll
            for (int cc = 0; cc < 4; ++cc) {
                const uint32_t d = (uint32_t)(i0 + cc + 1) + __umulhi(pick(r4, cc), (uint32_t)(p - 1));
                const uint32_t st = min(d, d - (uint32_t)p); // d < p: d - p wraps above d
                if constexpr (TB == 8) {
                    en[cc] = reinterpret_cast<const uint16_t *>(tab)[32 * b2 + st];
                } else {
                    const uint32_t k3 = (uint32_t)b2 + (st >> 5), at = 32 * k3 + ((st + k3) & 31);
                    en[cc] = tab[at];
                    if constexpr (TB == 32) en2[cc] = tab[1024 + at];
                }
            }
            if constexpr (TB == 8) {
                *reinterpret_cast<uint2 *>(res + 16 * k2 + (((c >> 1) ^ ((k2 >> 1) & 3)) << 2) + ((c & 1) << 1)) =
                    make_uint2(__byte_perm(en[0], en[1], 0x5410), __byte_perm(en[2], en[3], 0x5410));
            } else {
                uint32_t *at = res + 32 * k2 + ((c ^ (k2 & 7)) << 2);
                *reinterpret_cast<uint4 *>(at) = make_uint4(en[0], en[1], en[2], en[3]);
                if constexpr (TB == 32) *reinterpret_cast<uint4 *>(at + 1024) = make_uint4(en2[0], en2[1], en2[2], en2[3]);
            }
        }
    }
    __syncwarp(); // (a warp reads its own slots' entries)
}

// Adds the toggled edges of an element's trials in word w (32 individuals)
// into D: part `part` of `parts` of the first `ne` of its edges list(x), four at
// a time.  myD, myO: the flip planes and the parent's rows of the word,
// variable a at 32 a.
template <int R, int UB, class List>
__device__ __forceinline__ void bs_edges_add(const GomParams &P, const BsItem &I, List list, int ne, int part,
                                             int parts, int w, const uint32_t *myD, const uint32_t *myO,
                                             uint32_t (&D)[R + 1])
{
    for (int x = 4 * part; x < ne; x += 4 * parts) { // four edges' loads issued before their arithmetic
        int2 ed[4];
        uint32_t pos[4], neg[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) ed[u] = x + u < ne ? list(x + u) : make_int2(0, 0); // weight 0
#pragma unroll
        for (int u = 0; u < 4; ++u) { // the far end's word, and whether a trial flips it too
            neg[u] = x + u < I.n_out ? P.O[ed[u].x + w] : myO[ed[u].x];
            pos[u] = x + u < I.n_out ? 0u : myD[ed[u].x];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int ra = ed[u].y & kEdgeRowMask;
            const uint32_t tg = myD[ra] ^ pos[u], cut = myO[ra] ^ neg[u] ^ (uint32_t)(ed[u].y >> 31);
            pos[u] = tg & ~cut;
            neg[u] = tg & cut;
        }
        add_signed4<R + 1, UB>(D, pos, neg, ed);
    }
}

// Second part of an item, in its group: the parent's rows, the flip planes,
// the partial evaluation, acceptance and writes of all its trials (Alg. 2).
template <int SB, int R, int UB, bool LEARN>
__device__ __forceinline__ void bs_item(const GomParams &P, const BsMap &M, const BsItem &I, uint32_t g,
                                        BsLane<FitShared> &L, long long *s_f, unsigned long long *s_fc)
{
    const int slot = M.slot;
    const int W = P.W, p = P.p, S = SB <= 13 ? SB : min(P.bs_S, SB);
    const int w = M.w, b2 = M.e * P.Wv, s = I.s;
    const bool ke = I.ke;
    constexpr int EW = bs_entry_words(SB), TB = bs_table(SB);
    const uint32_t *tab = M.sm;
    uint32_t *res = M.sm + 32 * EW;
    uint32_t *sF = res; // flip planes, once every lane has read its entries back
    uint32_t *sX = M.sm + 64 * EW, *sRS = sX + 32 * S;
    const int lim = p - 32 * w; // >= 1
    const uint32_t vm = lim >= 32 ? 0xFFFFFFFFu : (1u << lim) - 1u; // this word's individuals

    uint32_t chg = kFull; // individuals that changed on F_j since the generation start
#pragma unroll
    for (int a8 = 0; a8 < SB; a8 += 8) {
        if (a8 < S) {
            constexpr int C = SB < 8 ? SB : 8;
            int at[C];
            uint32_t xo[C];
#pragma unroll
            for (int c = 0; c < C; ++c) at[c] = a8 + c < SB && ke && a8 + c < s ? __ldg(P.fv + I.f0 + a8 + c) * W + w : -1;
#pragma unroll
            for (int c = 0; c < C; ++c) xo[c] = at[c] >= 0 ? P.O[at[c]] : 0u;
            if constexpr (SB > 16) {
                if (a8 == 0) chg = 0;
#pragma unroll
                for (int c = 0; c < C; ++c) chg |= at[c] >= 0 ? xo[c] ^ P.P[at[c]] : 0u;
            }
#pragma unroll
            for (int c = 0; c < C; ++c)
                if (a8 + c < S) sX[32 * (a8 + c) + slot] = xo[c];
        }
    }

    // the entries back as planes: t1[a] the starts' bits, then t2[a] the
    // fall-through patterns' bits; f1: the individuals whose start differs
    uint32_t F[TB];
    uint32_t f1 = 0, same = kFull; // same: the fall-through pattern is the individual's own in P
    {
        uint32_t t2[TB];
        if constexpr (TB == 8) {
            const int sw = (slot >> 1) & 3;
#pragma unroll
            for (int h = 0; h < 2; ++h) { // chunk i holds individuals 8 i .. 8 i + 7; half h of each
                uint32_t A[4][2];          // [i][k]: individuals 8 i + 4 h + 2 k, + 1
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint2 v = *reinterpret_cast<const uint2 *>(res + 16 * slot + ((i ^ sw) << 2) + 2 * h);
                    A[i][0] = v.x;
                    A[i][1] = v.y;
                }
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int r = 4 * h + 2 * k;
                    const uint32_t l0 = __byte_perm(A[0][k], A[1][k], 0x5140), h0 = __byte_perm(A[0][k], A[1][k], 0x7362);
                    const uint32_t l1 = __byte_perm(A[2][k], A[3][k], 0x5140), h1 = __byte_perm(A[2][k], A[3][k], 0x7362);
                    F[r] = __byte_perm(l0, l1, 0x5410);
                    t2[r] = __byte_perm(l0, l1, 0x7632);
                    F[r + 1] = __byte_perm(h0, h1, 0x5410);
                    t2[r + 1] = __byte_perm(h0, h1, 0x7632);
                }
            }
            transpose_lane<TB>(F);
            transpose_lane<TB>(t2);
        } else if constexpr (TB == 16) {
#pragma unroll
            for (int i = 0; i < 4; ++i) { // individuals 4 i .. + 3 and 16 + 4 i .. + 3
                const uint4 u = *reinterpret_cast<const uint4 *>(res + 32 * slot + ((i ^ (slot & 7)) << 2));
                const uint4 v = *reinterpret_cast<const uint4 *>(res + 32 * slot + (((i + 4) ^ (slot & 7)) << 2));
                F[4 * i] = __byte_perm(u.x, v.x, 0x5410);
                F[4 * i + 1] = __byte_perm(u.y, v.y, 0x5410);
                F[4 * i + 2] = __byte_perm(u.z, v.z, 0x5410);
                F[4 * i + 3] = __byte_perm(u.w, v.w, 0x5410);
                t2[4 * i] = __byte_perm(u.x, v.x, 0x7632);
                t2[4 * i + 1] = __byte_perm(u.y, v.y, 0x7632);
                t2[4 * i + 2] = __byte_perm(u.z, v.z, 0x7632);
                t2[4 * i + 3] = __byte_perm(u.w, v.w, 0x7632);
            }
            transpose_lane<TB>(F);
            transpose_lane<TB>(t2);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint4 u = *reinterpret_cast<const uint4 *>(res + 32 * slot + ((i ^ (slot & 7)) << 2));
                F[4 * i] = u.x;
                F[4 * i + 1] = u.y;
                F[4 * i + 2] = u.z;
                F[4 * i + 3] = u.w;
            }
            transpose_lane<TB>(F);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint4 u = *reinterpret_cast<const uint4 *>(res + 1024 + 32 * slot + ((i ^ (slot & 7)) << 2));
                t2[4 * i] = u.x;
                t2[4 * i + 1] = u.y;
                t2[4 * i + 2] = u.z;
                t2[4 * i + 3] = u.w;
            }
            transpose_lane<TB>(t2);
        }
#pragma unroll
        for (int a = 0; a < SB; ++a)
            if (a < S) f1 |= F[a] ^ sX[32 * a + slot];
        if constexpr (SB <= 16) {
#pragma unroll
            for (int a = 0; a < SB; ++a)
                if (a < S) same &= ~(t2[a] ^ I.xp[a]);
        }
        // every candidate from the start up to the next run start has the
        // start's pattern; when that is the parent's, the run start differs
        // and is the donor, with no run start at all the entry repeats P_d:
        // no flips, no donor
#pragma unroll
        for (int a = 0; a < SB; ++a)
            if (a < S) F[a] = ((f1 & F[a]) | (~f1 & t2[a])) ^ sX[32 * a + slot];
    }
    tile_sync(M); // every lane has read its entries: their slots take the flip planes
    uint32_t hd = 0; // individuals with a donor
#pragma unroll
    for (int a = 0; a < SB; ++a)
        if (a < S) {
            const uint32_t Fa = ke ? F[a] & vm : 0u;
            hd |= Fa;
            sF[32 * a + slot] = Fa;
        }
    __syncwarp(); // every lane of a pair has stored its planes: the first one may correct them
    // An individual that is itself the run start the search falls through to
    // is skipped (a donor is another individual).  Its start equals the parent
    // and the fall-through is its own pattern in P, another one: only an
    // individual that changed in this generation can be (for the widest
    // class that is all that is checked here).
    uint32_t cand = ke ? ~f1 & I.rs & chg & same : 0u;
    while (cand) { // divergent, rare
        const int b = __ffs(cand) - 1, i = 32 * w + b;
        cand &= cand - 1;
        uint32_t fl;
        if (!self_hit<SB>(&fl, tab, sRS + b2, I.nz, b2, I.j, i, g, p, P.seed)) continue;
        hd = (hd & ~(1u << b)) | ((fl ? 1u : 0u) << b);
        if (M.sub == 0)
            for (int a = 0; a < s; ++a) {
                uint32_t *row = sF + 32 * a + slot;
                *row = (*row & ~(1u << b)) | (((fl >> a) & 1u) << b);
            }
    }
    __syncwarp();

    // ---- phase 2: bit-plane partial evaluation, acceptance, write
    unsigned i_acc = 0, i_dl = 0, i_imp = 0; // this pair's accepted, donor-less and improving trials
    // each item adds less than 2^R to an individual's sum: flush before it could pass 2^kFitPlanes
    if (L.since_flush >= (1 << (kFitPlanes - R))) bs_flush(L, s_f);
    {
        const uint32_t *myD = sF + slot, *myO = sX + slot; // variable a at word 32 a
        // the delta of every trial, R + 1 planes two's complement: an edge that
        // a trial toggles adds |w| if it was uncut (with its sign folded into
        // the cut bit), -|w| if it was cut (Eq. 1); no partial sum leaves
        // (-2^R, 2^R) since the element's sum of |w| is below 2^R
        uint32_t D[R + 1];
#pragma unroll
        for (int t = 0; t <= R; ++t) D[t] = 0;
        bs_edges_add<R, UB>(P, I, [&](int x) { return __ldg(P.bdep + I.d0 + x); }, ke ? I.n_out + I.n_in : 0, M.sub, 1 << M.lsh, w, myD, myO, D);
        for (int off = 1; off < 1 << M.lsh; off <<= 1) { // the sums of the pair's lanes
            uint32_t carry = 0;
#pragma unroll
            for (int t = 0; t <= R; ++t) {
                const uint32_t a = D[t], b = __shfl_xor_sync(kFull, a, off);
                D[t] = a ^ b ^ carry;
                carry = (a & b) | (a & carry) | (b & carry);
            }
        }
        uint32_t nzd = 0;
#pragma unroll
        for (int t = 0; t <= R; ++t) nzd |= D[t];
        const uint32_t neg = D[R];
        const uint32_t pos = nzd & ~neg;
        const uint32_t eqv = P.eqw[(g & 1) * W + w];
        const uint32_t acc = hd & (pos | (~nzd & ~eqv));
        if (ke && M.sub == 0) {
            i_acc = __popc(acc);
            i_imp = __popc(acc & pos);
            i_dl = __popc(vm & ~hd);
            L.n_acc += i_acc;
            L.n_imp += i_imp;
            L.n_dl += i_dl;
            if (P.fi.on && acc) atomicOr(&P.fi.accw[w], acc); // Forced Improvement: who had an accepted step
        }
        if (acc) {
            for (int a = M.sub; a < s; a += 1 << M.lsh) {
                const uint32_t m = myD[32 * a] & acc;
                if (m) {
                    const int64_t v = __ldg(P.fv + I.f0 + a);
                    P.O[v * W + w] = myO[32 * a] ^ m;
                }
            }
            if (M.sub == 0) fit_add<R>(L, D, acc); // the accepted deltas (>= 0, below 2^R)
        }
    }
    ++L.since_flush;
    tile_sync(M); // the region may be rewritten
    if (LEARN && P.learn) bs_record(P, I.q, ke, I.audited, g, i_acc, i_dl, i_imp, s_fc);
}

// The elements of colour c that run: positions, or with the learned filter
// skipping, entries of the compacted list.
struct BsGroup {
    const int32_t *qlist;
    int ka, kz, items;
};

template <bool LEARN>
__device__ __forceinline__ BsGroup bs_group(const GomParams &P, const BsMap &M, int c)
{
    const bool cl = LEARN && P.learn == 2 && P.flt.compact;
    BsGroup G;
    G.qlist = cl ? P.flt.act : nullptr;
    G.ka = cl ? P.flt.act_ptr[c] : P.cptr[c];
    G.kz = cl ? P.flt.act_ptr[c + 1] : P.cptr[c + 1];
    G.items = (G.kz - G.ka + M.E - 1) / M.E;
    return G;
}

// One colour group (position t) on the bit-sliced path: items of E consecutive
// elements; tile x takes item x first -- prepared before `open`, the barrier
// that opens the group (false: it gave up) --, then items ntiles + the claims
// it draws from work[t] (P.dyn; one-warp tiles, of equal items), one ahead, or x + ntiles, x +
// 2 ntiles, ... (static stride).
template <int SB, int R, int UB, bool LEARN, class Open>
__device__ __forceinline__ bool phase_mix_bs(const GomParams &P, const BsMap &M, int t, int c, uint32_t g, Open open,
                                             BsLane<FitShared> &L, long long *s_f, unsigned long long *s_fc)
{
    const int lane = threadIdx.x & 31;
    const BsGroup G = bs_group<LEARN>(P, M, c);
    const bool dyn = P.dyn && M.nwi == 1;
    unsigned claim = 0;
    BsItem I;
    for (int it = M.tile, next = M.tile + M.ntiles, first = 1;; first = 0) { // (one call site of either part)
        const int k0 = G.ka + it * M.E;
        if (it < G.items) bs_prepare<SB, LEARN>(P, M, G.qlist, k0, min(k0 + M.E, G.kz), g, I);
        if (first && !open()) return false;
        if (it >= G.items) return true;
        if (dyn && lane == 0) claim = atomicAdd(&P.work[t], 1u);
        bs_item<SB, R, UB, LEARN>(P, M, I, g, L, s_f, s_fc);
        it = dyn ? M.ntiles + (int)__shfl_sync(kFull, claim, 0) : next;
        next += M.ntiles;
    }
}

// Adds the warp's counters and the lanes' fitness sums into the block's
// accumulators.
__device__ __forceinline__ void bs_finish_generation(const GomParams &P, BsLane<FitShared> &L, long long *s_f,
                                                     unsigned long long *s_cnt)
{
    bs_flush(L, s_f);
    count_flush(s_cnt, L.n_dl, L.n_acc, L.n_imp);
    L.n_dl = L.n_acc = L.n_imp = 0;
}

// Up to G generations of one context on the bit-sliced phase, on the blocks
// of the (virtual) grid V, the phases separated by grid barriers on `bar`:
// [generation start + group order] | group 0 | ... | group k-1 | and again,
// each tile preparing its first item of a group before its wait at the group's barrier;
// every block computes a generation's end from the fitness array after the
// barrier that closes its last group (block 0 of V records it).  s_keys: room
// for the k group keys of the order phase (it may overlay the regions and s_f, which
// are set up after it); fit, w: the lane's fitness planes and their word; s_f, s_cnt: the block's
// fitness accumulators and counters; s_fc: the learned filter's block
// counters (LEARN only).
// FI: the Forced Improvement option exists here.  mix(t, c, g, open, L) mixes the group at position t, colour c, calling open()
// -- the wait at the barrier that opens the group -- once in every thread, and
// is false when that gave up.
template <int R, bool LEARN, bool FI, class Mix>
__device__ __forceinline__ void bs_run(const GomParams &P, const VGrid &V, GomBarrier *bar, int G, int64_t target,
                                       unsigned long long *s_keys, uint32_t *fit, int w, long long *s_f,
                                       unsigned long long *s_cnt, unsigned long long *s_fc, Mix mix)
{
    const unsigned nblk = (unsigned)V.nblk;
    const bool lead = V.blk == 0;
    uint32_t g = P.st->g;
    GenEnd e{P.st->fe, P.st->improved, P.st->argmax};
    unsigned long long bnext = 0;
    if (threadIdx.x == 0) bnext = barrier_first(&bar->count, nblk);
    if (lead && threadIdx.x == 0) {
        P.st->call_g0 = g;
        P.st->target = target;
    }
    const bool tr = P.trace != nullptr && lead && threadIdx.x == 0;
    BsLane<FitShared> L;
    L.fit.v = fit;
    for (int qg = 0; qg < G; ++qg) {
        if (qg > 0 && phase_gen_end(P, target, g - 1, e, lead)) return;
        if (tr) P.trace[0] = global_ns();
        phase_gen_start(P, V, e.improved, e.argmax, g, true);
        phase_order(P, V, s_keys, g);
        if (LEARN) fc_zero(s_fc);
        acc_zero(P, s_f, s_cnt);
        bs_lane_zero(L, w); // (the order phase's keys overlay the planes)
        if (tr) P.trace[1] = P.trace[2] = global_ns();
        if (!grid_barrier(&bar->count, &P.st->err, nblk, bnext, kBarrierNs)) return;
        if (LEARN && P.learn && !phase_filter_select(P, V, g, &bar->count, nblk, bnext, P.learn == 2 && P.flt.compact))
            return;
        if (tr) P.trace[3] = global_ns();
        for (int t = 0; t < P.k; ++t) {
            const auto open = [&] {
                if (t > 0 && !grid_wait(&bar->count, &P.st->err, nblk, bnext, kBarrierNs)) return false;
                if (tr) P.trace[4 + 2 * t] = global_ns();
                return true;
            };
            if (!mix(t, P.order[t], g, open, L)) return;
            if (tr) P.trace[5 + 2 * t] = global_ns();
            if (t + 1 < P.k) grid_arrive(&bar->count, nblk);
        }
        bs_finish_generation(P, L, s_f, s_cnt);
        acc_flush(P, s_f, s_cnt);
        if (LEARN) fc_flush(P, s_fc);
        if (!grid_barrier(&bar->count, &P.st->err, nblk, bnext, kBarrierNs)) return;
        if (FI && P.fi.on && !fi_generation<(R <= 12 ? 12 : 16)>(P, V, &bar->count, nblk, bnext, e, P.order, s_f, s_cnt)) return;
        if (tr) P.trace[4 + 2 * P.k] = global_ns();
        ++g;
    }
    if (G > 0 && lead) phase_gen_end(P, target, g - 1, e, true);
}

template <int SB, int R, int UB, bool LEARN, bool FI = true>
__device__ __forceinline__ void bs_generations(const GomParams &P, const VGrid &V, GomBarrier *bar, int G,
                                               int64_t target, unsigned long long *s_keys, uint32_t *regions,
                                               long long *s_f, unsigned long long *s_cnt, unsigned long long *s_fc)
{
    const BsMap M = bs_map<LEARN>(P, V, regions, P.bs_words);
    bs_run<R, LEARN, FI>(P, V, bar, G, target, s_keys, bs_fit(P, regions), M.w, s_f, s_cnt, s_fc,
                     [&](int t, int c, uint32_t g, auto &open, BsLane<FitShared> &L) {
                         return phase_mix_bs<SB, R, UB, LEARN>(P, M, t, c, g, open, L, s_f, s_fc);
                     });
}

} // namespace
