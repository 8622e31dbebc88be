// gom_bs_multi.cuh -- the bit-sliced mixing of linkage models with elements of
// many sizes (linkage trees: half the elements are single variables, a few
// have a hundred): each colour group's elements in lists by class, the small
// ones (at most 8, 16 or 32 variables) as the items of gom_bs.cuh in their own
// class's tables, the large ones (33 to 128 variables) by a block each.
// Anonymous namespace: each translation unit that includes it compiles its
// own copy.
//
// A large element (bs_large_*): lane = population word; warp c of the block
// has the variables 32 c .. 32 c + 31.  The same three steps as a small item:
// donor tables from P by transposes inside the lanes, with the run starts and
// the differences combined over the warps through shared memory; one Philox
// call for four starts and one 16-byte table entry per pattern; the flip
// planes by the inverse transposes; then the element's edges split over the
// block's warps and their plane sums added.  Group of a 100x100 torus' tree of
// bound 128 (p = 1,024; 25 elements above 64 variables, 900 below 9): 85 -> 19
// us against a block per element and scalar deltas for every size.
#pragma once

#include "gom_bs.cuh"

namespace {

constexpr int kLargeChunks = 4; // 128 variables in words of 32

// Shared-memory words of a block's large element: the tables of P_d and N_d
// [32 Wv individuals][4], later the warps' plane sums; the trials' entries of
// both [4][Wv][32], later the flip planes [128][32]; the rows of O [128][32];
// partial masks [4 warps][32] of four kinds and block-wide ones; the
// variables' word offsets [128] and the element's edges [most of any].
__host__ __device__ __forceinline__ int bs_large_tab(int Wv, int warps)
{
    return 256 * Wv > warps * 21 * 32 ? 256 * Wv : warps * 21 * 32;
}
__host__ __device__ __forceinline__ int bs_large_res(int Wv) { return 256 * Wv > 4096 ? 256 * Wv : 4096; }
__host__ __device__ __forceinline__ int bs_large_words(int Wv, int warps, int edges)
{
    return bs_large_tab(Wv, warps) + bs_large_res(Wv) + 4096 + 6 * 128 + (2 * edges + 3) / 4 * 4;
}

struct BsLargeSm {
    uint32_t *tabP, *tabN, *res1, *res2, *sF, *sX, *sD;
    uint32_t *rs_c, *f1_c, *chg_c, *hd_c; // [4][32] per chunk
    uint32_t *rs, *hd, *acc;              // [32]
    int *var;                             // [128] v W
    int2 *edge;
};

__device__ __forceinline__ BsLargeSm bs_large_sm(const GomParams &P, uint32_t *sm)
{
    BsLargeSm S;
    const int Wv = P.Wv;
    S.tabP = sm;
    S.tabN = sm + 128 * Wv;
    S.sD = sm;
    S.res1 = sm + bs_large_tab(Wv, blockDim.x >> 5);
    S.res2 = S.res1 + 128 * Wv;
    S.sF = S.res1;
    S.sX = S.res1 + bs_large_res(Wv);
    S.rs_c = S.sX + 4096;
    S.f1_c = S.rs_c + 128;
    S.chg_c = S.f1_c + 128;
    S.hd_c = S.chg_c + 128;
    S.rs = S.hd_c + 128;
    S.hd = S.rs + 32;
    S.acc = S.hd + 32;
    S.var = reinterpret_cast<int *>(S.rs + 128);
    S.edge = reinterpret_cast<int2 *>(S.var + 128);
    return S;
}

// Table slot of individual i: rotated inside its word, so that the lanes of a
// word's individual r do not all hit the same banks.
__device__ __forceinline__ int large_slot(int i)
{
    const int w = i >> 5;
    return 32 * w + ((i + w) & 31);
}

__device__ __forceinline__ uint32_t or4(const uint32_t *x, int lane, int n)
{
    uint32_t y = x[lane];
    for (int c = 1; c < n; ++c) y |= x[32 * c + lane];
    return y;
}

// First part of a large element: donor tables and the trials' entries, from P
// only.  Every thread of the block (at least four warps).
__device__ __forceinline__ void bs_large_prepare(const GomParams &P, int q, uint32_t g, uint32_t *sm, BsItem &I)
{
    const BsLargeSm S = bs_large_sm(P, sm);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int W = P.W, Wv = P.Wv, p = P.p, w = lane;
    const bool kw = w < Wv;
    const int4 a = __ldg(P.hdr + 2 * q), b = __ldg(P.hdr + 2 * q + 1);
    I.q = q;
    I.j = a.x;
    I.f0 = a.y;
    I.d0 = a.z;
    I.s = a.w & 0xFF;
    I.n_in = a.w >> 8;
    I.n_out = b.x;
    const int s = I.s, nch = (s + 31) >> 5, v0 = 32 * wib;
    const bool mine = wib < nch;
    const int lim = p - 32 * w;
    const uint32_t vm = lim >= 32 ? 0xFFFFFFFFu : lim > 0 ? (1u << lim) - 1u : 0u;
    for (int x = threadIdx.x; x < I.n_out + I.n_in; x += blockDim.x) S.edge[x] = __ldg(P.bdep + I.d0 + x);
    for (int x = threadIdx.x; x < s; x += blockDim.x) S.var[x] = __ldg(P.fv + I.f0 + x) * W;
    uint32_t x[32];
#pragma unroll
    for (int r = 0; r < 32; ++r) x[r] = 0;
    if (mine) {
#pragma unroll
        for (int r8 = 0; r8 < 32; r8 += 8) {
            int at[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) at[r] = kw && v0 + r8 + r < s ? __ldg(P.fv + I.f0 + v0 + r8 + r) * W + w : -1;
#pragma unroll
            for (int r = 0; r < 8; ++r) x[r8 + r] = at[r] >= 0 ? P.P[at[r]] : 0u;
        }
        const int lastb = lim >= 32 ? 31 : lim > 0 ? lim - 1 : 0;
        uint32_t lst = 0, rs = 0;
#pragma unroll
        for (int r = 0; r < 32; ++r) lst |= ((x[r] >> lastb) & 1u) << r;
        const uint32_t prv = __shfl_sync(kFull, lst, w == 0 || !kw ? Wv - 1 : w - 1);
#pragma unroll
        for (int r = 0; r < 32; ++r) rs |= x[r] ^ __funnelshift_l(prv << (31 - r), x[r], 1);
        S.rs_c[32 * wib + lane] = kw ? rs & vm : 0u;
    }
    __syncthreads();
    I.rs = or4(S.rs_c, lane, nch);
    I.nz = __ballot_sync(kFull, I.rs != 0);
    if (wib == 0) S.rs[lane] = I.rs;
    if (mine) {
        const int fb = I.rs ? __ffs(I.rs) - 1 : 0;
        uint32_t fst = 0;
#pragma unroll
        for (int r = 0; r < 32; ++r) fst |= ((x[r] >> fb) & 1u) << r;
        const uint32_t later = I.nz & ~((2u << w) - 1u), any = later ? later : I.nz;
        uint32_t nx = __shfl_sync(kFull, fst, any ? __ffs(any) - 1 : w);
        transpose_lane<32>(x);
        if (kw) {
#pragma unroll
            for (int r = 31; r >= 0; --r) {
                const int at = 4 * (32 * w + ((r + w) & 31)) + wib;
                S.tabP[at] = x[r];
                S.tabN[at] = nx;
                if ((I.rs >> r) & 1u) nx = x[r];
            }
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int id = threadIdx.x; id < 8 * Wv; id += blockDim.x) {
        const int w2 = id >> 3, c4 = id & 7;
        const uint4 r4 = philox10_rk(make_uint4((uint32_t)I.j, (uint32_t)(8 * w2 + c4), g, kTagDonor), P.rk);
        int sl[4];
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
            const uint32_t d = (uint32_t)(32 * w2 + 4 * c4 + cc + 1) + __umulhi(pick(r4, cc), (uint32_t)(p - 1));
            sl[cc] = large_slot((int)min(d, d - (uint32_t)p));
        }
        const int to = 32 * w2 + ((c4 ^ (w2 & 7)) << 2);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint4 *tab = reinterpret_cast<const uint4 *>(h ? S.tabN : S.tabP);
            uint32_t *res = (h ? S.res2 : S.res1) + to;
            const uint4 e0 = tab[sl[0]], e1 = tab[sl[1]], e2 = tab[sl[2]], e3 = tab[sl[3]];
            *reinterpret_cast<uint4 *>(res) = make_uint4(e0.x, e1.x, e2.x, e3.x);
            *reinterpret_cast<uint4 *>(res + 32 * Wv) = make_uint4(e0.y, e1.y, e2.y, e3.y);
            if (nch > 2) *reinterpret_cast<uint4 *>(res + 64 * Wv) = make_uint4(e0.z, e1.z, e2.z, e3.z);
            if (nch > 3) *reinterpret_cast<uint4 *>(res + 96 * Wv) = make_uint4(e0.w, e1.w, e2.w, e3.w);
        }
    }
}

// The planes of chunk `c` from the trials' entries of word w (this lane's).
__device__ __forceinline__ void large_planes(const uint32_t *res, int Wv, int c, int w, uint32_t (&x)[32])
{
    const uint32_t *at = res + 32 * (Wv * c + w);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint4 v = *reinterpret_cast<const uint4 *>(at + ((i ^ (w & 7)) << 2));
        x[4 * i] = v.x;
        x[4 * i + 1] = v.y;
        x[4 * i + 2] = v.z;
        x[4 * i + 3] = v.w;
    }
    transpose_lane<32>(x);
}

// A large element's individual i, as self_hit of the small ones: its start is
// drawn again; false unless the next run start after it is i itself, else the
// donor's flips in fl[0 .. nch).
__device__ __noinline__ bool large_self_hit(uint32_t *fl, const uint32_t *tabP, const uint32_t *tabN, const uint32_t *rs,
                                            uint32_t nz, int nch, int j, int i, uint32_t g, int p, uint64_t seed)
{
    const uint4 r4 = philox10(make_uint4((uint32_t)j, (uint32_t)(i >> 2), g, kTagDonor), (uint32_t)seed,
                              (uint32_t)(seed >> 32));
    const uint32_t d = (uint32_t)(i + 1) + __umulhi(pick(r4, i & 3), (uint32_t)(p - 1));
    const int st = (int)min(d, d - (uint32_t)p);
    if (next_run_start(rs, nz, st + 1 == p ? 0 : st + 1) != i) return false;
    const int before = 4 * large_slot(i == 0 ? p - 1 : i - 1), behind = 4 * large_slot(i + 1 == p ? 0 : i + 1);
    int starts = 0;
    for (uint32_t m = nz; m; m &= m - 1) starts += __popc(rs[__ffs(m) - 1]);
    uint32_t diff = 0;
    for (int c = 0; c < nch; ++c) diff |= tabP[behind + c] ^ tabP[before + c];
    for (int c = 0; c < nch; ++c)
        fl[c] = diff ? tabP[behind + c] ^ tabP[before + c] : starts == 2 ? 0u : tabN[behind + c] ^ tabP[before + c];
    return true;
}

// Second part of a large element, in its group: rows, flip planes, delta,
// acceptance and writes.  Every thread of the block.
template <int R, int UB>
__device__ __forceinline__ void bs_large_item(const GomParams &P, const BsItem &I, uint32_t g, uint32_t *sm,
                                              BsLane<FitShared> &L, long long *s_f)
{
    const BsLargeSm S = bs_large_sm(P, sm);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, nwb = blockDim.x >> 5;
    const int W = P.W, Wv = P.Wv, p = P.p, w = lane, s = I.s, nch = (s + 31) >> 5, v0 = 32 * wib;
    const bool kw = w < Wv, mine = wib < nch;
    const int lim = p - 32 * w;
    const uint32_t vm = lim >= 32 ? 0xFFFFFFFFu : lim > 0 ? (1u << lim) - 1u : 0u;
    uint32_t F[32];
    __syncthreads(); // the entries are complete
    if (mine) {
        uint32_t chg = 0, f1 = 0;
#pragma unroll
        for (int r8 = 0; r8 < 32; r8 += 8) {
            int at[8];
            uint32_t xo[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) at[r] = kw && v0 + r8 + r < s ? S.var[v0 + r8 + r] + w : -1;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                xo[r] = at[r] >= 0 ? P.O[at[r]] : 0u;
                chg |= at[r] >= 0 ? xo[r] ^ P.P[at[r]] : 0u;
            }
#pragma unroll
            for (int r = 0; r < 8; ++r) S.sX[32 * (v0 + r8 + r) + lane] = xo[r];
        }
        if (kw) {
            large_planes(S.res1, Wv, wib, w, F);
#pragma unroll
            for (int r = 0; r < 32; ++r) f1 |= F[r] ^ S.sX[32 * (v0 + r) + lane];
        }
        S.f1_c[32 * wib + lane] = f1;
        S.chg_c[32 * wib + lane] = chg;
    }
    __syncthreads();
    const uint32_t f1 = or4(S.f1_c, lane, nch), chg = or4(S.chg_c, lane, nch);
    if (mine) {
        uint32_t hd = 0;
        if (kw) {
            uint32_t t2[32];
            large_planes(S.res2, Wv, wib, w, t2);
#pragma unroll
            for (int r = 0; r < 32; ++r) {
                F[r] = (((f1 & F[r]) | (~f1 & t2[r])) ^ S.sX[32 * (v0 + r) + lane]) & vm;
                hd |= F[r];
            }
        }
        S.hd_c[32 * wib + lane] = hd;
    }
    __syncthreads(); // every entry is read: their slots take the flip planes
    if (mine) {
#pragma unroll
        for (int r = 0; r < 32; ++r) S.sF[32 * (v0 + r) + lane] = kw ? F[r] : 0u;
    }
    __syncthreads();
    if (wib == 0) {
        uint32_t hd = or4(S.hd_c, lane, nch);
        uint32_t cand = kw ? ~f1 & I.rs & chg : 0u;
        while (cand) { // divergent, rare
            const int b = __ffs(cand) - 1;
            cand &= cand - 1;
            uint32_t fl[kLargeChunks];
            if (!large_self_hit(fl, S.tabP, S.tabN, S.rs, I.nz, nch, I.j, 32 * w + b, g, p, P.seed)) continue;
            hd &= ~(1u << b);
            for (int a = 0; a < s; ++a) {
                const uint32_t bit = (fl[a >> 5] >> (a & 31)) & 1u;
                uint32_t *row = S.sF + 32 * a + lane;
                *row = (*row & ~(1u << b)) | (bit << b);
                hd |= bit << b;
            }
        }
        S.hd[lane] = hd;
    }
    __syncthreads();
    uint32_t D[R + 1];
#pragma unroll
    for (int t = 0; t <= R; ++t) D[t] = 0;
    {   // lanes (part, word): the words a population leaves unused take a share of the edges each
        const int parts = 32 / Wv, part = lane / Wv, we = lane - part * Wv;
        bs_edges_add<R, UB>(P, I, [&](int x) { return S.edge[x]; }, part < parts ? I.n_out + I.n_in : 0, wib * parts + part, nwb * parts, we,
                            S.sF + we, S.sX + we, D);
        int off = 1;
        while (off < parts) off <<= 1;
        for (off >>= 1; off > 0; off >>= 1) {
            const bool has = part < off && part + off < parts;
            uint32_t carry = 0;
#pragma unroll
            for (int t = 0; t <= R; ++t) {
                const uint32_t a = D[t], other = __shfl_sync(kFull, a, (lane + off * Wv) & 31), b = has ? other : 0u;
                D[t] = a ^ b ^ carry;
                carry = (a & b) | (a & carry) | (b & carry);
            }
        }
    }
#pragma unroll
    for (int t = 0; t <= R; ++t) S.sD[32 * (wib * (R + 1) + t) + lane] = D[t];
    __syncthreads();
    if (wib == 0) {
        for (int h = 1; h < nwb; ++h) {
            uint32_t carry = 0;
#pragma unroll
            for (int t = 0; t <= R; ++t) {
                const uint32_t a = D[t], b = S.sD[32 * (h * (R + 1) + t) + lane];
                D[t] = a ^ b ^ carry;
                carry = (a & b) | (a & carry) | (b & carry);
            }
        }
        uint32_t nzd = 0;
#pragma unroll
        for (int t = 0; t <= R; ++t) nzd |= D[t];
        const uint32_t hd = S.hd[lane], pos = nzd & ~D[R];
        const uint32_t eqv = kw ? P.eqw[(g & 1) * W + w] : 0u;
        const uint32_t acc = hd & (pos | (~nzd & ~eqv));
        S.acc[lane] = acc;
        L.n_acc += __popc(acc);
        L.n_imp += __popc(acc & pos);
        L.n_dl += __popc(vm & ~hd);
        if (P.fi.on && acc) atomicOr(&P.fi.accw[w], acc);
        if (acc) { // the accepted deltas (>= 0, below 2^R)
            uint32_t x[32];
#pragma unroll
            for (int t = 0; t < 32; ++t) x[t] = t < R ? D[t < R ? t : 0] & acc : 0u;
            planes_add(x, s_f + 32 * w);
        }
    }
    __syncthreads();
    const uint32_t acc = S.acc[lane];
    if (acc)
        for (int a = wib; a < s; a += nwb) {
            const uint32_t m = S.sF[32 * a + lane] & acc;
            if (m) P.O[S.var[a] + w] = S.sX[32 * a + lane] ^ m;
        }
    __syncthreads(); // the region may be rewritten
}

// One colour group by element classes (position t, colour c): the lists
// P.ms_list[P.ms_ptr[5 c + h] .. P.ms_ptr[5 c + h + 1]), h = 0 large, 1 to 3
// at most 32, 16 and 8 variables.  Block b of the (virtual) grid takes the
// large elements b, b + nblk, ...; then, and at once in the other blocks, the
// tiles claim the small items, the larger classes first (without P.dyn they
// take them in a static stride).  Tiles of several warps claim as well: in a
// static stride the blocks with a large element came late to their share of the
// small ones (tree of bound 64 on the 50x50 torus, p = 64: 311 us a generation
// against 208, of bound 100 on a random 6-regular graph of 1,000 vertices, p =
// 512: 1,302 against 778).  The first one of either kind is prepared before
// open().
template <int R, int UB, class Open>
__device__ __forceinline__ bool phase_mix_multi(const GomParams &P, const VGrid &V, const BsMap &M, uint32_t *regions,
                                                int t, int c, uint32_t g, Open open, BsLane<FitShared> &L,
                                                long long *s_f)
{
    const int32_t *cp = P.ms_ptr + 5 * c;
    const int c0 = cp[0], c1 = cp[1], c2 = cp[2], c3 = cp[3], c4 = cp[4], E = M.E, nl = c1 - c0;
    const int n1 = (c2 - c1 + E - 1) / E, n2 = n1 + (c3 - c2 + E - 1) / E, n3 = n2 + (c4 - c3 + E - 1) / E;
    __shared__ int s_claim[kMsThreads / 32]; // per tile of several warps
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, tb = wib / M.nwi;
    const bool dyn = P.dyn, lead = lane == 0 && wib == tb * M.nwi;
    bool first = true;
    BsItem I;
    for (int x = V.blk; x < nl; x += V.nblk) { // block-uniform
        bs_large_prepare(P, P.ms_list[c0 + x], g, regions, I);
        if (first && !open()) return false;
        first = false;
        bs_large_item<R, UB>(P, I, g, regions, L, s_f);
    }
    unsigned claim = 0;
    if (dyn && lead) claim = atomicAdd(&P.work[t], 1u);
    for (int it = M.tile;; it += M.ntiles) {
        if (dyn && M.nwi == 1) {
            it = (int)__shfl_sync(kFull, claim, 0);
        } else if (dyn) { // (read by all before the next is written: an item's first part or the group's end waits)
            if (lead) s_claim[tb] = (int)claim;
            tile_sync(M);
            it = s_claim[tb];
        }
        int cls = 0, k0 = 0, k1 = 0;
        if (it < n1) {
            cls = 32;
            k0 = c1 + it * E;
            k1 = min(k0 + E, c2);
        } else if (it < n2) {
            cls = 16;
            k0 = c2 + (it - n1) * E;
            k1 = min(k0 + E, c3);
        } else if (it < n3) {
            cls = 8;
            k0 = c3 + (it - n2) * E;
            k1 = min(k0 + E, c4);
        }
        if (cls == 8)
            bs_prepare<8, false>(P, M, P.ms_list, k0, k1, g, I);
        else if (cls == 16)
            bs_prepare<16, false>(P, M, P.ms_list, k0, k1, g, I);
        else if (cls == 32)
            bs_prepare<32, false>(P, M, P.ms_list, k0, k1, g, I);
        if (first && !open()) return false;
        first = false;
        if (!cls) return true;
        if (dyn && lead) claim = atomicAdd(&P.work[t], 1u);
        if (cls == 8)
            bs_item<8, R, UB, false>(P, M, I, g, L, s_f, nullptr);
        else if (cls == 16)
            bs_item<16, R, UB, false>(P, M, I, g, L, s_f, nullptr);
        else
            bs_item<32, R, UB, false>(P, M, I, g, L, s_f, nullptr);
    }
}

// Dynamic shared-memory words of a block after the fitness accumulators: the
// warps' fitness planes, then the warps' item regions or a large element's.
__host__ __device__ __forceinline__ int bs_multi_words(int S, int wv, int warps, bool large, int edges)
{
    const int items = warps * (bs_warp_words(S) - 32 * kFitPlanes), big = large ? bs_large_words(wv, warps, edges) : 0;
    return warps * 32 * kFitPlanes + (items > big ? items : big);
}

template <int R, int UB, bool FI = true>
__device__ __forceinline__ void bs_multi_generations(const GomParams &P, const VGrid &V, GomBarrier *bar, int G,
                                                     int64_t target, unsigned long long *s_keys, uint32_t *area,
                                                     long long *s_f, unsigned long long *s_cnt)
{
    uint32_t *regions = area + (blockDim.x >> 5) * 32 * kFitPlanes;
    const BsMap M = bs_map<false>(P, V, regions, P.bs_words - 32 * kFitPlanes); // (the planes stand ahead)
    bs_run<R, false, FI>(P, V, bar, G, target, s_keys, area + threadIdx.x / 32 * 32 * kFitPlanes + (threadIdx.x & 31), M.w,
                     s_f, s_cnt, nullptr, [&](int t, int c, uint32_t g, auto &open, BsLane<FitShared> &L) {
                         return phase_mix_multi<R, UB>(P, V, M, regions, t, c, g, open, L, s_f);
                     });
}

} // namespace
