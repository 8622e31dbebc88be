// gom_rows.cuh -- the population between its two layouts, and its full
// evaluation: uint8 rows [individual][variable] packed into bit-sliced words
// [variable][word] and back, and the cut weights of a bit-sliced population
// (Sec. 6.2).  Shared by the handle's kernels (gom_kernels.cu) and the
// handle-less evaluation (gom_noalloc.cu).  Anonymous namespace: each
// translation unit that includes it compiles its own copy.
#pragma once

#include <cuda_runtime.h>

#include "gom_bitplane.cuh"

namespace {

// ---- rows <-> words.  Bound by memory: a warp moves 128 variables of 32
// individuals (one word column) with 4 bytes a lane and row, and the block
// turns the words of 128 variables through shared memory, so that both sides
// are read and written in whole lines.  torus1000, p = 256: import 709 -> 92
// us, export 600 -> 78 us (256 MB of rows; one byte a lane and row before).
constexpr int kRowVars = 128;
constexpr int kRowThreads = 256;

// Tiles of kRowVars variables a block takes at once: one per W warps.
__host__ __device__ constexpr int row_tiles(int W) { return W < kRowThreads / 32 ? kRowThreads / 32 / W : 1; }
// Words of the block's staging: [W][tile variables + 4] (the padding keeps
// both the 4-word columns and the W-word rows spread over the banks).
__host__ __device__ constexpr int row_stride(int W) { return row_tiles(W) * kRowVars + 4; }
__host__ __device__ constexpr int row_words(int W) { return W * row_stride(W); }

// Four bytes at `at` (any alignment) inside [base, end); bytes outside are 0.
__device__ __forceinline__ uint32_t load4(const uint8_t *at, const uint8_t *base, const uint8_t *end)
{
    const uintptr_t a = reinterpret_cast<uintptr_t>(at);
    const uint8_t *lo = reinterpret_cast<const uint8_t *>(a & ~uintptr_t(3));
    const unsigned m = (unsigned)(a & 3);
    if (lo >= base && lo + (m ? 8 : 4) <= end) { // whole words inside the buffer
        const uint32_t x = __ldg(reinterpret_cast<const uint32_t *>(lo));
        if (!m) return x;
        return __funnelshift_r(x, __ldg(reinterpret_cast<const uint32_t *>(lo) + 1), 8 * m);
    }
    uint32_t x = 0;
    for (int c = 0; c < 4; ++c)
        if (at + c >= base && at + c < end) x |= (uint32_t)__ldg(at + c) << (8 * c);
    return x;
}

// The 4 x 4 byte transpose of four words.
__device__ __forceinline__ void transpose_bytes(uint32_t (&x)[4])
{
    const uint32_t l0 = __byte_perm(x[0], x[1], 0x5140), h0 = __byte_perm(x[0], x[1], 0x7362);
    const uint32_t l1 = __byte_perm(x[2], x[3], 0x5140), h1 = __byte_perm(x[2], x[3], 0x7362);
    x[0] = __byte_perm(l0, l1, 0x5410);
    x[1] = __byte_perm(l0, l1, 0x7632);
    x[2] = __byte_perm(h0, h1, 0x5410);
    x[3] = __byte_perm(h0, h1, 0x7632);
}

// Whether the export goes one byte a thread: rows in whole lines take a block a
// tile of 128 variables, which has its word columns of 32 rows one after another (11
// us for up to 8 words, twice as long for 16, 1.7 times for rows that are not
// word-aligned), and a small population has few tiles.  One byte a thread takes 6 us and 4 a
// MB: n = 1,089, p = 1,024 12 us against 48, n = 100, p = 256 6 / 11, n = 10,000, p =
// 256 14 / 11.
inline bool export_small(int64_t n, int p, int W, const void *out)
{
    const bool aligned = !(n & 3) && !(reinterpret_cast<uintptr_t>(out) & 3);
    return n * p <= (int64_t)(aligned ? 1400000 : 2800000) * (W <= 8 ? 1 : W / 8);
}

// Packs rows in[p][n] (any non-zero byte is a 1) into words[n][W]; bits of
// individuals past p are zero.  Called by every thread of the grid's blocks
// (kRowThreads each); sm: row_words(W) words.  Above 8 words, where the tiles
// alone leave blocks idle, a block takes 8 words of a tile (evaluation of n = 25,
// p = 1,024, rows off the 4-byte words: 46 -> 27 us).
__device__ __forceinline__ void pack_rows(const uint8_t *in, int n, int p, int W, uint32_t *words, uint32_t *sm)
{
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int T = row_tiles(W), stride = row_stride(W), lw = __ffs(W) - 1;
    const uint8_t *end = in + (int64_t)p * n;
    const bool aligned = !(n & 3) && !(reinterpret_cast<uintptr_t>(in) & 3); // then no word passes a row's end
    const int64_t tiles = (n + kRowVars - 1) / kRowVars;
    // a block's words: lc = log2 of their number, lp = log2 of the parts of a tile (T = 1 where there are several)
    const int lc = lw > 3 && tiles < gridDim.x ? 3 : lw, lp = lw - lc, C = 1 << lc;
    for (int64_t u = blockIdx.x; (u >> lp) * T < tiles; u += gridDim.x) {
        const int64_t t0 = (u >> lp) * T;
        const int w0 = (int)(u & ((1 << lp) - 1)) << lc;
        for (int task = wib; task < T << lc; task += kRowThreads / 32) {
            const int c = task & (C - 1), w = w0 + c, lt = task >> lc; // a word of a local tile
            const int64_t v = (t0 + lt) * kRowVars + 4 * lane;
            const int rows = min(32, p - 32 * w);
            uint32_t acc[4] = {0, 0, 0, 0}; // byte c of acc[k]: individuals 8k .. 8k + 7 of variable v + c
            if (v < n) {
                const uint32_t valid = n - v >= 4 ? 0x01010101u : 0x01010101u >> (8 * (4 - (int)(n - v)));
                const uint8_t *at = in + 32 * (int64_t)w * n + v;
#pragma unroll
                for (int k = 0; k < 4; k += 2) { // 16 rows' loads in flight
                    uint32_t x[16];
                    if (aligned) {
#pragma unroll
                        for (int b = 0; b < 16; ++b)
                            x[b] = 8 * k + b < rows ? __ldg(reinterpret_cast<const uint32_t *>(at + (int64_t)(8 * k + b) * n)) : 0u;
                    } else {
#pragma unroll
                        for (int b = 0; b < 16; ++b) x[b] = 8 * k + b < rows ? load4(at + (int64_t)(8 * k + b) * n, in, end) : 0u;
                    }
#pragma unroll
                    for (int b = 0; b < 16; ++b) { // bit 7 of a byte: the byte is not zero
                        const uint32_t nz = (((x[b] & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x[b]) >> 7;
                        acc[k + (b >> 3)] |= (nz & valid) << (b & 7);
                    }
                }
            }
            transpose_bytes(acc);
            *reinterpret_cast<uint4 *>(sm + c * stride + lt * kRowVars + 4 * lane) =
                make_uint4(acc[0], acc[1], acc[2], acc[3]);
        }
        __syncthreads();
        const int64_t first = t0 * kRowVars * W + w0, total = min((int64_t)T * kRowVars, n - t0 * kRowVars) << lc;
        for (int x = threadIdx.x; x < total; x += kRowThreads)
            words[first + ((int64_t)(x >> lc) << lw) + (x & (C - 1))] = sm[(x & (C - 1)) * stride + (x >> lc)];
        __syncthreads();
    }
}

// Unpacks words[n][W] into rows out[p][n] of {0, 1}.
__device__ __forceinline__ void unpack_rows(const uint32_t *words, int n, int p, int W, uint8_t *out, uint32_t *sm)
{
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int T = row_tiles(W), stride = row_stride(W), lw = __ffs(W) - 1;
    const int64_t tiles = (n + kRowVars - 1) / kRowVars;
    for (int64_t t0 = (int64_t)blockIdx.x * T; t0 < tiles; t0 += (int64_t)gridDim.x * T) {
        const int64_t first = t0 * kRowVars * W, total = min((int64_t)T * kRowVars, n - t0 * kRowVars) * W;
        for (int x = threadIdx.x; x < T * kRowVars * W; x += kRowThreads)
            sm[(x & (W - 1)) * stride + (x >> lw)] = x < total ? words[first + x] : 0u;
        __syncthreads();
        for (int task = wib; task < T * W; task += kRowThreads / 32) {
            const int w = task & (W - 1), lt = task >> lw;
            const int64_t v0 = (t0 + lt) * kRowVars;
            const int rows = min(32, p - 32 * w), vars = (int)min((int64_t)kRowVars, n - v0);
            if (vars <= 0) continue;
            const uint4 q = *reinterpret_cast<const uint4 *>(sm + w * stride + lt * kRowVars + 4 * lane);
            uint32_t acc[4] = {q.x, q.y, q.z, q.w};
            transpose_bytes(acc); // byte c of acc[k]: individuals 8k .. 8k + 7 of variable v0 + 4 lane + c
#pragma unroll
            for (int b = 0; b < 32; ++b) {
                if (b >= rows) break;
                const uint32_t x = (acc[b >> 3] >> (b & 7)) & 0x01010101u;
                uint8_t *row = out + (32 * (int64_t)w + b) * n + v0;
                const unsigned m = (unsigned)(reinterpret_cast<uintptr_t>(row) & 3); // the same in every lane
                const int at = 4 * lane;
                if (m == 0) {
                    if (at + 4 <= vars) {
                        *reinterpret_cast<uint32_t *>(row + at) = x;
                    } else {
                        for (int c = 0; at + c < vars; ++c) row[at + c] = (uint8_t)(x >> (8 * c));
                    }
                } else {
                    // whole words start 4 - m bytes into the row: lane l stores the bytes 4 l - m .. 4 l + 3 - m
                    // of the tile, the first m of them from the lane before
                    const uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, x, 1);
                    const uint32_t y = __funnelshift_l(prev, x, 8 * m);
                    const int a0 = at - (int)m;
                    if (lane > 0 && a0 + 4 <= vars) {
                        *reinterpret_cast<uint32_t *>(row + a0) = y;
                    } else {
                        for (int c = lane > 0 ? 0 : (int)m; c < 4; ++c)
                            if (a0 + c < vars) row[a0 + c] = (uint8_t)(y >> (8 * c));
                    }
                    if (lane == 31) // the tile's last m bytes
                        for (int c = 4 - (int)m; c < 4; ++c)
                            if (at + c < vars) row[at + c] = (uint8_t)(x >> (8 * c));
                }
            }
        }
        __syncthreads();
    }
}

// ---- full evaluation: f[i] = sum over edges {u < v} of w_uv [x_u != x_v].
// On bit-planes: a lane takes one word (32 individuals) of one vertex at a
// time and adds four edges' weights at once in carry chains, about 35
// instructions for an edge of 32 lanes x 32 individuals, where one lane per
// individual took about 12 for 32.  Weights go in bytes: a pass over the
// edges per byte that any weight has (the first for |w| < 256).  A negative
// weight counts where the edge is not cut, less |w| for everyone.
// 1000x1000 torus, p = 256: 1638 -> 155 us; 200,000 vertices of degree 6, p =
// 512: 918 -> 119 us.
constexpr int kCutPlanes = 24;
constexpr int kCutFlush = 500; // four-edge steps: 500 * 4 * 255 * 32 slots < 2^24

// acc += sum over four edges of u d (u: a byte in y's bits sh .. sh + 7).
__device__ __forceinline__ void add_bytes4(uint32_t (&acc)[kCutPlanes], const uint32_t (&d)[4], const uint32_t (&u)[4])
{
    uint32_t A[2][9];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        uint32_t carry = 0;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const uint32_t i0 = bit_mask(d[2 * h], u[2 * h], t), i1 = bit_mask(d[2 * h + 1], u[2 * h + 1], t);
            A[h][t] = i0 ^ i1 ^ carry;
            carry = (i0 & i1) | (i0 & carry) | (i1 & carry);
        }
        A[h][8] = carry;
    }
    uint32_t S[10], carry = 0;
#pragma unroll
    for (int t = 0; t < 9; ++t) {
        S[t] = A[0][t] ^ A[1][t] ^ carry;
        carry = (A[0][t] & A[1][t]) | (A[0][t] & carry) | (A[1][t] & carry);
    }
    S[9] = carry;
    carry = 0;
#pragma unroll
    for (int t = 0; t < 10; ++t) {
        const uint32_t a = acc[t];
        acc[t] = a ^ S[t] ^ carry;
        carry = (a & S[t]) | (a & carry) | (S[t] & carry);
    }
#pragma unroll
    for (int t4 = 10; t4 < kCutPlanes; t4 += 7) { // rarely past the first planes
        if (!carry) return;
#pragma unroll
        for (int t = t4; t < t4 + 7; ++t) {
            const uint32_t a = acc[t];
            acc[t] = a ^ carry;
            carry &= a;
        }
    }
}

// Adds a warp's planes (lane = slot Wv + word) into s_f[32 word + b], times
// 2^shift, and clears them: the slots' planes added in a tree, then the sums
// of slot 0's lanes turned into numbers.  Warp-wide.
__device__ __forceinline__ void cut_flush(uint32_t (&acc)[kCutPlanes], int Wv, int slot, int w, int E, int shift, long long *s_f)
{
    const int lane = threadIdx.x & 31;
    int off = 1;
    while (off < E) off <<= 1;
    for (off >>= 1; off > 0; off >>= 1) {
        const bool has = slot < off && slot + off < E;
        uint32_t carry = 0;
#pragma unroll
        for (int t = 0; t < kCutPlanes; ++t) {
            const uint32_t a = acc[t];
            uint32_t b = __shfl_sync(0xFFFFFFFFu, a, (lane + off * Wv) & 31);
            b = has ? b : 0u;
            acc[t] = a ^ b ^ carry;
            carry = (a & b) | (a & carry) | (b & carry);
        }
    }
    if (slot == 0 && w < Wv) {
        uint32_t x[32];
#pragma unroll
        for (int t = 0; t < 32; ++t) x[t] = t < kCutPlanes ? acc[t] : 0u;
        transpose_lane<32>(x);
#pragma unroll
        for (int b = 0; b < 32; ++b)
            if (x[b])
                atomicAdd(reinterpret_cast<unsigned long long *>(&s_f[32 * w + b]), (unsigned long long)x[b] << shift);
    }
#pragma unroll
    for (int t = 0; t < kCutPlanes; ++t) acc[t] = 0;
}

// The cut weights of words[n][W] (Wv words in use, p individuals) added into
// out[p].  Called by every thread of the grid's blocks; s_f: the block's 32 W
// accumulators, s_const: one more.
__device__ __forceinline__ void cut_sums(const uint32_t *words, int n, int p, int W, const int64_t *row_ptr,
                                         const int32_t *col, const int32_t *wgt, long long *s_f, long long *s_const,
                                         int64_t *out)
{
    const int lane = threadIdx.x & 31;
    const int Wv = (p + 31) / 32, E = 32 / Wv;
    const int slot = lane / Wv, w = lane - slot * Wv;
    const bool in = slot < E;
    const int64_t gwarp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int q = threadIdx.x; q < 32 * Wv; q += blockDim.x) s_f[q] = 0;
    if (threadIdx.x == 0) *s_const = 0;
    __syncthreads();
    uint32_t acc[kCutPlanes];
#pragma unroll
    for (int t = 0; t < kCutPlanes; ++t) acc[t] = 0;
    uint32_t all = 0; // the bits any |w| of this warp has
    long long neg_sum = 0;
    for (int byte = 0; byte < 4; ++byte) {
        if (byte > 0 && !(all >> (8 * byte))) break;
        int steps = 0;
        // one vertex a slot; the next one's row bounds and the next four edges
        // are on their way while four edges' words arrive and are added
        int64_t u = gwarp * E + slot, e, end;
        int v[4], wt[4];
        const auto row = [&](int64_t x, int64_t *from, int64_t *to) {
            const bool have = in && x < n;
            *from = have ? __ldg(row_ptr + x) : 0;
            *to = have ? __ldg(row_ptr + x + 1) : 0;
        };
        const auto edges = [&](int64_t from, int64_t to) {
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                v[x] = from + x < to ? __ldg(col + from + x) : -1;
                wt[x] = from + x < to ? __ldg(wgt + from + x) : 0;
            }
        };
        row(u, &e, &end);
        edges(e, end);
        for (int64_t u0 = gwarp * E; u0 < n; u0 += nwarps * E) {
            int64_t e2, end2;
            row(u + nwarps * E, &e2, &end2);
            const uint32_t xu = in && u < n ? words[u * W + w] : 0u;
            for (bool more = true; more;) {
                uint32_t d[4], mag[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) d[x] = v[x] > u ? words[(int64_t)v[x] * W + w] : 0u; // each edge once
                uint32_t neg[4];
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    neg[x] = (uint32_t)(wt[x] >> 31);
                    mag[x] = v[x] > u ? ((uint32_t)wt[x] ^ neg[x]) - neg[x] : 0u;
                    if (byte == 0) {
                        all |= mag[x];
                        if (neg[x] && v[x] > u && w == 0) neg_sum += wt[x];
                    }
                    mag[x] >>= 8 * byte;
                }
                e += 4;
                more = __any_sync(0xFFFFFFFFu, e < end);
                edges(more ? e : e2, more ? end : end2);
#pragma unroll
                for (int x = 0; x < 4; ++x) d[x] ^= xu ^ neg[x];
                add_bytes4(acc, d, mag);
                if (++steps == kCutFlush) {
                    cut_flush(acc, Wv, slot, in ? w : Wv, E, 8 * byte, s_f);
                    steps = 0;
                }
            }
            u += nwarps * E;
            e = e2;
            end = end2;
        }
        if (byte == 0) all = __reduce_or_sync(0xFFFFFFFFu, all);
        cut_flush(acc, Wv, slot, in ? w : Wv, E, 8 * byte, s_f);
    }
    if (neg_sum) atomicAdd(reinterpret_cast<unsigned long long *>(s_const), (unsigned long long)neg_sum);
    __syncthreads();
    const long long c = *s_const;
    for (int i = threadIdx.x; i < p; i += blockDim.x)
        if (s_f[i] + c) atomicAdd(reinterpret_cast<unsigned long long *>(&out[i]), (unsigned long long)(s_f[i] + c));
}

// Blocks of `threads` for cut_sums: a warp per E vertices, at most `most`.
inline int cut_grid(int64_t n, int p, int threads, int most)
{
    const int64_t E = 32 / ((p + 31) / 32), warps = (n + E - 1) / E, blocks = (32 * warps + threads - 1) / threads;
    return static_cast<int>(blocks < 1 ? 1 : blocks > most ? most : blocks);
}

} // namespace
