// gom_ctx.h -- the context handle behind gom_ctx_t and the CUDA error
// helper, shared by the C ABI's translation units (gom_api.cu, gom_batch.cu).
#pragma once

#include <vector>

#include <cuda_runtime.h>

#include "gom_internal.h"

struct gom_ctx {
    GomParams prm{};
    cudaStream_t stream = nullptr;
    int32_t n = 0, p = 0, W = 0, k = 0;
    int64_t m = 0;
    int sms = 0;
    int grid_mix = 0, grid_fit = 0, grid_start = 0, grid_order = 0, grid_io = 0;
    const void *mix_fn = nullptr; // k_mix instance for this population and FOS
    size_t mix_smem = 0;          // its dynamic shared memory per block
    int mix_threads = kMixThreads; // its block size (fewer warps for very large elements)
    int run_threads = kMixThreads; // the persistent kernel's
    const void *run_fn = nullptr; // persistent generation kernel (same instance parameters)
    size_t run_smem = 0;          // its dynamic shared memory (staging or the k group keys)
    int grid_run = 0;             // its grid: co-resident blocks only
    bool can_persist = false;     // cooperative launch available and the sizes fit
    bool persistent = false;      // current path: k_run (true) or the per-generation graph
    // the bit-sliced mixing path (gom_bs.cu), where the FOS and weights allow it
    bool bs_can = false;          // available for this context
    bool bs_ok = false;           // and the learned filter runs on it (elements of at most 32 variables, 8-bit weights)
    bool bs_on = false;           // selected (GOM_OPT_BITSLICED)
    bool bs_one = true;           // the one-class kernels pay (bs_one_class_pays)
    bool bs_learn = false;        // the learned filter's do (bs_learn_pays)
    bool bs_fi = true;            // the persistent one does with Forced Improvement on: not with one-word populations
                                  //   in groups of at most 1,024, whose FI steps are most of the time and want the
                                  //   per-lane kernel's grid (random 6-regular 4,000, p = 32, generation 40: 672 us
                                  //   per lane, 773; 2D torus 300, p = 32 197, 94)
    int bs_set = -1;              // GOM_OPT_BITSLICED as the caller set it (-1: never set; batched launches
                                  //   then choose by the instance's share of warps)
    const void *run_bs_fn = nullptr, *mix_bs_fn = nullptr; // the instances for the learned filter's mode
    int bs_r = 0, bs_ub = 0;      // their accumulator and weight widths (elements above 32 variables have none)
    size_t bs_smem = 0;           // dynamic shared memory of both (warp regions, group keys)
    int bs_threads = 0;           // their block size
    int bs_grid_run = 0, bs_grid_mix = 0;
    // the bit-sliced path by element classes (gom_bs_multi.cu): linkage models of mixed sizes, elements above 32
    // variables included, where run_ms_fn is set; persistent path only, without the learned filter
    const void *run_ms_fn = nullptr;
    size_t ms_smem = 0;
    int ms_grid = 0, ms_ub = 0;
    int64_t ms_edges = 0;        // most edges of an element of at most 32 variables
    // Forced Improvement (GOM_OPT_FORCED_IMPROVEMENT)
    bool fi_ok = false;           // available: |w| <= 255, element sums of |w| below 2^16
    int fi_r = 16;                // bit-plane width of its accumulators
    int fi_grid = 0;              // grid of its per-group kernel on the per-launch path
    unsigned long long *trace_buf = nullptr; // workspace slot of the phase trace
    size_t order_smem = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaGraph_t tgraph = nullptr; // variant with event records around each mixing launch
    cudaGraphExec_t texec = nullptr;
    std::vector<cudaEvent_t> events;
    bool timing = false;
    bool timing_pending = false; // the events hold a generation not yet added to mix_ms
    double mix_ms = 0.0;
    int64_t timing_g0 = 0;       // generation counter when timing was (re)started
    int last_cuda = 0;
    // for batched launches (gom_batch_*)
    int wpi = 1;                 // words per mixing item
    int32_t variant = kVarNarrow; // kernel variant (mask and delta widths)
    int64_t max_items = 1;       // mixing items of the largest colour group
    double sum_se = 0.0;         // sum over elements of (variables + edges)
    int64_t max_group = 1;       // elements of the largest colour group
    int64_t max_s = 0;           // variables of the largest element
    int64_t max_edges = 0;       // most edges of one element
    std::vector<int32_t> celems; // element index at each colour-order position
    char *filter_base = nullptr; // learned-filter workspace (gom_filter_attach), or null
    int64_t filter_cap = 0;      // its training-log capacity
    char *base = nullptr;        // the workspace
    size_t state_bytes = 0;      // its state arrays: [0, state_bytes) (population, fitness, elitist, ...)
};


// The bit-sliced path runs the context's generations: by element class where
// the model has that (persistent, without the learned filter), else in one
// class.  The per-generation graph and the learned filter have their own
// defaults, where the caller has not set the option (use_bs_one: the graph's
// kernels, and with the filter the persistent one too).
inline bool use_ms(const gom_ctx *ctx) { return ctx->bs_on && ctx->run_ms_fn && !ctx->prm.learn; }
inline bool use_bs_one(const gom_ctx *ctx)
{
    const bool learn = ctx->prm.learn != 0, dflt = learn ? ctx->bs_learn : ctx->bs_on && ctx->bs_one;
    return ctx->run_bs_fn && (ctx->bs_ok || !learn) && (ctx->bs_set >= 0 ? ctx->bs_set == 1 : dflt);
}
inline bool use_bs_run(const gom_ctx *ctx)
{
    if (ctx->prm.learn) return use_bs_one(ctx);
    return ctx->bs_on && ctx->run_bs_fn && (!ctx->prm.fi.on || ctx->bs_fi || ctx->bs_set == 1);
}

// Weight and sum widths of the bit-sliced instances for |w| <= max_w and
// element sums of |w| <= max_abs_w; false where there is none.
inline bool bs_planes(int64_t max_w, int64_t max_abs_w, int *r, int *ub)
{
    static constexpr int kPlanes[4][2] = {{12, 8}, {16, 8}, {16, 12}, {20, 16}};
    for (const auto &c : kPlanes)
        if (max_abs_w < (int64_t(1) << c[0]) && max_w < (int64_t(1) << c[1])) {
            *r = c[0];
            *ub = c[1];
            return true;
        }
    return false;
}

inline int cuda_fail(gom_ctx *ctx, cudaError_t e)
{
    if (ctx) ctx->last_cuda = static_cast<int>(e);
    return GOM_E_CUDA;
}

// One staging slice (one mixing item) in shared memory -- the one definition
// of its layout; the kernels take these offsets (32-bit words): an 8-word
// item header, the element's variables, their outside-edge starts (s+1),
// their outside weight sums (int64), the rows of P on the element (W words
// each), the pattern table (32 W masks of 4, 8 or 16 bytes), its run starts (W
// words), each edge's {code, weight} (two words), each outside edge's parent
// words (WPI words), and in stage-all mode the item's donor start positions
// (one int per individual of its words).  Every offset is a multiple of 4
// words.
struct SliceLayout {
    int64_t off_fv, off_seg, off_wout, off_pr, off_pat, off_rs, off_cw, off_xw, off_ds;
    int64_t base_words; // a slice without the donor starts
    int64_t all_words;  // with them (stage-all mode)
};

inline SliceLayout slice_layout(int64_t max_s, int64_t max_edges, int W, int wpi, int32_t variant, bool split,
                                int nwg)
{
    auto round4 = [](int64_t x) { return (x + 3) & ~int64_t(3); };
    SliceLayout L{};
    L.off_fv = 8;
    L.off_seg = L.off_fv + round4(max_s);
    L.off_wout = L.off_seg + round4(max_s + 1);
    L.off_pr = L.off_wout + round4(2 * max_s);
    L.off_pat = L.off_pr + round4(max_s * W);
    L.off_rs = L.off_pat + int64_t(32) * W * (variant == kVarNarrow ? 1 : variant == kVarWide ? 2 : 4);
    L.off_cw = L.off_rs + round4(W);
    L.off_xw = L.off_cw + round4(2 * max_edges);
    L.off_ds = L.off_xw + round4(max_edges * wpi);
    L.base_words = L.off_ds;
    L.all_words = L.off_ds + int64_t(32) * wpi * (split ? 1 : nwg);
    return L;
}

// Words per item and split mode for p individuals when `warps` warps share
// the items of the largest colour group of `max_group` elements: one warp per
// element walking all its words in groups of min(W, 4) words, or, with fewer
// than about 4 elements per warp, one warp per (element, word group) so that
// the warps stay busy (then single words if the population has only one
// group of min(W, 4) words).  The kernel variant for elements of more than
// 64 variables has instances for groups of at most 2 words.
inline void item_split(int W, int32_t p, int64_t max_group, int64_t warps, int32_t variant, int *wpi, int *split)
{
    const int wv = (p + 31) / 32;
    const int most = variant == kVarHuge ? 2 : 4;
    *wpi = W < most ? W : most;
    *split = 0;
    if (max_group < 4 * warps && wv > 1) {
        *split = 1;
        if ((wv + *wpi - 1) / *wpi == 1) *wpi = 1;
    }
}

// Lanes per pair (2^lsh) and warps per tile of the bit-sliced path for a
// largest colour group of `max_group` elements of `wv` words on `warps` warps
// in blocks of `wpb`: the most lanes for which the group's tiles still fit the
// warps at once and every lane has four edges to add.  A group of few elements
// is bound by the latency of one item, and that is mostly its serial edges.
inline void bs_split(int wv, int64_t max_group, int64_t max_edges, int64_t warps, int wpb, int *lsh, int *nwi)
{
    *lsh = 0;
    *nwi = 1;
    for (int l = 1; l <= 5 && (int64_t(4) << (l - 1)) < max_edges; ++l) {
        int nw = 1;
        while (32 * nw < wv << l) nw *= 2;
        if (nw > wpb || wpb % nw) return;
        const int64_t E = nw > 1 ? 1 : (32 >> l) / wv;
        if ((max_group + E - 1) / E * nw > warps) return;
        *lsh = l;
        *nwi = nw;
    }
}

// What the choice between the two mixing paths goes by: population words of an
// element, elements of the largest colour group, variables and edges of the
// largest element, weight bits of the bit-plane instances, the colour groups
// and those of them that hold an element above 16 variables, whether half of
// the elements have at most 8 variables and the largest more (linkage trees),
// whether the per-lane path stages all groups at once, and its resident warps.
struct MixShape {
    int64_t wv, max_group, max_s, max_edges;
    int ub;
    int64_t groups, headed;
    bool mixed, stage_all;
    int64_t lane_warps;
};

// Whether the bit-sliced path is the faster one where both are available: its
// persistent kernels, over tori, random regular graphs of degree 3 to 12 and
// their linkage trees of bounds 2 to 128, p = 2 to 1,024 (figures: microseconds
// per generation, per lane / bit-sliced).
// - Up to 16 variables it is, from small groups on (2D torus 100, p = 256 111 /
//   70; 3D torus 50, p = 128 1046 / 312; random 12-regular 60,000, p = 512
//   5459 / 3372), unless the per-lane path has staged every group: then at one
//   word (2D torus 75, p = 32 73 / 75; singletons 23 / 30), in groups of at most
//   1,024 words (2D torus 10, p = 32 45 / 59), and up to six words where the
//   groups have few edges (singletons of the 50x50 torus, p = 64 15 / 19, 4 edges
//   times 2,500 words; of a random 10-regular graph of 3,000, p = 128 48 / 43).
//   Linkage trees in the class of 16 (bounds 14 to 16): up to four words, in all
//   but small groups five, only from one and a half waves of per-lane warps on
//   (bound 14, random 6-regular 4,000, p = 128 170 / 232; 75x75 torus, p = 160
//   153 / 171; 100x100 torus, p = 128 255 / 182).
// - Above 64 variables it is (a block takes a large element; tree of bound 70,
//   50x50 torus, p = 64 296 / 213; random 5-regular 40,000, p = 64 1408 / 1120).
// - From 17 to 64 variables its tables are at their widest, and one block of
//   eight warps fills an SM.  Up to four words the per-lane path splits elements
//   by word and wins while those items fit one wave of its warps (tree of bound
//   24, 50x50 torus, p = 64 121 / 140; 150x150, p = 64 236 / 169; at three and four
//   words three quarters of a wave: bound 30, 75x75, p = 128 180 / 171), and
//   where most groups hold an element above 16 variables (bound 40, random
//   5-regular 40,000, p = 64 618 / 749).  Above four words its items take four
//   words each and bit-planes win (bound 30, 50x50, p = 256 211 / 168), but not in groups
//   of at most 512 words (bound 30, random 3-regular 300, p = 256 161 / 173), nor
//   with 16-bit weights, whose adders are twice as long, up to 32 variables and
//   12 words in one wave (bound 24, 50x50, p = 160 283 / 304).
inline bool bs_pays(const MixShape &m)
{
    const int64_t words = m.max_group * m.wv;
    if (m.stage_all && (m.wv == 1 || words <= 1024 || (m.wv <= 6 && words * m.max_edges <= 19000))) return false;
    if (m.max_s <= 16 && m.max_s > 13 && m.mixed && (m.wv <= 4 || (m.wv == 5 && 2 * words > m.lane_warps)))
        return 2 * words > 3 * m.lane_warps;
    if (m.max_s <= 16 || m.max_s > 64) return true;
    if (m.wv <= 4) return words > m.lane_warps * (m.wv <= 2 ? 4 : 3) / 4 && 5 * m.headed <= 3 * m.groups;
    return words > 512 && !(m.ub > 8 && m.max_s <= 32 && m.wv <= 12 && words <= m.lane_warps);
}

// The same for the per-generation graph's kernels, which take all elements in
// the largest one's class.  In linkage trees, where that class is wide and most
// elements are small, per lane is the faster up to five words for 9 to 16
// variables (bound 12, 150x150 torus, p = 32 153 / 190; bound 14, 75x75, p = 160
// 177 / 211) and up to 15 words above (bound 30, 50x50, p = 64 158 / 275, p = 256
// 249 / 293, p = 512 as fast).
inline bool bs_one_class_pays(const MixShape &m)
{
    if (!m.mixed) return true;
    return m.max_s <= 16 ? m.wv > 5 || 2 * m.max_group * m.wv > 3 * m.lane_warps : m.wv > 15;
}

// The same for the learned filter's kernels, whose bookkeeping takes one lane
// per pair and whole warps: rows of at most 16 words, and items for at least a
// quarter of 20 warps per SM (random 10-regular 3,000, p = 32 1,634 / 4,824; random
// 16-regular 20,000, p = 1,024 19.3 / 29.6 ms).
inline bool bs_learn_pays(int64_t W, int64_t max_group, int64_t sms)
{
    const int64_t E = 32 / W;
    return W <= 16 && 4 * ((max_group + E - 1) / E) >= 20 * sms;
}

// Raises a kernel's dynamic shared memory limit to at least `bytes`, never
// lowers it: kernel instances are shared by every context (and batch), and a
// limit lowered below what an existing context launches with would make its
// launches fail.
inline cudaError_t raise_smem_limit(const void *fn, size_t bytes)
{
    cudaFuncAttributes fa{};
    cudaError_t e = cudaFuncGetAttributes(&fa, fn);
    if (e != cudaSuccess) return e;
    if (static_cast<size_t>(fa.maxDynamicSharedSizeBytes) >= bytes) return cudaSuccess;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
}

#define GOM_CUDA(ctx, call)                               \
    do {                                                  \
        cudaError_t e_ = (call);                          \
        if (e_ != cudaSuccess) return cuda_fail(ctx, e_); \
    } while (0)

// The counters of the generations of the context's last call into
// host_stats[0..num) (may be null) and their number (*run_out).  Waits for
// the stream.  GOM_E_TIMEOUT if the context's device error word is set.
int ctx_read_stats(gom_ctx *ctx, int32_t num, gom_gen_stats_t *host_stats, int32_t *run_out);

// gom_batch_create with the generations each instance makes for one of the
// others' (weights, or null: the same number), for the block shares.
int batch_create(gom_ctx_t *const *ctxs, int32_t num, const gom_batch_config_t *cfg, const double *weights,
                 void *d_workspace, size_t ws_bytes, void *cuda_stream, gom_batch_t **out);

// Rebuilds the per-generation graphs after a change of the parameters they
// copy (the timed variant only if it exists).  Waits for the stream.
int rebuild_graphs(gom_ctx *ctx);
