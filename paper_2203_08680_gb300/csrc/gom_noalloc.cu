// gom_noalloc.cu -- full fitness evaluation of a caller-given population with
// no device allocation at all: the scratch (the population packed into
// 32-individual words) is a fixed array in this file, resident on every GPU
// that loads the library.  For callers that cannot allocate device memory.
#include <cstdint>
#include <mutex>

#include <cuda.h>
#include <cuda_runtime.h>

#include "../../include/gom.h"
#include "gom_rows.cuh"

namespace {

// Scratch: packed population, one 32-bit word per (variable, 32 individuals).
constexpr int64_t kNoAllocWords = GOM_NOALLOC_MAX_WORDS;
static __device__ __align__(256) uint32_t g_noalloc_scratch[kNoAllocWords];

// The scratch array's device address is valid only in the CUDA context it was
// looked up in, so the set-up is cached per context, keyed by the context's
// unique id (never reused within a process, unlike the CUcontext handle or
// the device number: a context made after cudaDeviceReset, or one the caller
// made current itself, gets a new id and a new look-up).
constexpr int kCacheSlots = 64;
struct ScratchSlot {
    unsigned long long ctx_id;
    uint32_t *ptr;
};
std::mutex g_setup_mutex;
ScratchSlot g_slots[kCacheSlots] = {};
int g_nslots = 0;
using CtxGetCurrentFn = CUresult (*)(CUcontext *);
using CtxGetIdFn = CUresult (*)(CUcontext, unsigned long long *);
CtxGetCurrentFn g_ctx_current = nullptr;
CtxGetIdFn g_ctx_id = nullptr;

// Id of the current context.  With none current on this thread, the current
// device's primary context is made current first (cudaSetDevice does that and
// allocates nothing); a context the caller made current is left in place.
cudaError_t current_context_id(unsigned long long *id)
{
    cudaError_t e = cudaSuccess;
    if (!g_ctx_current || !g_ctx_id) {
        cudaDriverEntryPointQueryResult q1{}, q2{};
        void *f1 = nullptr, *f2 = nullptr;
        e = cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1);
        if (e != cudaSuccess || q1 != cudaDriverEntryPointSuccess) return cudaErrorNotSupported;
        e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2);
        if (e != cudaSuccess || q2 != cudaDriverEntryPointSuccess) return cudaErrorNotSupported;
        g_ctx_current = reinterpret_cast<CtxGetCurrentFn>(f1);
        g_ctx_id = reinterpret_cast<CtxGetIdFn>(f2);
    }
    CUcontext ctx = nullptr;
    if (g_ctx_current(&ctx) != CUDA_SUCCESS) return cudaErrorDeviceUninitialized;
    if (!ctx) {
        int dev = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaSetDevice(dev);
        if (e != cudaSuccess) return e;
        if (g_ctx_current(&ctx) != CUDA_SUCCESS || !ctx) return cudaErrorDeviceUninitialized;
    }
    if (g_ctx_id(ctx, id) != CUDA_SUCCESS) return cudaErrorDeviceUninitialized;
    return cudaSuccess;
}

// Device address of the scratch array in the current context: looked up with
// cudaGetSymbolAddress the first time a context calls (the host-side symbol
// is not a device address), then taken from the cache.
cudaError_t scratch_address(uint32_t **out)
{
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    unsigned long long id = 0;
    cudaError_t e = current_context_id(&id);
    if (e != cudaSuccess) return e;
    for (int s = 0; s < g_nslots; ++s)
        if (g_slots[s].ctx_id == id) {
            *out = g_slots[s].ptr;
            return cudaSuccess;
        }
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    // a full cache keeps working: the slot the id hashes to is replaced
    const int s = g_nslots < kCacheSlots ? g_nslots++ : static_cast<int>(id % kCacheSlots);
    g_slots[s] = ScratchSlot{id, static_cast<uint32_t *>(p)};
    *out = static_cast<uint32_t *>(p);
    return cudaSuccess;
}

__global__ void __launch_bounds__(kRowThreads, 4)
    k_noalloc_pack(const uint8_t *pop, int32_t n, int32_t p, int32_t W, uint32_t *words, int64_t *fit)
{
    __shared__ __align__(16) uint32_t sm[row_words(32)];
    pack_rows(pop, n, p, W, words, sm);
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < p; i += blockDim.x) fit[i] = 0; // for the sums that follow
}

__global__ void __launch_bounds__(256, 2)
    k_noalloc_cut(const uint32_t *words, int32_t n, int32_t p, int32_t W, const int64_t *row_ptr, const int32_t *col,
                  const int32_t *wgt, int64_t *fit)
{
    __shared__ long long s_f[1024], s_const;
    cut_sums(words, n, p, W, row_ptr, col, wgt, s_f, &s_const, fit);
}

} // namespace

extern "C" int gom_fitness_noalloc(const int64_t *d_row_ptr, const int32_t *d_col, const int32_t *d_weight,
                                   int32_t num_vertices, const uint8_t *d_pop, int32_t pop,
                                   int64_t *d_fitness_out, void *cuda_stream)
{
    if (!d_row_ptr || !d_col || !d_weight || !d_pop || !d_fitness_out || num_vertices < 1 || pop < 1)
        return GOM_E_ARG;
    if (pop > GOM_MAX_POPULATION) return GOM_E_LIMIT;
    int W = 1;
    while (32 * W < pop) W <<= 1;
    if (static_cast<int64_t>(num_vertices) * W > kNoAllocWords) return GOM_E_LIMIT;
    uint32_t *scratch = nullptr;
    if (scratch_address(&scratch) != cudaSuccess) return GOM_E_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    // eight (four) resident blocks a SM cover a GB300; fewer where the problem is small
    const int64_t tiles = ((num_vertices + kRowVars - 1) / kRowVars / row_tiles(W) + 1) * (W > 8 ? W / 8 : 1);
    k_noalloc_pack<<<static_cast<int>(tiles < 1216 ? tiles : 1216), kRowThreads, 0, s>>>(d_pop, num_vertices, pop, W, scratch,
                                                                                      d_fitness_out);
    if (cudaGetLastError() != cudaSuccess) return GOM_E_CUDA;
    k_noalloc_cut<<<cut_grid(num_vertices, pop, 256, 304), 256, 0, s>>>(scratch, num_vertices, pop, W, d_row_ptr, d_col,
                                                                        d_weight, d_fitness_out);
    if (cudaGetLastError() != cudaSuccess) return GOM_E_CUDA;
    return GOM_OK;
}
