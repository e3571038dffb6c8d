// Device scratch and pinned words that outlive one call.
//
// A call's device memory comes from a stream-ordered pool of this library, one per CUDA context,
// that keeps up to kPoolKeep bytes between calls and gives the rest back at the next
// synchronization: with the default pool (which keeps nothing) or cudaMalloc, a small call spent
// more time getting and returning its memory than on the GPU (165 us of a 190 us evaluation of 64
// points).  The pool is CUDA's own, safe for any threads and streams: a block freed on one stream is
// handed to another only once that is ordered or done.  Pinned words (the host's view of a counter)
// are kept on a short list.  Both are keyed on the context's unique ID, so that a device reset
// starts new ones.
#include <cuda.h>
#include <cuda_runtime.h>

#include <mutex>
#include <vector>

#include "ubqp_internal.cuh"

namespace ubqp {

namespace {

constexpr unsigned long long kPoolKeep = 128ull << 20;
constexpr size_t kPinnedKeep = 16;    // pinned blocks kept
constexpr size_t kPinnedBytes = 64;   // of this size

typedef CUresult (*PFN_ctx_current)(CUcontext*);
typedef CUresult (*PFN_ctx_id)(CUcontext, unsigned long long*);

template <class F>
F driver_fn(const char* name)
{
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion(name, &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return reinterpret_cast<F>(p);
}

std::mutex g_mu;
struct Pool {
    unsigned long long ctx_id;
    cudaMemPool_t pool;
};
std::vector<Pool> g_pools;
struct Pinned {
    unsigned long long ctx_id;
    void* p;
};
std::vector<Pinned> g_pinned;

cudaError_t context_pool(cudaMemPool_t* out)
{
    unsigned long long id = 0;
    cudaError_t e = current_context_id(&id);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(g_mu);
    for (const Pool& q : g_pools)
        if (q.ctx_id == id) {
            *out = q.pool;
            return cudaSuccess;
        }
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    e = cudaGetDevice(&props.location.id);
    cudaMemPool_t pool = nullptr;
    if (e == cudaSuccess) e = cudaMemPoolCreate(&pool, &props);
    if (e != cudaSuccess) return e;
    unsigned long long keep = kPoolKeep;
    e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e != cudaSuccess) {
        cudaMemPoolDestroy(pool);
        return e;
    }
    g_pools.push_back(Pool{id, pool});
    *out = pool;
    return cudaSuccess;
}

}  // namespace

cudaError_t current_context_id(unsigned long long* id)
{
    static PFN_ctx_current ctx_current = driver_fn<PFN_ctx_current>("cuCtxGetCurrent");
    static PFN_ctx_id ctx_id = driver_fn<PFN_ctx_id>("cuCtxGetId");
    if (!ctx_current || !ctx_id) return cudaErrorNotSupported;
    CUcontext ctx = nullptr;
    if (ctx_current(&ctx) == CUDA_SUCCESS && !ctx) {
        // no context current on this thread yet: make the device's primary context current
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaSetDevice(dev);
        if (e != cudaSuccess) return e;
        if (ctx_current(&ctx) != CUDA_SUCCESS) ctx = nullptr;
    }
    if (!ctx || ctx_id(ctx, id) != CUDA_SUCCESS) return cudaErrorDeviceUninitialized;
    return cudaSuccess;
}

cudaError_t work_alloc(void** p, size_t bytes, cudaStream_t s)
{
    cudaMemPool_t pool = nullptr;
    if (context_pool(&pool) != cudaSuccess) {   // no pool here: the default one
        cudaGetLastError();
        return cudaMallocAsync(p, bytes, s);
    }
    cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    if (e == cudaErrorMemoryAllocation) {
        // what the pool keeps may be in pieces too small for this: give it back and try again
        cudaGetLastError();
        cudaStreamSynchronize(s);
        cudaMemPoolTrimTo(pool, 0);
        e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    }
    return e;
}

cudaError_t pinned_get(void** p)
{
    unsigned long long id = 0;
    cudaError_t e = current_context_id(&id);
    if (e != cudaSuccess) return e;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        for (size_t i = 0; i < g_pinned.size(); ++i)
            if (g_pinned[i].ctx_id == id) {
                *p = g_pinned[i].p;
                g_pinned.erase(g_pinned.begin() + (ptrdiff_t)i);
                return cudaSuccess;
            }
    }
    return cudaMallocHost(p, kPinnedBytes);
}

cudaError_t smem_limit(const void* kernel, size_t* bytes)
{
    int dev = 0, blk = 0;
    cudaFuncAttributes fa;
    *bytes = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&blk, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kernel);
    if (e != cudaSuccess) return e;
    if ((size_t)blk > fa.sharedSizeBytes) *bytes = (size_t)blk - fa.sharedSizeBytes;
    return cudaSuccess;
}

cudaError_t open_smem(const void* kernel, size_t need)
{
    size_t most = 0;
    cudaError_t e = smem_limit(kernel, &most);
    if (e != cudaSuccess) return e;
    if (need > most) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

void pinned_put(void* p)
{
    unsigned long long id = 0;
    if (!p) return;
    if (current_context_id(&id) == cudaSuccess) {
        std::lock_guard<std::mutex> lk(g_mu);
        if (g_pinned.size() < kPinnedKeep) {
            g_pinned.push_back(Pinned{id, p});
            return;
        }
    }
    cudaFreeHost(p);
}

}  // namespace ubqp
