// ubqp_penalized_eval_noalloc: the penalized objective and its gradient for callers that
// must not allocate device memory.  Some callers manage every byte of device memory
// through their own pool or a fixed budget and may not call cudaMalloc/cudaFree (which
// can also synchronize the whole device); this entry point gives them the same
// computation as ubqp_penalized_eval, with the same kernel and the same tiles, with its scratch
// in a fixed static device array.
//
// The scratch (the row tiles' shares of h) lives in g_noalloc_scratch below.  Every GPU that loads
// the library holds it until the process exits.  All calls share it and it keeps the last call's
// contents; each call writes every word it later reads, so nothing has to start at zero.  Calls
// that overlap on the GPU (other streams, other host threads) race on it.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstring>
#include <mutex>

#include "../../include/ubqp.h"
#include "ubqp_internal.cuh"

namespace ubqp {

constexpr int kNoallocMaxLanes = 256;
constexpr int kNoallocMaxItems = 16384;
constexpr size_t kScratchBytes = UBQP_NOALLOC_SCRATCH_BYTES;
// the limits below admit at most kNoallocMaxItems blocks of 256 rows, i.e. this many tiles of 32
static_assert(((size_t)kNoallocMaxItems * 8 + kNoallocMaxLanes) * sizeof(double) <= kScratchBytes, "shares of h fit");

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

// Device address of g_noalloc_scratch in each CUDA context that has used this entry point.
// The key is the context's unique ID (current_context_id), not the device index: after a device
// reset the runtime creates a new primary context, reloads the module, and the array may
// live at another address; the new context has a new ID, so its address is resolved again.
static std::mutex g_noalloc_mu;
struct ScratchAddr {
    unsigned long long ctx_id;
    void* addr;
};
static ScratchAddr g_noalloc_addr[64];
static int g_noalloc_next = 0;

static cudaError_t noalloc_scratch(void** out)
{
    unsigned long long id = 0;
    cudaError_t e = current_context_id(&id);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    for (const ScratchAddr& a : g_noalloc_addr)
        if (a.addr && a.ctx_id == id) {
            *out = a.addr;
            return cudaSuccess;
        }
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    g_noalloc_addr[g_noalloc_next] = ScratchAddr{id, p};
    g_noalloc_next = (g_noalloc_next + 1) % 64;
    *out = p;
    return cudaSuccess;
}

static bool on_device(const void* ptr)
{
    if (!ptr) return false;
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, ptr) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace ubqp

using namespace ubqp;

extern "C" int ubqp_penalized_eval_noalloc(const void* Q, const void* b, const void* p, const void* x, int64_t n,
                                           int64_t batch, int dtype, void* h_out, void* g_out, void* stream)
{
    clear_error();
    if (!Q || !x || n < 1 || batch < 1 || (dtype != UBQP_DTYPE_F32 && dtype != UBQP_DTYPE_F64)) {
        set_error("ubqp_penalized_eval_noalloc: need Q, x, n >= 1, batch >= 1 and dtype UBQP_DTYPE_F32 or _F64");
        return UBQP_EINVAL;
    }
    const int64_t es = dtype == UBQP_DTYPE_F64 ? 8 : 4;
    // limits of the interface (they keep the shares of h within the static scratch)
    if (batch > kNoallocMaxLanes) {
        set_error("ubqp_penalized_eval_noalloc: batch = %lld exceeds the scratch limit of %d points", (long long)batch,
                  kNoallocMaxLanes);
        return UBQP_EINVAL;
    }
    if (n * es > 200 * 1024) {
        set_error("ubqp_penalized_eval_noalloc: n * element size = %lld bytes exceeds the limit of 200 KiB",
                  (long long)(n * es));
        return UBQP_EINVAL;
    }
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        set_error("ubqp_penalized_eval_noalloc: %s", cudaGetErrorString(cudaGetLastError()));
        return UBQP_ECUDA;
    }
    int rb = 8;
    while (rb < 256 && batch * n / rb > 8 * (int64_t)sms) rb *= 2;
    const int64_t nblk = (n + rb - 1) / rb;
    if (batch * nblk > kNoallocMaxItems) {
        set_error("ubqp_penalized_eval_noalloc: batch * ceil(n / %d) = %lld work items exceeds the limit of %d", rb,
                  (long long)(batch * nblk), kNoallocMaxItems);
        return UBQP_EINVAL;
    }
    const void* ptrs[6] = {Q, b, p, x, h_out, g_out};
    for (const void* q : ptrs) {
        if (q && (reinterpret_cast<uintptr_t>(q) % (uintptr_t)es) != 0) {
            set_error("ubqp_penalized_eval_noalloc: every pointer must be aligned to its element size");
            return UBQP_EINVAL;
        }
        if (q && !on_device(q)) {
            set_error("ubqp_penalized_eval_noalloc: all pointers must be device memory");
            return UBQP_EINVAL;
        }
    }
    void* scratch = nullptr;
    cudaError_t e = noalloc_scratch(&scratch);
    if (e != cudaSuccess) {
        set_error("ubqp_penalized_eval_noalloc: resolving the scratch array failed: %s", cudaGetErrorString(e));
        return UBQP_ECUDA;
    }
    cudaStream_t s = (cudaStream_t)stream;
    // (the launch of ubqp_penalized_eval, so both return the same values)
    e = launch_grad(Q, b, p, x, n, batch, dtype, h_out, g_out, scratch, sms, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) {
        set_error("ubqp_penalized_eval_noalloc: %s", cudaGetErrorString(e));
        return UBQP_ECUDA;
    }
    return UBQP_OK;
}
