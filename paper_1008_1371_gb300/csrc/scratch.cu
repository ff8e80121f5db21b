// scratch.cu -- device scratch of the calls.  The device's default pool gives
// its memory back at every synchronisation, and every call here ends with one:
// the next call's first allocation mapped memory anew, about 110 us, as long as
// a tenth of the smallest solve (24 x 24: 0.96 ms, 0.85 so; three small
// allocations: 110-120 us against 17 from a pool that keeps them; 20 of 64 MB:
// 2.8 ms against 0.05).  So the library has a pool of its own for each device (for
// each of a device's first kMaxPools contexts), which keeps at most kKeep bytes
// that no call is using: 256 MB, a thousandth of the device's memory, covers the
// scratch of everything that runs for less than about 50 ms.  What is above it
// goes back at the next synchronisation, and the rest with
// hsvd_release_scratch, or when another allocation would fail (the driver takes
// what a pool does not use).  The pool orders reuse by stream and is safe for
// several threads and streams; a call captured into a graph gets memory nodes
// as it would from the default pool.
#include <cuda.h>

#include <mutex>

#include "hsvd_internal.cuh"

namespace hsvd {
namespace {

constexpr unsigned long long kKeep = 256ull << 20;
constexpr int kMaxDevices = 64;
constexpr int kMaxPools = 4;  // contexts of a device with a pool; the default pool serves any other

struct Pool {
    unsigned long long ctx_id;  // the context the pool was made in (its number is never used again)
    cudaMemPool_t pool;
};
std::mutex g_pool_mutex;
Pool g_pool[kMaxDevices][kMaxPools] = {};

typedef CUresult (*CtxGetCurrentFn)(CUcontext *);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long *);

// the current context's pool, made at its first use (a device reset starts a new
// context); null where there is none (the default pool serves then).  A pool
// stays with its context: calls made in several contexts in turn find theirs.
cudaMemPool_t current_pool(bool make) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
    const unsigned long long ctx = current_context_id();
    if (ctx == 0) return nullptr;
    std::lock_guard<std::mutex> lock(g_pool_mutex);
    int k = 0;
    for (; k < kMaxPools && g_pool[dev][k].pool; ++k)
        if (g_pool[dev][k].ctx_id == ctx) return g_pool[dev][k].pool;
    if (!make || k == kMaxPools) return nullptr;
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
        cudaGetLastError();  // the default pool serves
        return nullptr;
    }
    unsigned long long keep = kKeep;
    if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
        cudaGetLastError();
        cudaMemPoolDestroy(pool);
        return nullptr;
    }
    g_pool[dev][k] = {ctx, pool};
    return pool;
}

}  // namespace

unsigned long long current_context_id() {
    struct Fns {
        CtxGetCurrentFn current = nullptr;
        CtxGetIdFn id = nullptr;
        Fns() {
            void *f = nullptr;
            cudaDriverEntryPointQueryResult q;
            if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
                q == cudaDriverEntryPointSuccess)
                current = reinterpret_cast<CtxGetCurrentFn>(f);
            f = nullptr;
            if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
                q == cudaDriverEntryPointSuccess)
                id = reinterpret_cast<CtxGetIdFn>(f);
        }
    };
    static const Fns fns;
    CUcontext ctx = nullptr;
    unsigned long long id = 0;
    if (!fns.current || !fns.id || fns.current(&ctx) != CUDA_SUCCESS || !ctx || fns.id(ctx, &id) != CUDA_SUCCESS)
        return 0;
    return id;
}

cudaError_t scratch_alloc(void **p, size_t bytes, cudaStream_t st) {
    cudaMemPool_t pool = current_pool(true);
    return pool ? cudaMallocFromPoolAsync(p, bytes, pool, st) : cudaMallocAsync(p, bytes, st);
}

}  // namespace hsvd

using namespace hsvd;

extern "C" int hsvd_release_scratch(void) {
    cudaMemPool_t pool = current_pool(false);
    if (!pool) return HSVD_OK;
    return cudaMemPoolTrimTo(pool, 0) == cudaSuccess ? HSVD_OK : HSVD_ERR_CUDA;
}
