// limits.cu -- what a launch on a stream can count on: a stream of a green
// context has part of the device's SMs, and clusters only as large as the part
// keeps on one GPC.  Kernels whose CTAs wait for each other (a cooperative grid,
// a cluster beyond the portable size) take their size from here.
#include <cuda.h>

#include "hsvd_internal.cuh"

namespace hsvd {

StreamLimits stream_limits(cudaStream_t st) {
    typedef CUresult (*StreamGetCtxFn)(CUstream, CUcontext *, CUgreenCtx *);
    typedef CUresult (*GetResourceFn)(CUgreenCtx, CUdevResource *, CUdevResourceType);
    struct Fns {
        StreamGetCtxFn stream_ctx = nullptr;
        GetResourceFn resource = nullptr;
        Fns() {
            void *f = nullptr;
            cudaDriverEntryPointQueryResult q;
            if (cudaGetDriverEntryPointByVersion("cuStreamGetCtx", &f, 12050, cudaEnableDefault, &q) == cudaSuccess &&
                q == cudaDriverEntryPointSuccess)
                stream_ctx = reinterpret_cast<StreamGetCtxFn>(f);
            f = nullptr;
            if (cudaGetDriverEntryPointByVersion("cuGreenCtxGetDevResource", &f, 12040, cudaEnableDefault, &q) ==
                    cudaSuccess &&
                q == cudaDriverEntryPointSuccess)
                resource = reinterpret_cast<GetResourceFn>(f);
        }
    };
    static const Fns fns;
    StreamLimits l = {152, 16};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&l.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        cudaGetLastError();
    CUcontext ctx = nullptr;
    CUgreenCtx green = nullptr;
    CUdevResource r = {};
    if (!fns.stream_ctx || !fns.resource || fns.stream_ctx(st, &ctx, &green) != CUDA_SUCCESS || !green ||
        fns.resource(green, &r, CU_DEV_RESOURCE_TYPE_SM) != CUDA_SUCCESS || r.sm.smCount < 1)
        return l;
    l.sms = (int)r.sm.smCount < l.sms ? (int)r.sm.smCount : l.sms;
    const int together = (int)r.sm.smCoscheduledAlignment;
    l.cluster = together < 1 ? 1 : (together < 16 ? together : 16);
    return l;
}

}  // namespace hsvd
