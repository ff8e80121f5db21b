// pointwise.cu -- the pointwise one-sided hyperbolic Jacobi method (Sec. 2,
// Alg. 4.5) for one factor: k_pointwise_cl, a thread-block cluster with one
// warp per pair of a step (pw_cluster.cuh), and for the shapes whose columns do not fit its
// shared memory (two columns of more than about 6,900 rows) k_pointwise, one
// CTA running pw_solve (pw_core.cuh) with G in shared memory and W in global.
#include <algorithm>

#include "pw_cluster.cuh"

namespace hsvd {
namespace {

constexpr int kThreads = 1024;
// of k_pointwise: G and 20 bytes a column within 200 KB (pointwise_fits, so n <= 158), and 12 more a column
constexpr size_t kOneCtaSmemMax = 200 * 1024 + 158 * 12;

template <bool FEW>
__global__ void __launch_bounds__(kThreads, 1)
k_pointwise(const double *__restrict__ G, int64_t ldg, int m, int n, const int8_t *__restrict__ J,
            int m_pad, int n_pad, double tol, double tstop, int max_sweeps, int sort, double *__restrict__ W,
            double *__restrict__ sigma, double *__restrict__ U, int64_t ldu, double *__restrict__ V,
            int64_t ldv, int *__restrict__ out, long long *__restrict__ rot_out) {
    extern __shared__ __align__(16) double smem[];
    __shared__ PwScalars sc;
    PwArrays sh = {};
    sh.Gs = smem;
    sh.gs = n_pad;
    sh.Wg = W;
    pw_carve(sh, smem + (size_t)m_pad * n_pad, n_pad);
    pw_solve<kThreads, FEW>(G, ldg, m, n, J, m_pad, n_pad, tol, tstop, max_sweeps, sort, sh, sc, sigma, U, ldu, V,
                       ldv, &out[0], &out[1], rot_out, &out[2], 0, 0);
}

__global__ void __launch_bounds__(32 * kMaxClPairs)
k_pointwise_cl(const double *__restrict__ G, int64_t ldg, int m, int n, const int8_t *__restrict__ J, int P,
               double tol, double tstop, int max_sweeps, int sort, double *__restrict__ sigma,
               double *__restrict__ U, int64_t ldu, double *__restrict__ V, int64_t ldv, int *__restrict__ out,
               long long *__restrict__ rot_out) {
    extern __shared__ __align__(16) double smem[];
    pw_cluster_solve(smem, G, ldg, m, n, J, P, tol, tstop, max_sweeps, sort, sigma, U, ldu, V, ldv, out, rot_out);
}

}  // namespace

size_t pointwise_smem_bytes(int64_t m_pad, int64_t n_pad) {
    return (size_t)m_pad * n_pad * sizeof(double) + (size_t)n_pad * (sizeof(double) + 3 * sizeof(int));
}

// The sizes the method accepts: G and 20 bytes a column within 200 KB (so
// n <= 158); the one-CTA kernel's arrays, 32 bytes a column, then fit an SM.
bool pointwise_fits(int64_t m, int64_t n) {
    const int64_t n_pad = n + (n & 1);
    return n_pad <= 2048 && pointwise_smem_bytes(pw_rows_pad(m, n), n_pad) <= 200 * 1024;
}

cudaError_t launch_pointwise(const double *G, int64_t ldg, int m, int n, const int8_t *J,
                             double tol, double tstop, int max_sweeps, int sort, double *Wws, double *sigma,
                             double *U, int64_t ldu, double *V, int64_t ldv, int *dev_out,
                             long long *dev_rot, cudaStream_t st) {
    const int n_pad = n + (n & 1);
    const int m_pad = pw_rows_pad(m, n);
    const int half = n_pad / 2;
    // the smallest cluster with at most four pairs a CTA, else the largest
    int max_c = 1;  // of the clusters that the stream's SMs hold
    for (const int limit = stream_limits(st).cluster; 2 * max_c <= std::min(kMaxCl, limit);) max_c *= 2;
    for (int C = 1; C <= max_c; C *= 2) {
        const int P = (half + C - 1) / C;
        const size_t smem = pw_cluster_smem(m_pad, n_pad, P, V != nullptr);
        if (C / 2 >= half && C > 1) break;
        if (smem > kClSmemMax || P > kMaxClPairs || (P > 4 && C < max_c)) continue;
        cudaError_t e =
            cudaFuncSetAttribute(k_pointwise_cl, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmemMax);
        if (e == cudaSuccess && C > 8)
            e = cudaFuncSetAttribute(k_pointwise_cl, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(C);
        cfg.blockDim = dim3(32 * P);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = C;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (C > 8) {  // launch only what the GPU can hold at once
            int clusters = 0;
            e = cudaOccupancyMaxActiveClusters(&clusters, k_pointwise_cl, &cfg);
            if (e != cudaSuccess || clusters < 1) {
                cudaGetLastError();
                break;
            }
        }
        return cudaLaunchKernelEx(&cfg, k_pointwise_cl, G, ldg, m, n, J, P, tol, tstop, max_sweeps, sort,
                                  sigma, U, ldu, V, ldv, dev_out, dev_rot);
    }
    auto kern = n <= kPwFew ? k_pointwise<true> : k_pointwise<false>;
    const size_t smem = (size_t)m_pad * n_pad * sizeof(double) + pw_aux_bytes(n_pad);
    cudaError_t e =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOneCtaSmemMax);
    if (e != cudaSuccess) return e;
    kern<<<1, kThreads, smem, st>>>(G, ldg, m, n, J, m_pad, n_pad, tol, tstop, max_sweeps, sort, Wws,
                                           sigma, U, ldu, V, ldv, dev_out, dev_rot);
    return cudaGetLastError();
}

}  // namespace hsvd
