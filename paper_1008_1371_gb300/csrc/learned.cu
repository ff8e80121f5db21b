// learned.cu -- the learned form of the blocked method: a small MLP predicts,
// from the previous sweep's record of a block-pair visit, whether that visit
// will need a rotation (its pivot block fails the test of Eq. 2.3); visits
// predicted to pass are skipped.  The plain full sweep stays the judge: a
// masked sweep that rotates nothing is followed by a full sweep, and only a
// full sweep without rotations ends the iteration (Sec. 2 stopping rule), so
// the result never depends on the network.
//
// Network: 8 features -> 64 (ReLU) -> 64 (ReLU) -> 1 (logit), weights rounded
// to BF16, FP32 accumulation.  The same forward code serves inference in the
// solver and the training kernels (forward + backward, then Adam).
//
// Parameter vector (FP32 master copy, kMlpParams floats):
//   W1[64][8], b1[64], W2[64][64], b2[64], w3[64], b3.
//
// Features of a visit v (pair of block columns I, J) for sweep k, from the
// record r[v] the inner solve wrote at v's last computed visit:
//   f0 = log2(max scaled |a_ij| over the I x J block / tol) / 64
//   f1 = log2(Frobenius norm of the scaled I x J block) / 64
//   f2 = inner rotations applied / b^2
//   f3 = k / max_sweeps
//   f4 = fraction of (i in I, j in J) with opposite signs (hyperbolic pairs)
//   f5 = log2(mean d over I / mean d over J) / 64
//   f6 = |I - J| / nb
//   f7 = 1 if v was skipped in sweep k - 1, else 0
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "hsvd_internal.cuh"

namespace hsvd {

namespace {

constexpr int kF = 8, kH = 64;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kH * kF, kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH,
              kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH, kParams = kOffB3 + 1;
static_assert(kParams == HSVD_MLP_PARAMS, "parameter count");

constexpr int kTrainSamples = 64;  // samples per CTA of the training kernel
constexpr int kTrainThreads = 512;
constexpr int kInferThreads = 256;  // 32 samples at a time
constexpr int kRow = kH + 4;        // rows of 64 values in shared memory: 16-byte accesses to 8 rows at once
constexpr int kRow1 = kF + 4;       // rows of W1, likewise

__device__ __forceinline__ float bf16_round(float w) { return __bfloat162float(__float2bfloat16_rn(w)); }

// the network in shared memory: weights rounded to BF16, biases FP32
struct Net {
    alignas(16) float w1[kH * kRow1], w2[kH * kRow], b1[kH], b2[kH], w3[kH], b3;
};

__device__ __forceinline__ void load_net(const float *__restrict__ p, Net &net) {
    const int tid = threadIdx.x;
#pragma unroll 8
    for (int e = tid; e < kH * kH; e += blockDim.x) net.w2[(e / kH) * kRow + e % kH] = bf16_round(p[kOffW2 + e]);
    for (int e = tid; e < kH * kF; e += blockDim.x) net.w1[(e / kF) * kRow1 + e % kF] = bf16_round(p[kOffW1 + e]);
    if (tid < kH) {
        net.b1[tid] = p[kOffB1 + tid];
        net.b2[tid] = p[kOffB2 + tid];
        net.w3[tid] = bf16_round(p[kOffW3 + tid]);
    }
    if (tid == 0) net.b3 = p[kOffB3];
}

// Forward pass of the CTA's T / 8 samples xs[s][kF]: h1, h2 [s][kRow] receive
// the post-ReLU activations.  A thread computes 2 samples by 4 units (s = tid /
// 16 and T / 16 on, unit j = tid % 16 and every 16 on), each sum from its bias
// through the inputs in order, so a value doesn't depend on the tile it is
// computed in; per 4 inputs 6 16-byte loads serve 32 FMAs.  Ends with a barrier.
template <int T>
__device__ __forceinline__ void mlp_layers(const Net &net, const float *__restrict__ xs, float *__restrict__ h1,
                                           float *__restrict__ h2) {
    const int tj = threadIdx.x % 16, ts = threadIdx.x / 16;
    float a[2][4];
    auto layer = [&](const float *in, int ldi, const float *w, int ldw, const float *bias, int k, float *out) {
#pragma unroll
        for (int q = 0; q < 4; ++q) a[0][q] = a[1][q] = bias[tj + 16 * q];
#pragma unroll 4
        for (int i = 0; i < k; i += 4) {
            const float4 x0 = *reinterpret_cast<const float4 *>(in + ts * ldi + i);
            const float4 x1 = *reinterpret_cast<const float4 *>(in + (ts + T / 16) * ldi + i);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 u = *reinterpret_cast<const float4 *>(w + (tj + 16 * q) * ldw + i);
                a[0][q] = fmaf(u.w, x0.w, fmaf(u.z, x0.z, fmaf(u.y, x0.y, fmaf(u.x, x0.x, a[0][q]))));
                a[1][q] = fmaf(u.w, x1.w, fmaf(u.z, x1.z, fmaf(u.y, x1.y, fmaf(u.x, x1.x, a[1][q]))));
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            out[ts * kRow + tj + 16 * q] = fmaxf(a[0][q], 0.0f);
            out[(ts + T / 16) * kRow + tj + 16 * q] = fmaxf(a[1][q], 0.0f);
        }
        __syncthreads();
    };
    layer(xs, kF, net.w1, kRow1, net.b1, kF, h1);
    layer(h1, kRow, net.w2, kRow, net.b2, kH, h2);
}

// the logit of one sample from its h2
__device__ __forceinline__ float mlp_logit(const Net &net, const float *__restrict__ h2) {
    float z = net.b3;
#pragma unroll
    for (int i = 0; i < kH; i += 4) {
        const float4 h = *reinterpret_cast<const float4 *>(h2 + i), w = *reinterpret_cast<const float4 *>(net.w3 + i);
        z = fmaf(w.w, h.w, fmaf(w.z, h.z, fmaf(w.y, h.y, fmaf(w.x, h.x, z))));
    }
    return z;
}

// Tiles of 32 samples, a CTA every gridDim-th.  Bound by latencies at the sizes
// in use (loading the network, three dependent layers); a thread per sample,
// its activations in local memory, left most SMs without work.  Measured, the
// call: 4096 samples 14 us (of them 7 in the kernel), 60000 27 us; with a thread
// per sample 19 and 45.
__global__ void __launch_bounds__(kInferThreads) k_mlp_infer(const float *__restrict__ params,
                                                             const float *__restrict__ X, int n,
                                                             float *__restrict__ logits, int8_t *__restrict__ skip,
                                                             float logit_tau) {
    constexpr int S = kInferThreads / 8;
    __shared__ Net net;
    __shared__ alignas(16) float xs[S * kF], h1[S * kRow], h2[S * kRow];
    const int tid = threadIdx.x;
    load_net(params, net);
    for (int s0 = blockIdx.x * S; s0 < n; s0 += gridDim.x * S) {
        xs[tid] = s0 + tid / kF < n ? X[(size_t)s0 * kF + tid] : 0.0f;
        __syncthreads();
        mlp_layers<kInferThreads>(net, xs, h1, h2);
        if (tid < S && s0 + tid < n) {
            const float z = mlp_logit(net, h2 + tid * kRow);
            if (logits) logits[s0 + tid] = z;
            if (skip) skip[s0 + tid] = z < logit_tau ? 1 : 0;
        }
    }
}

struct TrainSmem {
    Net net;
    alignas(16) float xs[kTrainSamples * kF];
    alignas(16) float h1[kTrainSamples * kRow], h2[kTrainSamples * kRow];
    alignas(16) float d2[kTrainSamples * kRow], d1[kTrainSamples * kRow];  // dL/d(pre-activations)
    float dz[kTrainSamples], ls[kTrainSamples];
};

// Gradient of the mean binary cross-entropy with logits over n samples,
// L = mean(softplus(z) - y z), per CTA of kTrainSamples samples: partial
// sums over the CTA's samples in a fixed order (deterministic).  Every product
// is a small matrix product of register tiles (2 x 4 outputs a thread) over
// operands in shared memory.  Bound by the FP32 pipe of the SMs that have a CTA
// (64 of them with 4096 samples).  Measured, the call with the reduction: 4096
// samples 27 us, 60000 97 us; with a thread per sample for both passes 83 and 549.
__global__ void __launch_bounds__(kTrainThreads) k_mlp_grad_partial(const float *__restrict__ params,
                                                                    const float *__restrict__ X,
                                                                    const float *__restrict__ y, int n,
                                                                    float *__restrict__ gpart,
                                                                    float *__restrict__ lpart) {
    extern __shared__ __align__(16) unsigned char smem[];
    TrainSmem &sm = *reinterpret_cast<TrainSmem *>(smem);
    static_assert(kTrainThreads == kTrainSamples * kF && kTrainThreads == kH * kF, "one value a thread");
    const int tid = threadIdx.x;
    const int s0 = blockIdx.x * kTrainSamples;
    const int ns = min(kTrainSamples, n - s0);
    const float inv_n = 1.0f / (float)n;
    sm.xs[tid] = tid / kF < ns ? X[(size_t)s0 * kF + tid] : 0.0f;
    const float yy = tid < ns ? y[s0 + tid] : 0.0f;  // of the threads that finish a sample
    load_net(params, sm.net);
    __syncthreads();
    mlp_layers<kTrainThreads>(sm.net, sm.xs, sm.h1, sm.h2);
    if (tid < kTrainSamples) {
        const float z = mlp_logit(sm.net, sm.h2 + tid * kRow);
        if (tid < ns) {
            const float p = 1.0f / (1.0f + expf(-z));
            sm.dz[tid] = (p - yy) * inv_n;
            // softplus(z) - y z, written stably
            sm.ls[tid] = fmaxf(z, 0.0f) + log1pf(expf(-fabsf(z))) - yy * z;
        } else {
            sm.dz[tid] = 0.0f;
            sm.ls[tid] = 0.0f;
        }
    }
    __syncthreads();
    for (int e = tid; e < kTrainSamples * kH; e += kTrainThreads) {
        const int s = e / kH, j = e % kH;
        sm.d2[s * kRow + j] = sm.h2[s * kRow + j] > 0.0f ? sm.dz[s] * sm.net.w3[j] : 0.0f;
    }
    __syncthreads();
    const int t4 = 4 * (tid % 16), ts = tid / 16;  // 4 units, and a row of 32
    {                                              // d1 = (d2 W2) where h1 > 0: samples ts and ts + 32
        float a[2][4] = {};
#pragma unroll 4
        for (int j = 0; j < kH; ++j) {
            const float4 w = *reinterpret_cast<const float4 *>(sm.net.w2 + j * kRow + t4);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float d = sm.d2[(ts + 32 * h) * kRow + j];
                a[h][0] = fmaf(w.x, d, a[h][0]);
                a[h][1] = fmaf(w.y, d, a[h][1]);
                a[h][2] = fmaf(w.z, d, a[h][2]);
                a[h][3] = fmaf(w.w, d, a[h][3]);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int o = (ts + 32 * h) * kRow + t4;
#pragma unroll
            for (int q = 0; q < 4; ++q) sm.d1[o + q] = sm.h1[o + q] > 0.0f ? a[h][q] : 0.0f;
        }
    }
    __syncthreads();
    float *g = gpart + (size_t)blockIdx.x * kParams;
    {  // W2: units ts and ts + 32 by inputs t4 ..
        float a[2][4] = {};
#pragma unroll 4
        for (int s = 0; s < kTrainSamples; ++s) {
            const float4 x = *reinterpret_cast<const float4 *>(sm.h1 + s * kRow + t4);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float d = sm.d2[s * kRow + ts + 32 * h];
                a[h][0] = fmaf(d, x.x, a[h][0]);
                a[h][1] = fmaf(d, x.y, a[h][1]);
                a[h][2] = fmaf(d, x.z, a[h][2]);
                a[h][3] = fmaf(d, x.w, a[h][3]);
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < 4; ++q) g[kOffW2 + (ts + 32 * h) * kH + t4 + q] = a[h][q];
    }
    {  // W1: one value a thread
        const int j = tid / kF, i = tid % kF;
        float a = 0.0f;
#pragma unroll 8
        for (int s = 0; s < kTrainSamples; ++s) a = fmaf(sm.d1[s * kRow + j], sm.xs[s * kF + i], a);
        g[kOffW1 + tid] = a;
    }
    // the rest: sums over the samples of one array each
    const int j = tid % kH;
    float a = 0.0f;
    if (tid < 2 * kH) {
        const float *d = (tid < kH ? sm.d1 : sm.d2) + j;
#pragma unroll 8
        for (int s = 0; s < kTrainSamples; ++s) a += d[s * kRow];
        g[(tid < kH ? kOffB1 : kOffB2) + j] = a;
    } else if (tid < 3 * kH) {
#pragma unroll 8
        for (int s = 0; s < kTrainSamples; ++s) a = fmaf(sm.dz[s], sm.h2[s * kRow + j], a);
        g[kOffW3 + j] = a;
    } else if (tid == 3 * kH) {
#pragma unroll 8
        for (int s = 0; s < kTrainSamples; ++s) a += sm.dz[s];
        g[kOffB3] = a;
    } else if (tid == 4 * kH) {
#pragma unroll 8
        for (int s = 0; s < kTrainSamples; ++s) a += sm.ls[s];
        lpart[blockIdx.x] = a * inv_n;
    }
}

// Sum of the CTA partials, in CTA order: 32 values a CTA, whose 8 warps load
// kRedRows partials at a time (all in flight together) for warp 0 to add one by
// one.  The loss is value kParams.  Bound by the latency of one stage's loads:
// 64 partials 3.7 us.
constexpr int kRedRows = 128;
__global__ void __launch_bounds__(256) k_mlp_grad_reduce(const float *__restrict__ gpart,
                                                         const float *__restrict__ lpart, int nblk,
                                                         float *__restrict__ grad, float *__restrict__ loss) {
    __shared__ float buf[2][kRedRows][32];
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
    const int q = blockIdx.x * 32 + lane;
    const float *src = q < kParams ? gpart + q : lpart;
    const size_t ld = q < kParams ? kParams : 1;
    const bool live = q <= kParams;
    float a = 0.0f;
    int h = 0;
    for (int b0 = 0; b0 < nblk; b0 += kRedRows, h ^= 1) {
        float v[kRedRows / 8];
#pragma unroll
        for (int r = 0; r < kRedRows / 8; ++r) {
            const int b = b0 + warp + 8 * r;
            v[r] = live && b < nblk ? src[b * ld] : 0.0f;
        }
#pragma unroll
        for (int r = 0; r < kRedRows / 8; ++r) buf[h][warp + 8 * r][lane] = v[r];
        __syncthreads();  // one barrier a stage: the other buffer is written meanwhile
        if (warp == 0) {
            const int nb = min(kRedRows, nblk - b0);
#pragma unroll 16
            for (int b = 0; b < nb; ++b) a += buf[h][b][lane];
        }
    }
    if (warp == 0 && q < kParams) grad[q] = a;
    if (warp == 0 && q == kParams && loss) *loss = a;
}

// Adam (Kingma and Ba): m = b1 m + (1-b1) g, v = b2 v + (1-b2) g^2,
// p -= lr (m / (1 - b1^t)) / (sqrt(v / (1 - b2^t)) + eps)
__global__ void k_adam(float *__restrict__ p, float *__restrict__ m, float *__restrict__ v,
                       const float *__restrict__ g, int t, float lr, float b1, float b2, float eps) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= kParams) return;
    const float gq = g[q];
    const float mq = b1 * m[q] + (1.0f - b1) * gq;
    const float vq = b2 * v[q] + (1.0f - b2) * gq * gq;
    m[q] = mq;
    v[q] = vq;
    const float mh = mq / (1.0f - powf(b1, (float)t));
    const float vh = vq / (1.0f - powf(b2, (float)t));
    p[q] -= lr * mh / (sqrtf(vh) + eps);
}

// features of every visit (see the file comment); tab holds the first
// columns (I b, J b) of each visit, trace the inner solve's records
__global__ void k_features(const float *__restrict__ trace, const int8_t *__restrict__ prev_skip,
                           const int *__restrict__ tab, int nvis, int b, int nb, int sweep, int max_sweeps,
                           double tol, float *__restrict__ X) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= nvis) return;
    const float *r = trace + (size_t)v * HSVD_TRACE_FIELDS;
    const float tiny = 1e-30f;
    const float bi = (float)(tab[2 * v] / b), bj = (float)(tab[2 * v + 1] / b);
    float *x = X + (size_t)v * kF;
    x[0] = log2f(fmaxf(r[0], tiny) / (float)tol) * (1.0f / 64.0f);
    x[1] = log2f(fmaxf(r[1], tiny)) * (1.0f / 64.0f);
    x[2] = r[2] / (float)(b * b);
    x[3] = (float)sweep / (float)max_sweeps;
    x[4] = r[5];
    x[5] = log2f(fmaxf(r[3], tiny) / fmaxf(r[4], tiny)) * (1.0f / 64.0f);
    x[6] = fabsf(bi - bj) / (float)nb;
    x[7] = prev_skip ? (float)prev_skip[v] : 0.0f;
}

// training rows (8 features, label = the visit rotated in this sweep)
__global__ void k_export(const float *__restrict__ X, const float *__restrict__ trace, int nvis,
                         float *__restrict__ out) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= nvis) return;
#pragma unroll
    for (int i = 0; i < kF; ++i) out[(size_t)v * (kF + 1) + i] = X[(size_t)v * kF + i];
    out[(size_t)v * (kF + 1) + kF] = trace[(size_t)v * HSVD_TRACE_FIELDS + 2] > 0.0f ? 1.0f : 0.0f;
}

// the visit table of a masked sweep under the pair schedule: a skipped visit's
// entry becomes (-1, -1), which the Gram and inner-solve kernels treat as "no
// visit"; *kept counts the visits that stay
__global__ void k_mask_table(const int *__restrict__ outer, const int8_t *__restrict__ skip, int nvis,
                             int *__restrict__ tab, int *__restrict__ kept) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    const bool keep = v < nvis && !skip[v];
    if (v < nvis) {
        tab[2 * v] = keep ? outer[2 * v] : -1;
        tab[2 * v + 1] = keep ? outer[2 * v + 1] : -1;
    }
    const unsigned n = __popc(__ballot_sync(0xffffffffu, keep));
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(kept, (int)n);
}

}  // namespace

cudaError_t launch_features(const float *trace, const int8_t *prev_skip, const int *tab, int nvis, int b, int nb,
                            int sweep, int max_sweeps, double tol, float *X, cudaStream_t st) {
    k_features<<<(nvis + 127) / 128, 128, 0, st>>>(trace, prev_skip, tab, nvis, b, nb, sweep, max_sweeps, tol, X);
    return cudaGetLastError();
}

cudaError_t launch_mlp_infer(const float *params, const float *X, int n, float *logits, int8_t *skip,
                             float logit_tau, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    constexpr int S = kInferThreads / 8;
    // at most the CTAs that are on the chip together (4 on an SM): the network is loaded once for all their tiles
    const int tiles = (int)(((int64_t)n + S - 1) / S);
    k_mlp_infer<<<tiles < 4 * 152 ? tiles : 4 * 152, kInferThreads, 0, st>>>(params, X, n, logits, skip, logit_tau);
    return cudaGetLastError();
}

cudaError_t launch_mask_table(const int *outer, const int8_t *skip, int nvis, int *tab, int *kept, cudaStream_t st) {
    k_mask_table<<<(nvis + 127) / 128, 128, 0, st>>>(outer, skip, nvis, tab, kept);
    return cudaGetLastError();
}

cudaError_t launch_export(const float *X, const float *trace, int nvis, float *out, cudaStream_t st) {
    k_export<<<(nvis + 127) / 128, 128, 0, st>>>(X, trace, nvis, out);
    return cudaGetLastError();
}

int mlp_grad_blocks(int n) { return (n + kTrainSamples - 1) / kTrainSamples; }

cudaError_t launch_mlp_grad(const float *params, const float *X, const float *y, int n, float *gpart, float *lpart,
                            float *grad, float *loss, cudaStream_t st) {
    const int nblk = mlp_grad_blocks(n);
    const size_t smem = sizeof(TrainSmem);
    cudaError_t e = cudaFuncSetAttribute(k_mlp_grad_partial, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_mlp_grad_partial<<<nblk, kTrainThreads, smem, st>>>(params, X, y, n, gpart, lpart);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_mlp_grad_reduce<<<(kParams + 1 + 31) / 32, 256, 0, st>>>(gpart, lpart, nblk, grad, loss);
    return cudaGetLastError();
}

cudaError_t launch_adam(float *p, float *m, float *v, const float *g, int t, float lr, float b1, float b2, float eps,
                        cudaStream_t st) {
    k_adam<<<(kParams + 255) / 256, 256, 0, st>>>(p, m, v, g, t, lr, b1, b2, eps);
    return cudaGetLastError();
}

}  // namespace hsvd

using namespace hsvd;

extern "C" {

int hsvd_mlp_forward(const float *params, const float *X, int64_t n, float *logits, void *stream) {
    if (!params || !X || !logits || n < 0 || n > (1 << 30)) return HSVD_ERR_ARG;
    if (!all_device({params, X, logits})) return HSVD_ERR_ARG;
    return launch_mlp_infer(params, X, (int)n, logits, nullptr, 0.0f, static_cast<cudaStream_t>(stream)) ==
                   cudaSuccess
               ? HSVD_OK
               : HSVD_ERR_CUDA;
}

int hsvd_mlp_grad(const float *params, const float *X, const float *y, int64_t n, float *grad, float *loss,
                  void *stream) {
    if (!params || !X || !y || !grad || n < 1 || n > (1 << 26)) return HSVD_ERR_ARG;
    if (!all_device({params, X, y, grad, loss})) return HSVD_ERR_ARG;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int nblk = mlp_grad_blocks((int)n);
    float *gpart = nullptr;  // the partial gradients, then the partial losses
    if (scratch_alloc((void **)&gpart, sizeof(float) * (size_t)nblk * (HSVD_MLP_PARAMS + 1), st) != cudaSuccess)
        return HSVD_ERR_NOMEM;
    const cudaError_t e =
        launch_mlp_grad(params, X, y, (int)n, gpart, gpart + (size_t)nblk * HSVD_MLP_PARAMS, grad, loss, st);
    cudaFreeAsync(gpart, st);
    return e == cudaSuccess ? HSVD_OK : HSVD_ERR_CUDA;
}

int hsvd_mlp_adam(float *params, float *m, float *v, const float *grad, int t, float lr, float beta1, float beta2,
                  float eps, void *stream) {
    if (!params || !m || !v || !grad || t < 1 || !(lr > 0.0f)) return HSVD_ERR_ARG;
    if (!all_device({params, m, v, grad})) return HSVD_ERR_ARG;
    return launch_adam(params, m, v, grad, t, lr, beta1, beta2, eps, static_cast<cudaStream_t>(stream)) ==
                   cudaSuccess
               ? HSVD_OK
               : HSVD_ERR_CUDA;
}

}  // extern "C"
