// batched.cu -- the batched form: many independent factors (sizes mixed) in
// one persistent launch, each solved by the pointwise one-sided hyperbolic
// Jacobi method (Sec. 2, Alg. 4.5; the per-factor body is pw_solve).
//
// Work distribution.  The host sorts the factors by (group width, n), both
// decreasing, and the kernel's CTAs (1024 threads, or 512 with twice the
// registers a thread, one per SM, launched once and captured in a CUDA graph)
// take them in that order from one atomic counter (EVEN: but for every group's
// first): the largest first, so the long factors start early and the short ones
// fill the tail.
// A CTA starts as one group of 1024 threads.  When the next factor in the
// queue asks for a narrower group, the CTA splits into two groups of 512
// (each with half the shared memory and its own named barrier), and a 512
// group splits again into two groups of 256; every group then takes factors
// from the counter on its own.  The queue order makes the widths
// non-increasing, so a group never has to grow back.
//
// Residency.  In its group's shared memory a factor keeps G and W when both
// fit, otherwise G only (W then in a per-group slot of a global workspace,
// L2-resident), otherwise neither.
//
// The autotuner (host, tune_widths) picks the group width per size bucket by
// timing each width on a sample of that bucket's factors for two sweeps, and
// caches the choice per device and bucket layout.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <vector>

#include "pw_cluster.cuh"

namespace hsvd {
namespace {

constexpr int kBarriers = 7;  // 1 (1024) + 2 (512) + 4 (256)

struct BTask {
    const double *G;
    const int8_t *J;
    double *sigma, *U, *V;
    int64_t ldg, ldu, ldv;
    double tol;
    int m, n, idx, width;
};

struct BArgs {
    const BTask *tasks;
    int count;
    int *counter;        // factors taken (EVEN: beyond the first ones)
    int width;           // EVEN: the width of every factor
    int firsts;          // EVEN: factors given out at the start, one a group
    int max_sweeps, sort;
    double tstop;        // tangent threshold of the early stop, 0 = off
    double *ws;          // grid x ws_stride doubles
    int64_t ws_stride;   // doubles per CTA
    int *res;            // 3 per factor: status, sweeps, stop rule
    long long *rot;      // per factor
    int *where;          // per factor: 0 G and W shared, 1 G shared, 2 global
};

__device__ __forceinline__ int bar_id(int width, int g) { return width == 1024 ? 0 : (width == 512 ? 1 + g : 3 + g); }

template <int NT, bool FEW>
__device__ void solve_task(const BArgs &A, int k, int g, unsigned char *sm, size_t budget, double *wsg,
                           PwScalars *sc) {
    const BTask t = A.tasks[k];
    const int n_pad = t.n + (t.n & 1), m_pad = pw_rows_pad(t.m, t.n);
    const size_t gc = (size_t)m_pad * sizeof(double), wc = (size_t)n_pad * sizeof(double);
    const size_t ab = pw_aux_bytes(n_pad);
    // shared memory: the per-column arrays, then as many columns of G as fit,
    // then of W; the rest of both, and the arrays of a factor too large for
    // them, in the group's part of the workspace
    PwArrays a;
    a.Gg = wsg;
    a.Wg = wsg + (size_t)m_pad * n_pad;
    const bool aux_shared = ab <= budget;
    size_t left = aux_shared ? budget - ab : budget;
    unsigned char *at = aux_shared ? sm + ab : sm;
    pw_carve(a, aux_shared ? reinterpret_cast<void *>(sm)
                           : reinterpret_cast<void *>(a.Wg + (size_t)n_pad * n_pad), n_pad);
    a.Gs = reinterpret_cast<double *>(at);
    a.gs = (int)min((size_t)n_pad, left / gc);
    left -= a.gs * gc;
    a.Ws = a.Gs + (size_t)a.gs * m_pad;
    a.ws = t.V ? (int)min((size_t)n_pad, left / wc) : n_pad;
    const int where = a.gs < n_pad ? 2 : (a.ws < n_pad ? 1 : 0);
    const int bar = bar_id(NT, g);
    int *res = A.res + 3 * (size_t)t.idx;
    pw_solve<NT, FEW>(t.G, t.ldg, t.m, t.n, t.J, m_pad, n_pad, t.tol, A.tstop, A.max_sweeps, A.sort, a, sc[bar], t.sigma,
                 t.U, t.ldu, t.V, t.ldv, &res[0], &res[1], &A.rot[t.idx], &res[2], bar, NT == 512 ? 2 * g : g);
    if ((threadIdx.x & (NT - 1)) == 0) A.where[t.idx] = where;
}

// EVEN is for queues of one width narrower than a CTA: the first factor of every
// group f is dealt out, back and forth, so that no SM has three while another has
// one.  By the counter the CTAs that start first can take one for each of their
// groups: 200 factors of n = 64 then take 9.6 or 12.7 ms from process to process, 304
// of n = 256 on 256 threads 613 or 704; dealt out 9.6 and 450.  It is a template
// argument for the registers of the other kernels (1 % there).
__device__ __forceinline__ int first_factor(int f) {
    return f * (int)gridDim.x + ((f & 1) ? (int)(gridDim.x - 1 - blockIdx.x) : (int)blockIdx.x);
}

// Group g of width NT: solves factors from the queue, starting with factor k
// (k < 0: take one from the counter first).
template <int NT, bool FEW, bool EVEN, int CTA>
__device__ void group_loop(const BArgs &A, int k, int g, unsigned char *sm, size_t budget, double *wsg,
                           int64_t wsg_len, PwScalars *sc, int *fetch) {
    const int bar = bar_id(NT, g);
    const int tid = threadIdx.x & (NT - 1);
    for (;;) {
        if (k < 0) {
            if (tid == 0) fetch[bar] = (EVEN ? A.firsts : 0) + atomicAdd(A.counter, 1);
            grp_sync<NT>(bar);
            k = fetch[bar];
            grp_sync<NT>(bar);
        }
        if (k >= A.count) return;
        // small factors are all of one size bucket, so of one width: EVEN, or the CTA's
        if constexpr (NT > 256 && !(FEW && !EVEN && CTA == 1024)) {
            if ((EVEN ? A.width : A.tasks[k].width) < NT) {
                const int sub = tid / (NT / 2);
                const int other = EVEN ? first_factor((2 * g + 1) * (NT / 2) / A.width) : -1;
                group_loop<NT / 2, FEW, EVEN, CTA>(A, sub == 0 ? k : other, 2 * g + sub, sm + sub * (budget / 2),
                                                   budget / 2, wsg + sub * (wsg_len / 2), wsg_len / 2, sc, fetch);
                return;
            }
        }
        if constexpr (!EVEN || NT < 1024) solve_task<NT, FEW>(A, k, g, sm, budget, wsg, sc);
        k = -1;
    }
}

// CTA threads: 1024 (64 registers a thread) or 512 (128: the per-thread
// state of pw_solve without spills)
template <int CTA, bool FEW, bool EVEN>
__global__ void __launch_bounds__(CTA, 1) k_batched(BArgs A, int smem_budget) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ PwScalars sc[kBarriers];
    __shared__ int fetch[kBarriers];
    group_loop<CTA, FEW, EVEN, CTA>(A, EVEN ? first_factor(0) : -1, 0, smem, (size_t)smem_budget,
                                    A.ws + (size_t)blockIdx.x * A.ws_stride, A.ws_stride, sc, fetch);
}

// A few factors, too few to fill the SMs one each: one cluster per factor, in
// queue order (pw_cluster.cuh; P pairs a CTA for the factor's size).
__global__ void __launch_bounds__(32 * kMaxClPairs) k_batched_cl(BArgs A, int C) {
    extern __shared__ __align__(16) double dsmem[];
    const BTask t = A.tasks[blockIdx.x / C];
    const int half = (t.n + 1) / 2, P = (half + C - 1) / C;
    if (blockIdx.x % C == 0 && threadIdx.x == 0) A.where[t.idx] = 0;
    int *res = A.res + 3 * (size_t)t.idx;
    pw_cluster_solve(dsmem, t.G, t.ldg, t.m, t.n, t.J, P, t.tol, A.tstop, A.max_sweeps, A.sort, t.sigma, t.U, t.ldu,
                     t.V, t.ldv, res, &A.rot[t.idx]);
}

// ------------------------------------------------------------------ host side

constexpr int kSmemBudget = 220 * 1024;  // one CTA per SM
const int kBucketEdges[] = {16, 40, 72, 128, 192, 1 << 30};
constexpr int kBuckets = 5;

int bucket_of(int64_t n) {
    for (int b = 0; b < kBuckets; ++b)
        if (n < kBucketEdges[b + 1]) return b;
    return kBuckets - 1;
}

size_t need_bytes(int64_t m, int64_t n) {
    const int64_t n_pad = n + (n & 1), m_pad = pw_rows_pad(m, n);
    return (size_t)(m_pad * n_pad + n_pad * n_pad) * sizeof(double);
}

// workspace doubles per CTA: a group of width w owns w/cta of the slot, and
// must hold G and W of any factor it may take, and the per-column arrays
int64_t ws_stride_for(const std::vector<BTask> &tasks, int cta) {
    size_t s = 0;
    for (const BTask &t : tasks)
        s = std::max(s, (need_bytes(t.m, t.n) + pw_aux_bytes(t.n + (t.n & 1))) * (size_t)(cta / t.width));
    return (int64_t)((s / sizeof(double) + 31) / 32 * 32);
}

// pairs a CTA and shared memory of the largest factor on clusters of C CTAs
struct ClShape {
    int P = 0;
    size_t smem = 0;
};
ClShape cluster_shape(const std::vector<BTask> &tasks, int C) {
    ClShape s;
    for (const BTask &t : tasks) {
        const int64_t n_pad = t.n + (t.n & 1), P = (n_pad / 2 + C - 1) / C;
        s.P = std::max(s.P, (int)P);
        s.smem = std::max(s.smem, pw_cluster_smem(pw_rows_pad(t.m, t.n), n_pad, P, t.V != nullptr));
    }
    return s;
}

cudaError_t cluster_config(int count, int C, const ClShape &s, cudaStream_t st, cudaLaunchConfig_t &cfg,
                           cudaLaunchAttribute *attr) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3((unsigned)(count * C));
    cfg.blockDim = dim3(32 * s.P);
    cfg.dynamicSmemBytes = s.smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaFuncSetAttribute(k_batched_cl, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kClSmemMax);
    if (e == cudaSuccess && C > 8)
        e = cudaFuncSetAttribute(k_batched_cl, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

// Cluster size for a batch of at most one factor per SM, 0: the queue of groups.
// Both are estimated in cycles a step, times the steps of a sweep, from the FP64
// instructions a warp issues (64 cycles on its quarter of an SM) and what a step
// takes besides them, fitted to whole calls on n = 4 to 256: on groups a factor
// has an SM to itself, at most a warp per pair forms dots, and the packed
// rotations and three barriers take 10,200 cycles; on clusters a warp per pair
// has a rotation of its own (56 instructions) and one barrier, 2,000.  0.8: the
// later sweeps skip rotations and kept dots.  The clusters share the SMs' FP64
// pipes, which no residency count shows (114 factors of n = 40: 3,200 cycles by
// the longest factor, 17,000 by the pipes), at 250 cycles a CTA and more where the
// factors alone fill the SMs.  Clusters must be
// estimated a quarter faster than groups, since they share the SMs less evenly than
// the pipes' sum says; a smaller cluster must win 6 %.  Measured, the kernel in ms,
// groups / this choice: n = 8: 4 factors 0.39 / 0.21, 152 0.40 / 0.23; n = 16: 4 0.76
// / 0.45; n = 40: 38 3.3 / 2.6, 114 3.4 / 3.4 (clusters of 16: 7.2); n = 64: 38 6.6 /
// 3.9, 76 6.9 / 6.9 (8.0); n = 256: 38 219 / 150; n from 10 to 70: 152 12.0 / 8.4, 114
// 12.4 / 5.5; 16 to 128: 152 36 / 30; 1024 x 8: 4 0.96 / 0.56.
int few_clusters(const std::vector<BTask> &tasks, const StreamLimits &limits, cudaStream_t st) {
    const int sms = limits.sms;
    if ((int)tasks.size() > sms) return 0;
    double groups = 0.0, pipes = 0.0, steps = 0.0;
    int most = 0;  // pairs of the largest factor
    for (const BTask &t : tasks) {
        const double m = pw_rows_pad(t.m, t.n), n = t.n + (t.n & 1), half = n / 2;
        const double rows = 0.8 * (7.0 * m + 4.0 * n) / 32.0;
        // columns outside the group's shared memory: read from L2 twice a step
        const int width = t.n < kBucketEdges[2] ? 256 : (t.n < kBucketEdges[3] ? 512 : 1024);
        const double room = (double)kSmemBudget * width / 1024 - (double)pw_aux_bytes(t.n + (t.n & 1));
        const double out = std::max(0.0, 1.0 - room / (double)need_bytes(t.m, t.n));
        const double slow = width == 256 ? std::min(1.35, 1.0 + out) : 1.0 + 0.25 * out;
        groups = std::max(groups, n * (std::max(half, 4.0) * rows * 16.0 * slow + 10200.0));
        pipes += n * half * (rows + 56.0) * 16.0;
        steps += n;
        most = std::max(most, (t.n + 1) / 2);
    }
    const double line = 0.77 * groups;
    const double per_cta = 250.0 * std::max(1.0, 2.0 * (double)tasks.size() / sms);
    double best = 0.0;
    int best_c = 0;
    for (int C : {16, 8, 4, 2, 1}) {
        const ClShape s = cluster_shape(tasks, C);
        if (C > most || C > limits.cluster || s.P > kMaxClPairs || s.smem > kClSmemMax) continue;
        double c_max = 0.0, c_sum = 0.0;
        for (const BTask &t : tasks) {
            const double m = pw_rows_pad(t.m, t.n), n = t.n + (t.n & 1);
            const double turns = ceil(ceil(n / 2 / C) / 4.0);  // pairs per quarter of an SM
            const double c = n * (turns * (0.8 * (7.0 * m + 4.0 * n) / 32.0 + 56.0) * 64.0 + 2000.0);
            c_max = std::max(c_max, c);
            c_sum += c;
        }
        const double bound = best_c ? std::min(line, 0.94 * best) : line;
        double c = std::max(c_max, (pipes + per_cta * C * steps) / sms);
        if (c >= bound) continue;
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr[1];
        int resident = 0;
        if (cluster_config((int)tasks.size(), C, s, st, cfg, attr) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&resident, k_batched_cl, &cfg) != cudaSuccess || resident < 1) {
            cudaGetLastError();
            continue;
        }
        c = std::max(c, c_sum / resident);
        if (c < bound) {
            best = c;
            best_c = C;
        }
    }
    return best_c;
}

void (*batched_kernel(int cta, bool few, bool even))(BArgs, int) {
    if (cta == 512) return few ? k_batched<512, true, false> : k_batched<512, false, false>;
    return few ? (even ? k_batched<1024, true, true> : k_batched<1024, true, false>)
               : (even ? k_batched<1024, false, true> : k_batched<1024, false, false>);
}

// Runs the persistent kernel over `tasks` (already in queue order), or with
// C > 0 one cluster of C CTAs per factor, as one captured graph: counter reset
// + the launch.
cudaError_t run_batch(const std::vector<BTask> &tasks, int max_sweeps, int sort, double tstop, bool use_graph,
                      int grid, int cta, int C, int *res, long long *rot, int *where, cudaStream_t st, float *ms) {
    const int count = (int)tasks.size();
    const int64_t stride = C ? 0 : ws_stride_for(tasks, cta);
    bool few = true;  // every factor has few pairs (pw_solve)
    for (const BTask &t : tasks) few = few && t.n <= kPwFew;
    bool even = cta == 1024 && tasks[0].width < cta;  // one width, narrower than a CTA
    for (const BTask &t : tasks) even = even && t.width == tasks[0].width;
    void (*kern)(BArgs, int) = batched_kernel(cta, few, even);
    const ClShape shape = C ? cluster_shape(tasks, C) : ClShape{};
    auto launch = [&](const BArgs &A, cudaStream_t on) -> cudaError_t {
        if (C) {
            cudaLaunchConfig_t cfg;
            cudaLaunchAttribute attr[1];
            const cudaError_t ce = cluster_config(count, C, shape, on, cfg, attr);
            return ce != cudaSuccess ? ce : cudaLaunchKernelEx(&cfg, k_batched_cl, A, C);
        }
        kern<<<grid, cta, kSmemBudget, on>>>(A, kSmemBudget);
        return cudaGetLastError();
    };
    BTask *d_tasks = nullptr;
    int *d_counter = nullptr;
    double *d_ws = nullptr;
    cudaError_t e = scratch_alloc((void **)&d_tasks, sizeof(BTask) * (size_t)count, st);
    if (e == cudaSuccess) e = scratch_alloc((void **)&d_counter, sizeof(int), st);
    if (e == cudaSuccess) e = scratch_alloc((void **)&d_ws, sizeof(double) * (size_t)grid * stride + 64, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(d_tasks, tasks.data(), sizeof(BTask) * (size_t)count, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBudget);
    BArgs A;
    A.tasks = d_tasks;
    A.count = count;
    A.counter = d_counter;
    A.width = tasks[0].width;
    A.firsts = grid * (cta / A.width);
    A.max_sweeps = max_sweeps;
    A.sort = sort;
    A.tstop = tstop;
    A.ws = d_ws;
    A.ws_stride = stride;
    A.res = res;
    A.rot = rot;
    A.where = where;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (e == cudaSuccess && ms) {
        e = cudaEventCreate(&e0);
        if (e == cudaSuccess) e = cudaEventCreate(&e1);
    }
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    if (e == cudaSuccess && use_graph) {
        // the memset and the launch form the graph; a stream that is itself
        // being captured gets the two nodes directly
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        e = cudaStreamIsCapturing(st, &cs);
        if (e == cudaSuccess && cs != cudaStreamCaptureStatusNone) use_graph = false;
    }
    if (e == cudaSuccess && use_graph) {
        cudaStream_t cap = nullptr;
        e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            cudaMemsetAsync(d_counter, 0, sizeof(int), cap);
            const cudaError_t le = launch(A, cap);
            e = cudaStreamEndCapture(cap, &graph);
            if (e == cudaSuccess) e = le;
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
        if (cap) cudaStreamDestroy(cap);
        if (e == cudaSuccess && ms) e = cudaEventRecord(e0, st);
        if (e == cudaSuccess) e = cudaGraphLaunch(exec, st);
        if (e == cudaSuccess && ms) e = cudaEventRecord(e1, st);
    } else if (e == cudaSuccess) {
        e = cudaMemsetAsync(d_counter, 0, sizeof(int), st);
        if (e == cudaSuccess && ms) e = cudaEventRecord(e0, st);
        if (e == cudaSuccess) e = launch(A, st);
        if (e == cudaSuccess && ms) e = cudaEventRecord(e1, st);
    }
    if (e == cudaSuccess && ms) {
        e = cudaEventSynchronize(e1);
        if (e == cudaSuccess) e = cudaEventElapsedTime(ms, e0, e1);
    }
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (d_tasks) cudaFreeAsync(d_tasks, st);
    if (d_counter) cudaFreeAsync(d_counter, st);
    if (d_ws) cudaFreeAsync(d_ws, st);
    return e;
}

// queue order: width decreasing, then n decreasing, then input order
void order_tasks(std::vector<BTask> &tasks) {
    std::stable_sort(tasks.begin(), tasks.end(), [](const BTask &a, const BTask &b) {
        if (a.width != b.width) return a.width > b.width;
        return a.n > b.n;
    });
}

std::mutex g_tune_mu;
std::map<long long, std::vector<int>> g_tune_cache;  // tune_key -> width per bucket

// Picks the group width of every size bucket present: each candidate width is
// timed on (SMs x 1024 / width) factors of the bucket, two sweeps each, and
// scored by sum(m n^2) / time.  A bucket with fewer factors than the narrowest
// width has groups cannot show what a full GPU does with it and is not timed:
// it takes that width, the fastest per factor or within 1% of it wherever it
// was measured (4000 factors of n in [16, 64]: 256: 46.6 ms, 512: 55.9, 1024:
// 81.2; 2000 of [100, 140]: 390, 398, 426).
// The choice is kept by device, CTA size, buckets present and buckets filled.
long long tune_key(int dev, int cta, const std::vector<BTask> &all, int grid, int *filled) {
    int n[kBuckets] = {}, mask = 0;
    *filled = 0;
    for (const BTask &t : all) ++n[bucket_of(t.n)];
    for (int b = 0; b < kBuckets; ++b) {
        mask |= (n[b] > 0) << b;
        *filled |= (n[b] >= grid * (cta / 256)) << b;
    }
    return ((long long)dev << 32) | ((long long)cta << 16) | (*filled << 8) | mask;
}

cudaError_t tune_widths(const std::vector<BTask> &all, int grid, int cta, int *res, long long *rot, int *where,
                        cudaStream_t st, std::vector<int> &width, float *ms_total) {
    width.assign(kBuckets, 256);
    int dev = 0, filled = 0;
    cudaGetDevice(&dev);
    const long long key = tune_key(dev, cta, all, grid, &filled);
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end()) {
            width = it->second;
            return cudaSuccess;
        }
    }
    for (int b = 0; b < kBuckets; ++b) {
        if (!(filled & (1 << b))) continue;
        std::vector<BTask> members;
        for (const BTask &t : all)
            if (bucket_of(t.n) == b) members.push_back(t);
        double best = -1.0;
        for (int w : {1024, 512, 256}) {
            if (w > cta) continue;
            const size_t want = (size_t)grid * (cta / w);
            std::vector<BTask> sample;
            const size_t stepk = std::max<size_t>(1, members.size() / want);
            for (size_t i = 0; i < members.size() && sample.size() < want; i += stepk) sample.push_back(members[i]);
            double work = 0.0;
            for (BTask &t : sample) {
                t.width = w;
                work += (double)t.m * t.n * t.n;
            }
            order_tasks(sample);
            float ms = 0.f;
            const cudaError_t e = run_batch(sample, 2, 1, 0.0, false, grid, cta, 0, res, rot, where, st, &ms);
            if (e != cudaSuccess) return e;
            if (ms_total) *ms_total += ms;
            const double score = work / std::max(ms, 1e-3f);
            if (score > best) {
                best = score;
                width[b] = w;
            }
        }
    }
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tune_cache[key] = width;
    return cudaSuccess;
}

// The autotuner's widths give the most factors per second of a long queue; in a
// short one a factor solved by a quarter of an SM can outlast all the others.
// A bucket's width doubles while its largest factor at that width (work m n^2,
// cta / width times slower than on a whole SM) would take longer than an SM's
// share of the work of this and the smaller buckets, which the queue holds
// last; up to one warp for every four pairs (more only wait), and never below
// a smaller bucket's width, so that the queue stays largest first.
// Measured (n uniform on [16, 256], kernel, queue at 256 everywhere / at these
// widths / on clusters): 600 factors 387 / 274 ms, 1000: 522 / 460, 300: 296 / 239,
// 40: 247 / 207 / 46, 100: 286 / 239 / 142.
void widen_for_tail(const std::vector<BTask> &tasks, int sms, int cta, std::vector<int> &width) {
    double sum[kBuckets] = {}, most[kBuckets] = {};
    for (const BTask &t : tasks) {
        const double w = (double)t.m * t.n * t.n;
        const int b = bucket_of(t.n);
        sum[b] += w;
        most[b] = std::max(most[b], w);
    }
    double below = 0.0;
    for (int b = 0; b < kBuckets; ++b) {
        below += sum[b];
        int &w = width[(size_t)b];
        const int cap = std::min(cta, b < 2 ? 256 : (b < 3 ? 512 : 1024));
        while (w < cap && most[b] * (cta / w) > below / sms) w *= 2;
        if (b > 0) w = std::max(w, width[(size_t)b - 1]);
    }
}

}  // namespace
}  // namespace hsvd

using namespace hsvd;

extern "C" {

void hsvd_default_batch_opts(hsvd_batch_opts *o) {
    if (!o) return;
    memset(o, 0, sizeof *o);
    o->tol = 0.0;
    o->max_sweeps = 30;
    o->sort = 1;
    o->group_width = 0;
    o->use_graph = 1;
}

int hsvd_solve_batched_ex(int64_t count, const double *const *G, const int64_t *m, const int64_t *n,
                          const int64_t *ldg, const int8_t *const *J, double *const *sigma, double *const *U,
                          double *const *V, int *sweeps, int *status, const hsvd_batch_opts *opts,
                          hsvd_batch_info *info, void *stream) {
    hsvd_batch_opts o;
    if (opts) o = *opts;
    else hsvd_default_batch_opts(&o);
    if (count < 0 || (count > 0 && (!G || !m || !n || !ldg || !J || !sigma))) return HSVD_ERR_ARG;
    if (o.max_sweeps <= 0) o.max_sweeps = 30;
    if (o.group_width != 0 && o.group_width != 256 && o.group_width != 512 && o.group_width != 1024)
        return HSVD_ERR_ARG;
    if (o.cta_threads != 0 && o.cta_threads != 512 && o.cta_threads != 1024) return HSVD_ERR_ARG;
    const int cta = o.cta_threads ? o.cta_threads : 1024;
    if (o.group_width > cta) return HSVD_ERR_ARG;
    if (o.reserved) return HSVD_ERR_ARG;
    if (o.tstop < 0.0) o.tstop = HSVD_TSTOP_PAPER;
    if (!(o.tstop >= 0.0 && o.tstop <= 1.0)) return HSVD_ERR_ARG;
    if (info) memset(info, 0, sizeof *info);
    if (count == 0) return HSVD_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // host arrays: stage through device copies, one copy per matrix
    const bool host = !is_device_ptr(G[0]);
    std::vector<BTask> tasks((size_t)count);
    size_t g_off = 0, j_off = 0, s_off = 0, u_off = 0, v_off = 0;
    for (int64_t k = 0; k < count; ++k) {
        if (n[k] < 1 || m[k] < n[k] || ldg[k] < m[k] || n[k] > 2048 || m[k] > 4096) return HSVD_ERR_ARG;
        if (!G[k] || !J[k] || !sigma[k]) return HSVD_ERR_ARG;
        // all of one kind: host arrays are staged, device arrays used in place
        if (is_device_ptr(G[k]) == host || is_device_ptr(J[k]) == host || is_device_ptr(sigma[k]) == host)
            return HSVD_ERR_ARG;
        if ((U && U[k] && is_device_ptr(U[k]) == host) || (V && V[k] && is_device_ptr(V[k]) == host))
            return HSVD_ERR_ARG;
        if (need_bytes(m[k], n[k]) > (size_t)1 << 30) return HSVD_ERR_ARG;
        BTask &t = tasks[(size_t)k];
        t.m = (int)m[k];
        t.n = (int)n[k];
        t.idx = (int)k;
        t.ldg = host ? m[k] : ldg[k];
        t.ldu = m[k];
        t.ldv = n[k];
        t.tol = o.tol > 0.0 ? o.tol : (double)n[k] * 0x1p-53;
        g_off += (size_t)(m[k] * n[k]);
        j_off += (size_t)n[k];
        s_off += (size_t)n[k];
        if (U && U[k]) u_off += (size_t)(m[k] * n[k]);
        if (V && V[k]) v_off += (size_t)(n[k] * n[k]);
    }
    int rc = HSVD_OK;
    double *dG = nullptr, *dS = nullptr, *dU = nullptr, *dV = nullptr;
    int8_t *dJ = nullptr;
    int *d_res = nullptr, *d_where = nullptr;
    long long *d_rot = nullptr;
    auto fail = [&](int code) {
        if (rc == HSVD_OK) rc = code;
    };
    if (scratch_alloc((void **)&d_res, sizeof(int) * 3 * (size_t)count, st) != cudaSuccess ||
        scratch_alloc((void **)&d_where, sizeof(int) * (size_t)count, st) != cudaSuccess ||
        scratch_alloc((void **)&d_rot, sizeof(long long) * (size_t)count, st) != cudaSuccess)
        fail(HSVD_ERR_NOMEM);
    if (rc == HSVD_OK && host) {
        if (scratch_alloc((void **)&dG, sizeof(double) * g_off + 16, st) != cudaSuccess ||
            scratch_alloc((void **)&dJ, j_off + 16, st) != cudaSuccess ||
            scratch_alloc((void **)&dS, sizeof(double) * s_off + 16, st) != cudaSuccess ||
            scratch_alloc((void **)&dU, sizeof(double) * u_off + 16, st) != cudaSuccess ||
            scratch_alloc((void **)&dV, sizeof(double) * v_off + 16, st) != cudaSuccess)
            fail(HSVD_ERR_NOMEM);
    }
    size_t go = 0, jo = 0, so = 0, uo = 0, vo = 0;
    for (int64_t k = 0; k < count && rc == HSVD_OK; ++k) {
        BTask &t = tasks[(size_t)k];
        if (host) {
            t.G = dG + go;
            t.J = dJ + jo;
            t.sigma = dS + so;
            t.U = (U && U[k]) ? dU + uo : nullptr;
            t.V = (V && V[k]) ? dV + vo : nullptr;
            if (cudaMemcpy2DAsync(dG + go, sizeof(double) * m[k], G[k], sizeof(double) * ldg[k], sizeof(double) * m[k],
                                  n[k], cudaMemcpyHostToDevice, st) != cudaSuccess ||
                cudaMemcpyAsync(dJ + jo, J[k], n[k], cudaMemcpyHostToDevice, st) != cudaSuccess)
                fail(HSVD_ERR_CUDA);
            go += (size_t)(m[k] * n[k]);
            jo += (size_t)n[k];
            so += (size_t)n[k];
            if (t.U) uo += (size_t)(m[k] * n[k]);
            if (t.V) vo += (size_t)(n[k] * n[k]);
        } else {
            t.G = G[k];
            t.J = J[k];
            t.sigma = sigma[k];
            t.U = U ? U[k] : nullptr;
            t.V = V ? V[k] : nullptr;
        }
    }
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int grid = (int)std::min<int64_t>(sms, count);
    std::vector<int> width(kBuckets, o.group_width ? o.group_width : cta);
    float ms_tune = 0.f;
    int tuned = 0;
    const int C = (o.group_width || o.cta_threads) ? 0 : few_clusters(tasks, stream_limits(st), st);
    if (rc == HSVD_OK && o.group_width == 0 && C == 0) {
        std::vector<int> w;
        const bool cached = [&] {
            std::lock_guard<std::mutex> lk(g_tune_mu);
            int filled = 0;
            return g_tune_cache.count(tune_key(dev, cta, tasks, sms, &filled)) > 0;
        }();
        if (tune_widths(tasks, sms, cta, d_res, d_rot, d_where, st, w, &ms_tune) != cudaSuccess) fail(HSVD_ERR_CUDA);
        else width = w;
        tuned = cached ? 2 : 1;
    }
    if (o.group_width == 0 && C == 0) widen_for_tail(tasks, sms, cta, width);
    for (BTask &t : tasks) t.width = width[(size_t)bucket_of(t.n)];
    order_tasks(tasks);
    float ms = 0.f;
    if (rc == HSVD_OK &&
        run_batch(tasks, o.max_sweeps, o.sort ? 1 : 0, o.tstop, o.use_graph != 0, grid, cta, C, d_res, d_rot, d_where,
                  st, &ms) != cudaSuccess)
        fail(HSVD_ERR_CUDA);
    std::vector<int> h_res(3 * (size_t)count, 0), h_where((size_t)count, 0);
    std::vector<long long> h_rot((size_t)count, 0);
    if (rc == HSVD_OK &&
        (cudaMemcpyAsync(h_res.data(), d_res, sizeof(int) * 3 * (size_t)count, cudaMemcpyDeviceToHost, st) !=
             cudaSuccess ||
         cudaMemcpyAsync(h_where.data(), d_where, sizeof(int) * (size_t)count, cudaMemcpyDeviceToHost, st) !=
             cudaSuccess ||
         cudaMemcpyAsync(h_rot.data(), d_rot, sizeof(long long) * (size_t)count, cudaMemcpyDeviceToHost, st) !=
             cudaSuccess))
        fail(HSVD_ERR_CUDA);
    if (rc == HSVD_OK && host) {
        // results back, one copy per array
        size_t so2 = 0, uo2 = 0, vo2 = 0;
        for (int64_t k = 0; k < count && rc == HSVD_OK; ++k) {
            if (cudaMemcpyAsync(sigma[k], dS + so2, sizeof(double) * n[k], cudaMemcpyDeviceToHost, st) != cudaSuccess)
                fail(HSVD_ERR_CUDA);
            so2 += (size_t)n[k];
            if (U && U[k]) {
                if (cudaMemcpyAsync(U[k], dU + uo2, sizeof(double) * m[k] * n[k], cudaMemcpyDeviceToHost, st) !=
                    cudaSuccess)
                    fail(HSVD_ERR_CUDA);
                uo2 += (size_t)(m[k] * n[k]);
            }
            if (V && V[k]) {
                if (cudaMemcpyAsync(V[k], dV + vo2, sizeof(double) * n[k] * n[k], cudaMemcpyDeviceToHost, st) !=
                    cudaSuccess)
                    fail(HSVD_ERR_CUDA);
                vo2 += (size_t)(n[k] * n[k]);
            }
        }
    }
    if (cudaStreamSynchronize(st) != cudaSuccess) fail(HSVD_ERR_CUDA);
    int worst = HSVD_OK;
    if (rc == HSVD_OK) {
        for (int64_t k = 0; k < count; ++k) {
            const int s_k = h_res[3 * (size_t)k];
            if (status) status[k] = s_k;
            if (sweeps) sweeps[k] = h_res[3 * (size_t)k + 1];
            if (s_k < 0 && worst >= 0) worst = s_k;
            else if (s_k == HSVD_NOT_CONVERGED && worst == HSVD_OK) worst = s_k;
        }
        if (info) {
            info->grid = C ? (int)count * C : grid;
            info->cta_threads = C ? 32 * cluster_shape(tasks, C).P : cta;
            info->tuned = tuned;
            for (int b = 0; b < 5; ++b) info->bucket_width[b] = width[(size_t)b];
            info->ms_kernel = ms;
            info->ms_tune = ms_tune;
            info->kernel_launches = 1;
            for (int64_t k = 0; k < count; ++k) {
                info->rotations += h_rot[(size_t)k];
                info->max_sweeps_run = std::max(info->max_sweeps_run, h_res[3 * (size_t)k + 1]);
                info->tangent_stops += h_res[3 * (size_t)k + 2] == HSVD_STOP_TANGENT;
                info->resident[std::min(2, std::max(0, h_where[(size_t)k]))] += 1;
            }
        }
    }
    if (d_res) cudaFreeAsync(d_res, st);
    if (d_where) cudaFreeAsync(d_where, st);
    if (d_rot) cudaFreeAsync(d_rot, st);
    if (dG) cudaFreeAsync(dG, st);
    if (dJ) cudaFreeAsync(dJ, st);
    if (dS) cudaFreeAsync(dS, st);
    if (dU) cudaFreeAsync(dU, st);
    if (dV) cudaFreeAsync(dV, st);
    if (host) cudaStreamSynchronize(st);
    return rc != HSVD_OK ? rc : worst;
}

int hsvd_solve_batched(int64_t count, const double *const *G, const int64_t *m, const int64_t *n, const int64_t *ldg,
                       const int8_t *const *J, double tol, int max_sweeps, double *const *sigma, double *const *U,
                       double *const *V, int *sweeps, int *status, void *stream) {
    hsvd_batch_opts o;
    hsvd_default_batch_opts(&o);
    o.tol = tol;
    o.max_sweeps = max_sweeps;
    return hsvd_solve_batched_ex(count, G, m, n, ldg, J, sigma, U, V, sweeps, status, &o, nullptr, stream);
}

}  // extern "C"
