// hypqr.cu -- the hyperbolic QR factorisation that shortens a wide factor
// (Sec. 1: a G whose transpose is tall is reduced by a hyperbolic QR of G^T,
// and V is premultiplied by the transformation).
//
// A = G^T (n x m, n > m) with signature S = J is reduced by J-orthogonal
// Householder reflectors H = I - beta v v^T S (H^T S H = S on the rows they
// touch) with row interchanges, and columns chosen on the trailing J-Gram
// C = X^T S X (X the trailing rows k.. of the remaining columns) by the
// Bunch-Parlett rule, alpha_bp = (1 + sqrt 17) / 8:
//   1 x 1 when the largest |C_jj| is at least alpha_bp times the largest
//     |C_ij|: that column moves to position k and is reduced to R_kk e_k;
//   2 x 2 otherwise: the columns x, y of the largest |C_ij| move to k, k + 1;
//     z = x + tau y (tau = +-1 so that |z^T S z| = |C_xx + C_yy| + 2 |C_xy|)
//     is reduced at row k, then y's rows k+1.. at row k + 1; R gets a full
//     2 x 2 diagonal block.
// A reduction of z at row r: if S_r is not the sign of gamma = z^T S z (rows
// r..), row r is interchanged with the row of that sign holding the largest
// |z_i| (ties: the smallest i); alpha = -sign(z_r) sqrt|gamma| keeps the
// J-norm, v = z - alpha e_r, beta = 2 / (v^T S v) = 1 / (S_r sqrt|gamma|
// (sqrt|gamma| + |z_r|)).  gamma = 0 means A^T J A is singular: HSVD_ERR_RANK.
//
// On the GPU the trailing J-Gram is kept as an m x m matrix: formed once, and
// after every finished row r downdated by S_r w_r w_r^T (w_r row r of the
// transformed A), since the reflectors and interchanges leave the J-Gram of
// the rows they touch unchanged.  The pivot choice reads it; gamma, tau and the
// reflectors are computed from the columns themselves.  One round per
// reflector: select (one CTA: the next position, pivot, column swaps, z,
// interchange, v, beta), apply (one CTA per column; R's entries of the step),
// downdate (the trailing J-Gram, with per-CTA maxima for the next pivot).  The
// position and phase live on the device; the host launches m rounds.
//
// Afterwards T A C = [R; 0] with T^T Jh T = J (T the product of the
// interchanges and reflectors, Jh the signature after the interchanges), so
// G J G^T = F Jh_1 F^T with the square F = C R^T (m x m), whose HSVD
// F V_F = U Sigma gives V = T^T [V_F; 0]: G V = U Sigma and V^T J V = Jh_1.
#include <cuda_runtime.h>

#include <vector>

#include "hsvd_internal.cuh"

namespace hsvd {
namespace {

constexpr int kSelThreads = 1024;
constexpr int kColThreads = 256;
constexpr int kDownThreads = 256;
constexpr int kDownGrid = 304;
constexpr int kTile = 32;
constexpr size_t kTtSmem = 100 * 1024;  // a column and its signature in shared memory: two CTAs of k_hq_apply_t on an SM

struct HqState {
    int k;      // first column of the current step
    int phase;  // 0: first (or only) reflector of the step, 1: the second of a 2 x 2 step
    int s;      // size of the current step (1 or 2; 0 before the first)
    int r0;     // row of the current reflector
    int bad;    // gamma = 0 (A^T J A singular): HSVD_ERR_RANK
    int done;   // every column reduced
    double alpha;
};

// per-CTA maxima of the trailing J-Gram: |diagonal| with its index, |off-diagonal| with (r, q), r < q
struct HqMax {
    double dmax, omax;
    int di, r, q, pad;
};

__device__ __forceinline__ HqMax hq_none() {
    HqMax m;
    m.dmax = -1.0;
    m.omax = -1.0;
    m.di = m.r = m.q = 0x7fffffff;
    m.pad = 0;
    return m;
}

// The keys (magnitudes, or -1 for none) compare as their bit patterns: the same
// order, without FP64 comparisons, each of which would take a 64-cycle turn of
// its warp on the FP64 pipe.
constexpr long long kInfBits = 0x7FF0000000000000ll;  // above it: NaNs
__device__ __forceinline__ long long hq_bits(double x) { return __double_as_longlong(x); }

__device__ __forceinline__ void hq_merge(HqMax &a, const HqMax &b) {
    if (hq_bits(b.dmax) > hq_bits(a.dmax) || (hq_bits(b.dmax) == hq_bits(a.dmax) && b.di < a.di)) {
        a.dmax = b.dmax;
        a.di = b.di;
    }
    if (hq_bits(b.omax) > hq_bits(a.omax) ||
        (hq_bits(b.omax) == hq_bits(a.omax) && (b.q < a.q || (b.q == a.q && b.r < a.r)))) {
        a.omax = b.omax;
        a.r = b.r;
        a.q = b.q;
    }
}

__device__ __forceinline__ HqMax hq_shfl(const HqMax &a, int o) {
    HqMax b;
    b.dmax = __shfl_xor_sync(0xffffffffu, a.dmax, o);
    b.omax = __shfl_xor_sync(0xffffffffu, a.omax, o);
    b.di = __shfl_xor_sync(0xffffffffu, a.di, o);
    b.r = __shfl_xor_sync(0xffffffffu, a.r, o);
    b.q = __shfl_xor_sync(0xffffffffu, a.q, o);
    b.pad = 0;
    return b;
}

// the maximum entries (i, j >= k) seen by the CTA's threads into its slot
// (NT threads in a 1-D or 2-D block, whole warps)
template <int NT>
__device__ void hq_block_max(HqMax a, HqMax *out) {
    __shared__ HqMax red[NT / 32];
    const int lt = (int)(threadIdx.x + threadIdx.y * blockDim.x);
    for (int o = 16; o > 0; o >>= 1) hq_merge(a, hq_shfl(a, o));
    if ((lt & 31) == 0) red[lt >> 5] = a;
    __syncthreads();
    if (lt == 0) {
        HqMax t = red[0];
        for (int w = 1; w < NT / 32; ++w) hq_merge(t, red[w]);
        *out = t;
    }
}

__device__ __forceinline__ void hq_see(HqMax &a, int i, int j, double v) {
    const long long av = hq_bits(v) & 0x7fffffffffffffffll;
    if (av > kInfBits) return;  // a NaN is no maximum
    if (i == j) {
        if (av > hq_bits(a.dmax) || (av == hq_bits(a.dmax) && i < a.di)) {
            a.dmax = __longlong_as_double(av);
            a.di = i;
        }
    } else if (i < j) {  // the upper triangle stands for both
        if (av > hq_bits(a.omax) || (av == hq_bits(a.omax) && (j < a.q || (j == a.q && i < a.r)))) {
            a.omax = __longlong_as_double(av);
            a.r = i;
            a.q = j;
        }
    }
}

// A (n x m, column-major) = G^T, G m x n (ldg)
__global__ void k_hq_transpose(const double *__restrict__ G, int64_t ldg, int m, int n, double *__restrict__ A) {
    __shared__ double t[kTile][kTile + 1];
    const int i0 = blockIdx.x * kTile, j0 = blockIdx.y * kTile;  // i: row of G (< m), j: column of G (< n)
    for (int y = threadIdx.y; y < kTile; y += blockDim.y) {
        const int i = i0 + threadIdx.x, j = j0 + y;
        t[y][threadIdx.x] = (i < m && j < n) ? G[i + (int64_t)j * ldg] : 0.0;
    }
    __syncthreads();
    for (int y = threadIdx.y; y < kTile; y += blockDim.y) {
        const int j = j0 + threadIdx.x, i = i0 + y;  // A(j, i) = G(i, j)
        if (i < m && j < n) A[j + (int64_t)i * n] = t[threadIdx.x][y];
    }
}

// C = A^T S A (m x m, full symmetric), 32 x 32 tiles, and the per-CTA maxima
__global__ void __launch_bounds__(kTile * 8)
k_hq_gram(const double *__restrict__ A, int n, int m, const int8_t *__restrict__ s, double *__restrict__ C,
          HqMax *__restrict__ mx) {
    __shared__ double ta[kTile][kTile + 1], tb[kTile][kTile + 1];
    const int i0 = blockIdx.x * kTile, j0 = blockIdx.y * kTile;
    const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int r0 = 0; r0 < n; r0 += kTile) {
        for (int y = ty; y < kTile; y += 8) {
            const int r = r0 + tx;
            const double sg = (r < n) ? (double)s[r] : 0.0;
            ta[y][tx] = (r < n && i0 + y < m) ? A[r + (int64_t)(i0 + y) * n] * sg : 0.0;
            tb[y][tx] = (r < n && j0 + y < m) ? A[r + (int64_t)(j0 + y) * n] : 0.0;
        }
        __syncthreads();
        for (int u = 0; u < 4; ++u) {
            const int jy = ty + 8 * u;
#pragma unroll 8
            for (int r = 0; r < kTile; ++r) acc[u] = fma(ta[tx][r], tb[jy][r], acc[u]);
        }
        __syncthreads();
    }
    HqMax a = hq_none();
    for (int u = 0; u < 4; ++u) {
        const int i = i0 + tx, j = j0 + ty + 8 * u;
        if (i < m && j < m) {
            C[i + (int64_t)j * m] = acc[u];
            hq_see(a, i, j, acc[u]);
        }
    }
    hq_block_max<kTile * 8>(a, &mx[blockIdx.x + blockIdx.y * gridDim.x]);
}

// swaps columns a and b of X (rows 0..rows-1, ld)
__device__ void swap_cols(double *X, int64_t ld, int rows, int a, int b) {
    if (a == b) return;
    for (int i = threadIdx.x; i < rows; i += blockDim.x) {
        const double t = X[i + (int64_t)a * ld];
        X[i + (int64_t)a * ld] = X[i + (int64_t)b * ld];
        X[i + (int64_t)b * ld] = t;
    }
}

// Sum over the CTA of one value per thread, in every thread of warp 0: a
// butterfly in each warp, then the warps' sums in order (those past the last
// thread with a value, `count` values in all, are exact zeros and are skipped).
// V values at once, value v in lane v of warp 0 of the ordered sums.
template <int V>
__device__ __forceinline__ double hq_cta_sums(const double (&x)[V], double (*red)[4], int count) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nw = min((count + 31) / 32, kSelThreads / 32);
    if (warp < nw) {
#pragma unroll
        for (int v = 0; v < V; ++v) {
            double y = x[v];
            for (int o = 16; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
            if (lane == 0) red[warp][v] = y;
        }
    }
    __syncthreads();
    double t = 0.0;
    if (warp == 0 && lane < V)
        for (int w = 0; w < nw; ++w) t += red[w][lane];
    return t;
}

// One reflector's set-up (one CTA): the state's next position; at phase 0 the
// pivot choice and column swaps of a new step, then z, gamma, the row
// interchange, v and beta.  A chain of reductions: what can be compared as
// integers is, the FP64 sums run on the warps that hold values only, and the
// square root and quotients on one warp (each FP64 instruction of 32 warps
// would take the SM's pipe 500 cycles).  Measured at 400 x 900: 32 us a launch
// with every thread in every step, 15 us so.
__global__ void __launch_bounds__(kSelThreads)
k_hq_select(double *__restrict__ A, int n, int m, int8_t *__restrict__ s, double *__restrict__ C,
            const HqMax *__restrict__ mx, int nmx, int *__restrict__ cperm, double *__restrict__ z,
            double *__restrict__ Vr, double *__restrict__ beta, int *__restrict__ rswap, int8_t *__restrict__ bsize,
            HqState *__restrict__ st) {
    __shared__ double red[kSelThreads / 32][4];
    __shared__ HqMax mred[kSelThreads / 32];
    __shared__ int s_choice[3];
    __shared__ double s_sc[4];  // gamma, tau, alpha
    __shared__ long long s_best[kSelThreads / 32];
    __shared__ int s_bi[kSelThreads / 32], s_ip;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (st->done || st->bad) return;
    // where the last round left off
    int k = st->k, phase = st->phase;
    const int ls = st->s;
    __syncthreads();
    if (ls == 1 || (ls == 2 && phase == 1)) {
        k += ls;
        phase = 0;
    } else if (ls == 2) {
        phase = 1;
    }
    if (tid == 0) {
        st->k = k;
        st->phase = phase;
    }
    int sz = ls;
    if (phase == 0) {
        if (k >= m) {
            if (tid == 0) {
                st->done = 1;
                st->s = 0;
            }
            return;
        }
        // pivot choice on the trailing J-Gram
        const int mw = min((nmx + 31) / 32, kSelThreads / 32);  // warps with maxima
        if (warp < mw) {
            HqMax a = hq_none();
            for (int i = tid; i < nmx; i += kSelThreads) hq_merge(a, mx[i]);
            for (int o = 16; o > 0; o >>= 1) hq_merge(a, hq_shfl(a, o));
            if (lane == 0) mred[warp] = a;
        }
        __syncthreads();
        if (warp == 0) {
            HqMax t = lane < mw ? mred[lane] : hq_none();
            for (int o = 16; o > 0; o >>= 1) hq_merge(t, hq_shfl(t, o));
            if (lane == 0) {
                const double alpha_bp = (1.0 + sqrt(17.0)) / 8.0;
                if (k == m - 1 || !(t.omax > 0.0) || t.dmax >= alpha_bp * t.omax) {
                    s_choice[0] = (t.di >= k && t.di < m) ? 1 : 0;
                    s_choice[1] = t.di;
                } else {
                    s_choice[0] = (t.r >= k && t.q < m && t.r < t.q) ? 2 : 0;
                    s_choice[1] = t.r;
                    s_choice[2] = t.q;
                }
            }
        }
        __syncthreads();
        sz = s_choice[0];
        if (sz == 0) {  // no finite pivot left
            if (tid == 0) st->bad = 1;
            return;
        }
        // columns to positions k (and k + 1): W, the rows and columns of C, the permutation
        auto swap_both = [&](int a0, int b0) {
            swap_cols(A, n, n, a0, b0);
            swap_cols(C, m, m, a0, b0);
            __syncthreads();
            if (a0 != b0)
                for (int j = tid; j < m; j += kSelThreads) {
                    const double t = C[a0 + (int64_t)j * m];
                    C[a0 + (int64_t)j * m] = C[b0 + (int64_t)j * m];
                    C[b0 + (int64_t)j * m] = t;
                }
            if (tid == 0 && a0 != b0) {
                const int t = cperm[a0];
                cperm[a0] = cperm[b0];
                cperm[b0] = t;
            }
            __syncthreads();
        };
        if (sz == 1) {
            swap_both(k, s_choice[1]);
        } else {
            const int pr = s_choice[1], pq = s_choice[2];
            swap_both(k, pr);
            swap_both(k + 1, pq == k ? pr : pq);
        }
        const double *x = A + (int64_t)k * n, *y = A + (int64_t)(k + 1) * n;
        double tau = 0.0;
        if (sz == 2) {
            // tau from the J-norms and J-product of x and y over rows k..
            double g[3] = {0.0, 0.0, 0.0};
            if (warp * 32 < n - k)
                for (int i = k + tid; i < n; i += kSelThreads) {
                    const double sg = (double)s[i], xi = x[i], yi = y[i], sx = sg * xi;
                    g[0] = fma(sx, xi, g[0]);
                    g[1] = fma(sg * yi, yi, g[1]);
                    g[2] = fma(sx, yi, g[2]);
                }
            const double t = hq_cta_sums<3>(g, red, n - k);
            if (warp == 0) {
                const double a0 = __shfl_sync(0xffffffffu, t, 0), a1 = __shfl_sync(0xffffffffu, t, 1),
                             a2 = __shfl_sync(0xffffffffu, t, 2);
                if (lane == 0) s_sc[1] = ((a0 + a1 >= 0.0) == (a2 >= 0.0)) ? 1.0 : -1.0;
            }
            __syncthreads();
            tau = s_sc[1];
        }
        for (int i = tid; i < n; i += kSelThreads) z[i] = i < k ? 0.0 : (sz == 2 ? fma(tau, y[i], x[i]) : x[i]);
        if (tid == 0) {
            st->s = sz;
            st->r0 = k;
            bsize[k] = (int8_t)sz;
            if (sz == 2) bsize[k + 1] = 0;
        }
    } else {
        // the second reflector of a 2 x 2 step: y's rows k + 1..
        const double *y = A + (int64_t)(k + 1) * n;
        for (int i = tid; i < n; i += kSelThreads) z[i] = i <= k ? 0.0 : y[i];
        if (tid == 0) st->r0 = k + 1;
    }
    __syncthreads();
    const int r0 = phase == 0 ? k : k + 1;
    // gamma = z^T S z over rows r0..
    double gs[1] = {0.0};
    if (warp * 32 < n - r0)
        for (int i = r0 + tid; i < n; i += kSelThreads) gs[0] = fma((double)s[i] * z[i], z[i], gs[0]);
    const double gsum = hq_cta_sums<1>(gs, red, n - r0);
    if (tid == 0) s_sc[0] = gsum;
    __syncthreads();
    const double gamma = s_sc[0];
    const long long gb = hq_bits(gamma);
    if ((gb & 0x7fffffffffffffffll) == 0) {
        if (tid == 0) st->bad = 1;
        return;
    }
    const int sg = gb > 0 && gb <= kInfBits ? 1 : -1;
    // the row interchange when S_r0 is not the sign of gamma: the row of that
    // sign with the largest |z_i|, ties to the smallest i
    if (s[r0] != sg) {
        long long best = -1;
        int bi = 0x7fffffff;
        for (int i = r0 + 1 + tid; i < n; i += kSelThreads) {
            const long long az = hq_bits(z[i]) & 0x7fffffffffffffffll;
            if (s[i] == sg && az <= kInfBits && (az > best || (az == best && i < bi))) {
                best = az;
                bi = i;
            }
        }
        auto reduce = [&]() {
            for (int o = 16; o > 0; o >>= 1) {
                const long long ob = __shfl_xor_sync(0xffffffffu, best, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (ob > best || (ob == best && oi < bi)) {
                    best = ob;
                    bi = oi;
                }
            }
        };
        reduce();
        if (lane == 0) {
            s_best[warp] = best;
            s_bi[warp] = bi;
        }
        __syncthreads();
        if (warp == 0) {
            best = s_best[lane];
            bi = s_bi[lane];
            reduce();
            if (lane == 0) s_ip = (bi > r0 && bi < n) ? bi : -1;
        }
        __syncthreads();
        const int ip = s_ip;
        if (ip < 0) {
            if (tid == 0) st->bad = 1;
            return;
        }
        for (int j = tid; j < m; j += kSelThreads) {
            const double t = A[r0 + (int64_t)j * n];
            A[r0 + (int64_t)j * n] = A[ip + (int64_t)j * n];
            A[ip + (int64_t)j * n] = t;
        }
        if (tid == 0) {
            const double tz = z[r0];
            z[r0] = z[ip];
            z[ip] = tz;
            const int8_t ts = s[r0];
            s[r0] = s[ip];
            s[ip] = ts;
            rswap[r0] = ip;
        }
    } else if (tid == 0) {
        rswap[r0] = r0;
    }
    __syncthreads();
    // alpha, v (zero above r0) and beta
    if (warp == 0) {
        const double root = sqrt(fabs(gamma)), zr = z[r0];
        const double alpha = zr >= 0.0 ? -root : root;
        if (lane == 0) {
            const double vsv = 2.0 * (double)s[r0] * root * (root + fabs(zr));
            s_sc[2] = alpha;
            st->alpha = alpha;
            beta[r0] = 2.0 / vsv;
            Vr[(int64_t)r0 * n + r0] = zr - alpha;
        }
    }
    double *v = Vr + (int64_t)r0 * n;
    for (int i = tid; i < n; i += kSelThreads)
        if (i != r0) v[i] = i < r0 ? 0.0 : z[i];
}

// y <- y - beta (v^T S y) v over rows r0.. for every column c >= k (one CTA per
// column), then R's entries of the step: the reduced columns' rows below them
// are alpha and zeros
__global__ void __launch_bounds__(kColThreads)
k_hq_apply(double *__restrict__ A, int n, int m, const int8_t *__restrict__ s, const double *__restrict__ Vr,
           const double *__restrict__ beta, const HqState *__restrict__ st) {
    __shared__ double red[kColThreads / 32];
    if (st->done || st->bad) return;
    const int k = st->k, r0 = st->r0, sz = st->s, ph = st->phase;
    const int c = k + (int)blockIdx.x;
    if (c >= m) return;
    double *y = A + (int64_t)c * n;
    const int tid = threadIdx.x;
    // column c ends as alpha at row `top` and zeros below (c = k of a 1 x 1 step,
    // c = k + 1 of a finished 2 x 2 one); its other rows are not touched here
    if ((sz == 1 && c == k) || (sz == 2 && ph == 1 && c == k + 1)) {
        for (int i = r0 + tid; i < n; i += kColThreads) y[i] = i == r0 ? st->alpha : 0.0;
        return;
    }
    const double *v = Vr + (int64_t)r0 * n;
    double d = 0.0;
    for (int i = r0 + tid; i < n; i += kColThreads) d = fma((double)s[i] * v[i], y[i], d);
    for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    if ((tid & 31) == 0) red[tid >> 5] = d;
    __syncthreads();
    if (tid < 32) {
        double t = tid < kColThreads / 32 ? red[tid] : 0.0;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (tid == 0) red[0] = t;
    }
    __syncthreads();
    const double f = beta[r0] * red[0];
    const bool cut = sz == 2 && ph == 1 && c == k;  // the block's first column: zeros below row k + 1
    for (int i = r0 + tid; i < n; i += kColThreads) y[i] = cut && i > r0 ? 0.0 : fma(-f, v[i], y[i]);
}

// the trailing J-Gram without the finished rows: C_ij -= S_r A(r, i) A(r, j),
// i, j >= first remaining column; per-CTA maxima of the new trailing block
__global__ void __launch_bounds__(kDownThreads)
k_hq_downdate(const double *__restrict__ A, int n, int m, const int8_t *__restrict__ s, double *__restrict__ C,
              const HqState *__restrict__ st, HqMax *__restrict__ mx) {
    // the step's rows, once its last reflector is applied
    const int nr = st->done || st->bad ? 0 : (st->s == 1 ? 1 : (st->phase == 1 ? 2 : 0));
    HqMax a = hq_none();
    if (nr > 0) {
        const int r = st->k, c0 = r + nr, nt = m - c0;
        const double s0 = (double)s[r], s1 = nr == 2 ? (double)s[r + 1] : 0.0;
        const int64_t total = (int64_t)nt * nt;
        for (int64_t e = (int64_t)blockIdx.x * kDownThreads + threadIdx.x; e < total;
             e += (int64_t)gridDim.x * kDownThreads) {
            const int i = c0 + (int)(e % nt), j = c0 + (int)(e / nt);
            double v = C[i + (int64_t)j * m];
            v = fma(-s0 * A[r + (int64_t)i * n], A[r + (int64_t)j * n], v);
            if (nr == 2) v = fma(-s1 * A[r + 1 + (int64_t)i * n], A[r + 1 + (int64_t)j * n], v);
            C[i + (int64_t)j * m] = v;
            hq_see(a, i, j, v);
        }
    }
    hq_block_max<kDownThreads>(a, &mx[blockIdx.x]);
}

// F (m x m) = C R^T: F(cperm[j], l) = R(l, j), R the block upper triangle of A's first m rows
__global__ void k_hq_form_f(const double *__restrict__ A, int n, int m, const int *__restrict__ cperm,
                            const int8_t *__restrict__ bsize, double *__restrict__ F) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)m * m) return;
    const int l = (int)(e % m), j = (int)(e / m);
    const bool in_r = l <= j || (l == j + 1 && bsize[j] == 2);
    F[cperm[j] + (int64_t)l * m] = in_r ? A[l + (int64_t)j * n] : 0.0;
}

// X (n x m, ldx) <- T^T X: for every step k from the last to the first, H_k^T X
// = X - beta_k S v_k (v_k^T X) with the signature S of step k (recovered from
// the final one by undoing the later interchanges), then the row interchange of
// step k.  A column needs nothing of the others: one CTA per column does all
// the steps, the column and the signature in shared memory, or for more rows
// than fit the column in place and the signature in column j of `work` (n x m).
// Bound by the FP64 pipe (the reductions as much as the column itself).
// Measured, 400 columns of 900 rows: 1.6 ms; with a launch per step and one for
// its signature 4.2 ms and 800 launches' gaps.  In place, the whole call on 200
// columns of 14000 rows: 35.0 ms, against 45.6.
template <bool SMEM>
__global__ void __launch_bounds__(kColThreads)
k_hq_apply_t(double *__restrict__ X, int64_t ldx, int n, int m, const double *__restrict__ Vr,
             const double *__restrict__ beta, const int *__restrict__ rswap, const int8_t *__restrict__ s_end,
             double *__restrict__ work) {
    extern __shared__ __align__(16) double sm[];
    __shared__ double red[2][kColThreads / 32];
    const int j = blockIdx.x, tid = threadIdx.x;
    double *x = X + (int64_t)j * ldx;
    double *y = SMEM ? sm : x;
    int8_t *s = reinterpret_cast<int8_t *>(SMEM ? sm + n : work + (int64_t)j * n);
    for (int i = tid; i < n; i += kColThreads) {
        if (SMEM) y[i] = x[i];
        s[i] = s_end[i];
    }
    __syncthreads();
    for (int k = m - 1; k >= 0; --k) {
        const double *v = Vr + (int64_t)k * n;
        const double b = beta[k];
        const int ip = rswap[k];
        double d = 0.0;
        for (int i = k + tid; i < n; i += kColThreads) d = fma(v[i], y[i], d);
        for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        if ((tid & 31) == 0) red[k & 1][tid >> 5] = d;
        __syncthreads();
        // the warps' sums by a butterfly, in every warp
        double t = red[k & 1][tid & (kColThreads / 32 - 1)];
        for (int o = kColThreads / 64; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        const double f = b * t;
        for (int i = k + tid; i < n; i += kColThreads) y[i] = fma(s[i] > 0 ? -f : f, v[i], y[i]);
        if (ip != k) {  // the same in every thread
            __syncthreads();
            if (tid == 0) {
                const double u = y[k];
                y[k] = y[ip];
                y[ip] = u;
                const int8_t w = s[k];
                s[k] = s[ip];
                s[ip] = w;
            }
        }
        __syncthreads();
    }
    if (SMEM)
        for (int i = tid; i < n; i += kColThreads) x[i] = y[i];
}

// V (n x m, ldv) <- [V_F; 0]
__global__ void k_hq_embed(const double *__restrict__ VF, int m, int n, double *__restrict__ V, int64_t ldv) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)n * m) return;
    const int i = (int)(e % n), j = (int)(e / n);
    V[i + (int64_t)j * ldv] = i < m ? VF[i + (int64_t)j * m] : 0.0;
}

}  // namespace

size_t hypqr_state_bytes() { return sizeof(HqState); }
// per-CTA maxima: the Gram's tiles or the downdate's CTAs, whichever is more
size_t hypqr_mx_bytes(int64_t m) {
    const int64_t tiles = ((m + kTile - 1) / kTile) * ((m + kTile - 1) / kTile);
    return sizeof(HqMax) * (size_t)(tiles > kDownGrid ? tiles : kDownGrid);
}

// The hyperbolic QR of A = G^T (G m x n, m < n) and F = C R^T.  Outputs, all
// device: F (m x m), Jh (n signs after the interchanges; Jh_1 = the first m);
// the reflectors stay in the workspace `hq` for hypqr_apply_tt.  Returns
// HSVD_OK, HSVD_ERR_RANK or HSVD_ERR_CUDA.
int hypqr_factor(const double *G, int64_t m64, int64_t n64, int64_t ldg, const int8_t *J, HypQr &hq, double *F,
                 cudaStream_t st, long long *launches) {
    const int m = (int)m64, n = (int)n64;
    HqState *state = static_cast<HqState *>(hq.state);
    HqMax *mx = static_cast<HqMax *>(hq.mx);
    auto ck = [](cudaError_t e) { return e == cudaSuccess; };
    std::vector<int> p((size_t)m);
    for (int j = 0; j < m; ++j) p[(size_t)j] = j;
    HqState s0 = {};
    if (!ck(cudaMemcpyAsync(hq.cperm, p.data(), sizeof(int) * m, cudaMemcpyHostToDevice, st)) ||
        !ck(cudaMemcpyAsync(state, &s0, sizeof s0, cudaMemcpyHostToDevice, st)) ||
        !ck(cudaMemcpyAsync(hq.s, J, (size_t)n, cudaMemcpyDeviceToDevice, st)) ||
        !ck(cudaMemsetAsync(hq.Vr, 0, sizeof(double) * (size_t)n * m, st)))
        return HSVD_ERR_CUDA;
    k_hq_transpose<<<dim3((m + kTile - 1) / kTile, (n + kTile - 1) / kTile), dim3(kTile, 8), 0, st>>>(G, ldg, m, n,
                                                                                                     hq.A);
    const dim3 gg((m + kTile - 1) / kTile, (m + kTile - 1) / kTile);
    const int nmx0 = (int)(gg.x * gg.y);  // the Gram's maxima, one per tile (hypqr_mx_bytes)
    k_hq_gram<<<gg, dim3(kTile, 8), 0, st>>>(hq.A, n, m, hq.s, hq.C, mx);
    if (!ck(cudaGetLastError())) return HSVD_ERR_CUDA;
    long long nl = 2;
    // m rounds, one reflector each
    for (int r = 0; r < m; ++r) {
        k_hq_select<<<1, kSelThreads, 0, st>>>(hq.A, n, m, hq.s, hq.C, mx, r == 0 ? nmx0 : kDownGrid, hq.cperm, hq.z,
                                               hq.Vr, hq.beta, hq.rswap, hq.bsize, state);
        k_hq_apply<<<m, kColThreads, 0, st>>>(hq.A, n, m, hq.s, hq.Vr, hq.beta, state);
        k_hq_downdate<<<kDownGrid, kDownThreads, 0, st>>>(hq.A, n, m, hq.s, hq.C, state, mx);
        if (!ck(cudaGetLastError())) return HSVD_ERR_CUDA;
        nl += 3;
    }
    k_hq_form_f<<<(unsigned)(((int64_t)m * m + 255) / 256), 256, 0, st>>>(hq.A, n, m, hq.cperm, hq.bsize, F);
    HqState fin = {};
    if (!ck(cudaGetLastError()) || !ck(cudaMemcpyAsync(&fin, state, sizeof fin, cudaMemcpyDeviceToHost, st)) ||
        !ck(cudaStreamSynchronize(st)))
        return HSVD_ERR_CUDA;
    if (launches) *launches += nl + 1;
    if (fin.bad) return HSVD_ERR_RANK;
    // m rounds reduce m columns: the last one finished its step
    return fin.done || (fin.k + fin.s >= m && (fin.s == 1 || fin.phase == 1)) ? HSVD_OK : HSVD_ERR_CUDA;
}

// V (n x m, ldv) <- T^T [V_F; 0], V_F (m x m): the reflectors in reverse order,
// each with the signature of its step (recovered from the final one by
// undoing the later interchanges; hq.A may be written).
int hypqr_apply_tt(HypQr &hq, int64_t m64, int64_t n64, const double *VF, double *V, int64_t ldv, cudaStream_t st,
                   long long *launches) {
    const int m = (int)m64, n = (int)n64;
    k_hq_embed<<<(unsigned)(((int64_t)n * m + 255) / 256), 256, 0, st>>>(VF, m, n, V, ldv);
    const size_t smem = (size_t)n * (sizeof(double) + 1);
    if (smem <= kTtSmem) {
        if (cudaFuncSetAttribute(k_hq_apply_t<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTtSmem) !=
            cudaSuccess)
            return HSVD_ERR_CUDA;
        k_hq_apply_t<true><<<m, kColThreads, smem, st>>>(V, ldv, n, m, hq.Vr, hq.beta, hq.rswap, hq.s, nullptr);
    } else {  // A's columns are free: R is in F
        k_hq_apply_t<false><<<m, kColThreads, 0, st>>>(V, ldv, n, m, hq.Vr, hq.beta, hq.rswap, hq.s, hq.A);
    }
    if (launches) *launches += 2;
    return cudaGetLastError() == cudaSuccess ? HSVD_OK : HSVD_ERR_CUDA;
}

}  // namespace hsvd
