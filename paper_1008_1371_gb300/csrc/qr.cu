// qr.cu -- the shortening front end for tall factors (Sec. 1): G = Q R by
// Householder reflections, the HSVD of the square R, and U = Q [U_R; 0].
// R V = U_R Sigma gives G V = Q R V = (Q [U_R; 0]) Sigma with the same J-unitary
// V, and Householder QR is column-wise backward stable, so relative accuracy
// for column-scaled factors carries over.  One sweep of the blocked method on
// the m x n factor costs 2 n^2 (4m + 2n) flops, on R 12 n^3; the QR and the
// application of Q cost about 4 m n^2 once.
//
// Blocked QR with panels of width kQB (compact WY form, H_1 ... H_w =
// I - V T V^T, T upper triangular):
//   k_qr_panel_cl  factors one panel column by column on a 16-CTA cluster
//                (reflector as in LAPACK's dlarfg: beta = -sign(alpha) ||x||,
//                tau = (beta - alpha) / beta, v = x / (alpha - beta) below the
//                unit diagonal); k_qr_panel, one CTA, for fewer than 32 rows.
//   k_qr_vtc     partial products V^T [V C] over row splits (C: the trailing
//                columns, or U when Q is applied; V for T).
//   k_qr_sum     Y = V^T V, the sum of its partials.
//   k_qr_tbuild  T from tau and Y (T_jj = tau_j,
//                T_{0:j,j} = -tau_j T_{0:j,0:j} V_{:,0:j}^T v_j).
//   k_qr_tz      Z = op(T) (sum of the partials of C): op = T^T for the
//                factorisation (Q^T C), T for applying Q.
//   k_qr_update  C -= V Z.
// Every product is an FP64 FMA chain (the library is compiled without
// floating-point contraction).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "hsvd_internal.cuh"

namespace cg = cooperative_groups;

namespace hsvd {
namespace {

constexpr int kQB = 32;         // panel width
constexpr int kPanelThreads = 256;
constexpr int kVtcThreads = 256;
constexpr int kVtcRows = 32;    // rows per shared-memory slice

// V's entry (i, a) for the panel starting at column j0: zero above the
// diagonal, one on it, the stored reflector below
__device__ __forceinline__ double v_entry(const double *__restrict__ A, int64_t lda, int64_t i, int j0, int a) {
    const int64_t d = (int64_t)j0 + a;
    if (i < d) return 0.0;
    if (i == d) return 1.0;
    return A[i + d * lda];
}

// One CTA factors columns j0 .. j0 + w - 1 of A over rows j0 .. m - 1.  For
// column j: one pass forms x^T x and x^T a_c over the rows below j for the
// later panel columns c, a block reduction gives beta, tau and w_c = v^T a_c,
// and a second pass stores v and updates the later columns.
__global__ void __launch_bounds__(kPanelThreads)
k_qr_panel(double *__restrict__ A, int64_t lda, int64_t m, int j0, int w, double *__restrict__ tau) {
    __shared__ double red[kPanelThreads / 32][kQB];
    __shared__ double sw[kQB];   // w_c of the current column
    __shared__ double s_scale, s_tau;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int jj = 0; jj < w; ++jj) {
        const int64_t j = (int64_t)j0 + jj;
        const double *x = A + j * lda;
        // pass A: acc[0] = sum x_i^2, acc[c] = sum x_i a_{i, j + c} (rows i > j)
        double acc[kQB];
#pragma unroll
        for (int c = 0; c < kQB; ++c) acc[c] = 0.0;
        for (int64_t i = j + 1 + tid; i < m; i += kPanelThreads) {
            const double xi = x[i];
            double val[kQB];
#pragma unroll
            for (int c = 1; c < kQB; ++c)
                if (jj + c < w) val[c] = A[i + (j + c) * lda];
            acc[0] = fma(xi, xi, acc[0]);
#pragma unroll
            for (int c = 1; c < kQB; ++c)
                if (jj + c < w) acc[c] = fma(xi, val[c], acc[c]);
        }
#pragma unroll
        for (int c = 0; c < kQB; ++c) {
            double v = acc[c];
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0) red[warp][c] = v;
        }
        __syncthreads();
        if (tid < kQB) {
            double s = 0.0;
            for (int q = 0; q < kPanelThreads / 32; ++q) s += red[q][tid];
            red[0][tid] = s;  // warp 0's row is read only below, after the barrier
        }
        __syncthreads();
        if (tid == 0) {
            const double alpha = x[j], xnorm2 = red[0][0];
            double t = 0.0, scale = 0.0, beta = alpha;
            if (xnorm2 > 0.0) {
                beta = -copysign(sqrt(fma(alpha, alpha, xnorm2)), alpha);
                t = (beta - alpha) / beta;
                scale = 1.0 / (alpha - beta);
            }
            s_tau = t;
            s_scale = scale;
            tau[j] = t;
            A[j + j * lda] = beta;
        }
        __syncthreads();
        const double t = s_tau, scale = s_scale;
        if (tid > 0 && tid < kQB && jj + tid < w) {
            const int c = tid;  // w_c = a_{j, j+c} + scale * sum_{i>j} x_i a_{i, j+c}
            sw[c] = fma(scale, red[0][c], A[j + (j + c) * lda]);
        }
        __syncthreads();
        // pass B: v below the diagonal, then a_c -= tau w_c v for the later
        // columns; a row's loads are all issued before its stores
        double *xm = A + j * lda;
        for (int64_t i = j + 1 + tid; i < m; i += kPanelThreads) {
            const double vi = xm[i] * scale;
            double val[kQB];
#pragma unroll
            for (int c = 1; c < kQB; ++c)
                if (jj + c < w) val[c] = A[i + (j + c) * lda];
            xm[i] = vi;
#pragma unroll
            for (int c = 1; c < kQB; ++c)
                if (jj + c < w) A[i + (j + c) * lda] = fma(-t * sw[c], vi, val[c]);
        }
        if (tid > 0 && tid < kQB && jj + tid < w) {  // row j: v_j = 1
            double *ac = A + (j + tid) * lda;
            ac[j] = fma(-t, sw[tid], ac[j]);
        }
        __syncthreads();
    }
}

constexpr int kPanelCl = 16;
constexpr int kPanelClMaxRows = 832;  // rows per CTA kept in shared memory: 32 x 832 doubles = 208 KB

// Sums over the warp of N values a lane carries, v[i] of every lane: a butterfly
// (xor 16, 8, 4, 2, 1) that halves the values a lane carries at each level while
// it can, 31 adds for 32 values and 6 for 4.  Returns the sum of value
// warp_sums_index<N>(lane).
template <int N, int O>
__device__ __forceinline__ double warp_sums(double *v, int lane) {
    constexpr int H = (N + 1) / 2;
    const bool hi = lane & O;
#pragma unroll
    for (int i = 0; i < H; ++i) {
        if (i + H < N) {
            const double send = hi ? v[i] : v[i + H], keep = hi ? v[i + H] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
        } else {
            v[i] = v[i] + __shfl_xor_sync(0xffffffffu, v[i], O);
        }
    }
    if constexpr (O > 1) return warp_sums<H, O / 2>(v, lane);
    else return v[0];
}
template <int N, int O = 16>
__device__ __forceinline__ int warp_sums_index(int lane) {
    constexpr int H = (N + 1) / 2;
    int i = 0;
    if constexpr (O > 1) i = warp_sums_index<H, O / 2>(lane);
    return (lane & O) && i + H < N ? i + H : i;
}

// Two parts of a column step of k_qr_panel_cl over a thread's rows (first + tid,
// + 256, ...), for the columns from C0 on: the warp's dots of x with them into
// sums[C0 ..], and their update.  C0, the step's column rounded down to four, is
// a template argument because an FP64 instruction that is predicated off occupies
// the pipe like one that is not.
template <int C0, class Col>
__device__ __forceinline__ void panel_dots(Col col, int jj, int w, int first, int nrows, int lane, double *sums) {
    constexpr int N = kQB - C0;
    double acc[N];
#pragma unroll
    for (int c = 0; c < N; ++c) acc[c] = 0.0;
    const double *x = col(jj);
    for (int i = first; i < nrows; i += kPanelThreads) {
        const double xi = x[i];
        double v[N];
#pragma unroll
        for (int c = 0; c < N; ++c) v[c] = col(C0 + c < w ? C0 + c : jj)[i];
#pragma unroll
        for (int c = 0; c < N; ++c) acc[c] = fma(xi, v[c], acc[c]);
    }
    const double s = warp_sums<N, 16>(acc, lane);
    sums[C0 + warp_sums_index<N>(lane)] = s;
}
template <int C0, class Col>
__device__ __forceinline__ void panel_update(Col col, int jj, int w, int first, int nrows, double scale,
                                             const double *f) {
    constexpr int N = kQB - C0;
    double *x = col(jj);
    for (int i = first; i < nrows; i += kPanelThreads) {
        const double v = x[i] * scale;
        double a[N];
#pragma unroll
        for (int c = 0; c < N; ++c) a[c] = col(C0 + c < w ? C0 + c : jj)[i];
        x[i] = v;
#pragma unroll
        for (int c = 0; c < N; ++c) {
            const double r = fma(f[C0 + c], v, a[c]);
            if (C0 + c > jj && C0 + c < w) col(C0 + c)[i] = r;
        }
    }
}

// The same panel factorisation on a cluster of kPanelCl CTAs: CTA r owns rows
// j0 + r rp .. j0 + (r+1) rp - 1, kept in shared memory (column-major, stride
// rp) when SMEM, else worked on in place in A.  Per column, every CTA reduces
// its rows' part of x^T x and x^T a_c and writes it, with the diagonal row
// when it owns it, into every CTA (double-buffered by column parity); after
// one cluster barrier every CTA sums the same partials in the same order,
// forms beta, tau, w_c itself (warp 0: a column per lane, the two quotients side
// by side) and updates its own rows.  Bound by the FP64 pipe of the 16 SMs, two
// FMAs per entry of the trailing panel and column, about half of a column's
// cycles at 8192 rows; the rest is the chain of sums (8 warps, then 16 CTAs),
// square root and quotient, and the cluster barrier.  Measured at 8192 rows:
// 0.53 ms a panel with finished columns predicated off and the scalars on one
// thread between CTA barriers, 0.33 ms now, the same bits.
template <bool SMEM>
__global__ void __launch_bounds__(kPanelThreads)
k_qr_panel_cl(double *__restrict__ A, int64_t lda, int64_t m, int j0, int w, int rp, double *__restrict__ tau) {
    extern __shared__ __align__(16) double P[];  // [kQB][rp] when SMEM
    __shared__ double red[2][kPanelCl][kQB];     // partial sums from every CTA
    __shared__ double drow[2][kQB];              // the diagonal row of the column
    __shared__ double wred[kPanelThreads / 32][kQB];
    __shared__ double s_scale, sf[kQB];          // the column's scale; -tau w_c
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t row0 = (int64_t)j0 + (int64_t)rank * rp;
    const int64_t left = m - row0;
    const int nrows = left <= 0 ? 0 : (left < rp ? (int)left : rp);
    double *const Ab = A + row0 + (int64_t)j0 * lda;
    auto col = [&](int c) -> double * { return SMEM ? P + c * rp : Ab + (int64_t)c * lda; };
    if (SMEM)
        for (int e = tid; e < kQB * rp; e += kPanelThreads) {
            const int c = e / rp, i = e % rp;
            P[e] = (c < w && i < nrows) ? Ab[i + (int64_t)c * lda] : 0.0;
        }
    cluster.sync();  // every CTA loaded and running before any remote write
    for (int jj = 0; jj < w; ++jj) {
        const int buf = jj & 1;
        // local rows strictly below the diagonal row j0 + jj
        const int64_t below = (int64_t)j0 + jj + 1 - row0;
        const int first = (below <= 0 ? 0 : (below < rp ? (int)below : rp)) + tid;
        switch (jj / 4) {
            case 0: panel_dots<0>(col, jj, w, first, nrows, lane, wred[warp]); break;
            case 1: panel_dots<4>(col, jj, w, first, nrows, lane, wred[warp]); break;
            case 2: panel_dots<8>(col, jj, w, first, nrows, lane, wred[warp]); break;
            case 3: panel_dots<12>(col, jj, w, first, nrows, lane, wred[warp]); break;
            case 4: panel_dots<16>(col, jj, w, first, nrows, lane, wred[warp]); break;
            case 5: panel_dots<20>(col, jj, w, first, nrows, lane, wred[warp]); break;
            case 6: panel_dots<24>(col, jj, w, first, nrows, lane, wred[warp]); break;
            default: panel_dots<28>(col, jj, w, first, nrows, lane, wred[warp]); break;
        }
        __syncthreads();
        const int64_t dl = (int64_t)j0 + jj - row0;  // the diagonal row, local index
        const bool own_diag = dl >= 0 && dl < nrows;
        const bool cact = lane >= (jj & ~3) && lane < w;
        if (warp < 4) {  // a warp per quarter of the SM: the CTA's sums, into four CTAs each
            double ssum = 0.0;
            if (lane >= (jj & ~3))
                for (int q = 0; q < kPanelThreads / 32; ++q) ssum += wred[q][lane];
            const double dv = own_diag && cact ? col(lane)[dl] : 0.0;
#pragma unroll
            for (int r = 4 * warp; r < 4 * warp + 4; ++r) {
                *cluster.map_shared_rank(&red[buf][rank][lane], r) = ssum;
                if (own_diag) *cluster.map_shared_rank(&drow[buf][lane], r) = dv;
            }
        }
        cluster.sync();
        if (warp == 0) {  // every CTA: the same sums in the same order, a column per lane
            double tot = 0.0;
#pragma unroll
            for (int r = 0; r < kPanelCl; ++r) tot += red[buf][r][lane];
            const double alpha = drow[buf][jj], xnorm2 = __shfl_sync(0xffffffffu, tot, jj);
            double val = 0.0, beta = alpha;  // lane 0: tau, the others: the scale
            if (xnorm2 > 0.0) {
                beta = -copysign(sqrt(fma(alpha, alpha, xnorm2)), alpha);
                val = (lane == 0 ? beta - alpha : 1.0) / (lane == 0 ? beta : alpha - beta);
            }
            const double t = __shfl_sync(0xffffffffu, val, 0), scale = __shfl_sync(0xffffffffu, val, 1);
            const double sw = fma(scale, tot, drow[buf][lane]);
            sf[lane] = -t * sw;
            if (lane == 0) {
                s_scale = scale;
                if (rank == 0) tau[j0 + jj] = t;
            }
            if (own_diag) {
                if (lane == jj) col(jj)[dl] = beta;
                else if (lane > jj && lane < w) col(lane)[dl] = fma(-t, sw, drow[buf][lane]);
            }
        }
        __syncthreads();
        const double scale = s_scale;
        switch ((jj + 1) / 4) {
            case 0: panel_update<0>(col, jj, w, first, nrows, scale, sf); break;
            case 1: panel_update<4>(col, jj, w, first, nrows, scale, sf); break;
            case 2: panel_update<8>(col, jj, w, first, nrows, scale, sf); break;
            case 3: panel_update<12>(col, jj, w, first, nrows, scale, sf); break;
            case 4: panel_update<16>(col, jj, w, first, nrows, scale, sf); break;
            case 5: panel_update<20>(col, jj, w, first, nrows, scale, sf); break;
            case 6: panel_update<24>(col, jj, w, first, nrows, scale, sf); break;
            default: panel_update<28>(col, jj, w, first, nrows, scale, sf); break;
        }
        __syncthreads();
    }
    if (SMEM)
        for (int e = tid; e < kQB * rp; e += kPanelThreads) {
            const int c = e / rp, i = e % rp;
            if (c < w && i < nrows) Ab[i + (int64_t)c * lda] = P[e];
        }
    cluster.sync();  // no CTA leaves while another may still read its partials
}

// part[s][a][c] = sum over the rows of split s (from j0 on) of V(i, a) C(i, c0 + c),
// a < w, c < ncols; with ypart, two more tiles of columns (the first) are V
// itself, its partials [s][a][32] in ypart.  One CTA forms 32 x 16 sums over one
// split of 256 rows, two per thread: FP64-bound, so the tiles are small for the
// SMs' shares to come out even (32 x 32: 7 of 6.5 CTAs per SM at 8192 x 1024).
constexpr int kVtcCols = 16;
__global__ void __launch_bounds__(kVtcThreads)
k_qr_vtc(const double *__restrict__ A, int64_t lda, int64_t m, int j0, int w, const double *__restrict__ C,
         int64_t ldc, int c0, int ncols, int64_t rows_per, double *__restrict__ part, double *__restrict__ ypart) {
    __shared__ double Vs[kVtcRows][kQB + 1];
    __shared__ double Cs[kVtcRows][kVtcCols + 1];
    const int split = blockIdx.y, vt = ypart ? kQB / kVtcCols : 0;
    const bool is_v = (int)blockIdx.x < vt;
    const int ct0 = ((int)blockIdx.x - (is_v ? 0 : vt)) * kVtcCols;
    const int64_t r0 = (int64_t)j0 + (int64_t)split * rows_per;
    const int64_t r1 = m < r0 + rows_per ? m : r0 + rows_per;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    double acc[2] = {0.0, 0.0};
    for (int64_t rb = r0; rb < r1; rb += kVtcRows) {
        for (int e = tid; e < kVtcRows * kQB; e += kVtcThreads) {
            const int rr = e % kVtcRows, k = e / kVtcRows;
            const int64_t i = rb + rr;
            const bool in = i < r1;
            Vs[rr][k] = (in && k < w) ? v_entry(A, lda, i, j0, k) : 0.0;
            const int c = ct0 + k;
            if (!is_v && k < kVtcCols) Cs[rr][k] = in && c < ncols ? C[i + (int64_t)(c0 + c) * ldc] : 0.0;
        }
        __syncthreads();
        const double *X = is_v ? &Vs[0][ct0 + tx] : &Cs[0][tx];
        const int xs = is_v ? kQB + 1 : kVtcCols + 1;
#pragma unroll 8
        for (int rr = 0; rr < kVtcRows; ++rr) {
            const double x = X[rr * xs];
            acc[0] = fma(Vs[rr][ty], x, acc[0]);
            acc[1] = fma(Vs[rr][ty + 16], x, acc[1]);
        }
        __syncthreads();
    }
    const int nc = is_v ? kQB : ncols, c = ct0 + tx;
    double *pp = (is_v ? ypart : part) + (size_t)split * kQB * nc;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int a = ty + 16 * u;
        if (a < (is_v ? kQB : w) && c < nc) pp[(size_t)a * nc + c] = acc[u];
    }
}

// Y[a][c] = sum of the partials of V^T V in split order, one warp per row a
__global__ void __launch_bounds__(kQB) k_qr_sum(const double *__restrict__ ypart, int nsplit, double *__restrict__ Y) {
    const int e = blockIdx.x * kQB + threadIdx.x;
    double s = 0.0;
#pragma unroll 8
    for (int k = 0; k < nsplit; ++k) s += ypart[(size_t)k * kQB * kQB + e];
    Y[e] = s;
}

// T of the panel from tau and Y = V^T V: T_{r,j} = -tau_j sum_{k=r}^{j-1}
// T_{r,k} Y_{k,j}, T_jj = tau_j.  Warp r holds row r, lane j column j: once
// T_{r,k} is known it goes into the sums of every later column at once, a chain
// of two FP64 instructions a column instead of a sum over k per column (45 us
// with the partials' sum in the same kernel; 12 us, and 7 us for k_qr_sum: the
// same sums in the same order).
__global__ void __launch_bounds__(kQB * kQB)
k_qr_tbuild(const double *__restrict__ Y, int w, const double *__restrict__ tau_j0, double *__restrict__ T) {
    __shared__ double Ys[kQB][kQB + 1];
    const int r = threadIdx.x >> 5, j = threadIdx.x & 31;
    Ys[r][j] = Y[r * kQB + j];
    __syncthreads();
    const double tj = j < w ? tau_j0[j] : 0.0;
    double s = 0.0, t = r == j ? tj : 0.0;  // t: T_{r,j}
    for (int k = r; k < w - 1; ++k) {
        const double tk = __shfl_sync(0xffffffffu, t, k);
        if (j > k) s = fma(tk, Ys[k][j], s);
        if (j == k + 1 && j < w) t = -tj * s;
    }
    T[r * kQB + j] = t;
}

// Z[a][c] = sum_b op(T)[a][b] X[b][c], X the sum of the partials; op = T^T
// when trans (the factorisation applies H^T), T otherwise (Q applied).  One CTA
// per 8 columns, one entry a thread: the sums are bound by the FP64 pipe, and 32
// columns a CTA left most SMs idle (43 us a launch; 8 columns: 13 us).
constexpr int kTzCols = 8;
__global__ void __launch_bounds__(kQB * kTzCols)
k_qr_tz(const double *__restrict__ part, int nsplit, int w, int ncols, const double *__restrict__ T, int trans,
        double *__restrict__ Z) {
    __shared__ double Xs[kQB][kTzCols + 1];
    __shared__ double Ts[kQB][kQB + 1];
    const int tx = threadIdx.x % kTzCols, a = threadIdx.x / kTzCols, c = blockIdx.x * kTzCols + tx;
    for (int e = threadIdx.x; e < kQB * kQB; e += kQB * kTzCols) Ts[e / kQB][e % kQB] = T[e];
    double s = 0.0;
    if (a < w && c < ncols) {
        const double *pp = part + (size_t)a * ncols + c;
        const size_t step = (size_t)kQB * ncols;
#pragma unroll 8
        for (int q = 0; q < nsplit; ++q) s += pp[q * step];
    }
    Xs[a][tx] = s;
    __syncthreads();
    if (a >= w || c >= ncols) return;
    s = 0.0;
#pragma unroll 8
    for (int b = 0; b < w; ++b) s = fma(trans ? Ts[b][a] : Ts[a][b], Xs[b][tx], s);
    Z[(size_t)a * ncols + c] = s;
}

// C(i, c0 + c) -= sum_a V(i, a) Z[a][c] for rows i >= j0; one CTA per (row
// chunk of 64, column tile of 32)
__global__ void __launch_bounds__(256)
k_qr_update(double *__restrict__ C, int64_t ldc, int64_t m, int c0, int ncols, const double *__restrict__ A,
            int64_t lda, int j0, int w, const double *__restrict__ Z) {
    __shared__ double Vs[kQB][64];
    __shared__ double Zs[kQB][kQB];
    const int64_t r0 = (int64_t)j0 + (int64_t)blockIdx.x * 64;
    const int ct0 = blockIdx.y * kQB;
    const int tid = threadIdx.x;
    for (int e = tid; e < kQB * 64; e += 256) {
        const int a = e / 64, rr = e % 64;
        const int64_t i = r0 + rr;
        Vs[a][rr] = (i < m && a < w) ? v_entry(A, lda, i, j0, a) : 0.0;
    }
    for (int e = tid; e < kQB * kQB; e += 256) {
        const int a = e / kQB, c = e % kQB;
        Zs[a][c] = (a < w && ct0 + c < ncols) ? Z[(size_t)a * ncols + ct0 + c] : 0.0;
    }
    __syncthreads();
    const int rr = tid & 63, cg = tid >> 6;  // 64 rows x 4 column groups of 8
    const int64_t i = r0 + rr;
    if (i >= m) return;
    double s[8], old[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) s[k] = 0.0;
    for (int a = 0; a < w; ++a) {
        const double v = Vs[a][rr];
#pragma unroll
        for (int k = 0; k < 8; ++k) s[k] = fma(v, Zs[a][cg * 8 + k], s[k]);
    }
    // every load before any store (the columns of C are disjoint)
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int c = ct0 + cg * 8 + k;
        old[k] = c < ncols ? C[i + (int64_t)(c0 + c) * ldc] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int c = ct0 + cg * 8 + k;
        if (c < ncols) C[i + (int64_t)(c0 + c) * ldc] = old[k] - s[k];
    }
}

// the panel on a 16-CTA cluster: rows in shared memory when they fit, else in
// place in A
template <bool SMEM>
cudaError_t launch_panel_cl(double *A, int64_t lda, int64_t m, int j0, int w, int rp, double *tau, cudaStream_t st) {
    const size_t smem = SMEM ? (size_t)kQB * rp * sizeof(double) : 0;
    // the limit for every rp: it belongs to the function, not to this launch
    constexpr size_t kMax = SMEM ? (size_t)kQB * kPanelClMaxRows * sizeof(double) : 0;
    cudaError_t e = cudaFuncSetAttribute(k_qr_panel_cl<SMEM>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_qr_panel_cl<SMEM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMax);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kPanelCl);
    cfg.blockDim = dim3(kPanelThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kPanelCl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;  // launch only what the GPU can hold at once
    e = cudaOccupancyMaxActiveClusters(&clusters, k_qr_panel_cl<SMEM>, &cfg);
    if (e != cudaSuccess) return e;
    if (clusters < 1) return cudaErrorInvalidConfiguration;
    return cudaLaunchKernelEx(&cfg, k_qr_panel_cl<SMEM>, A, lda, m, j0, w, rp, tau);
}

cudaError_t panel_cluster(double *A, int64_t lda, int64_t m, int j0, int w, double *tau, cudaStream_t st) {
    const int64_t L = m - j0;
    const int rp = (int)((L + kPanelCl - 1) / kPanelCl);
    if (L < 2 * kPanelCl) return cudaErrorInvalidValue;
    return rp <= kPanelClMaxRows ? launch_panel_cl<true>(A, lda, m, j0, w, rp, tau, st)
                                 : launch_panel_cl<false>(A, lda, m, j0, w, rp, tau, st);
}

constexpr int kMaxSplit = 64;
int qr_nsplit(int64_t rows) {
    const int64_t s = (rows + 255) / 256;  // at least 256 rows per split
    return (int)std::max<int64_t>(1, std::min<int64_t>(s, kMaxSplit));
}

// Workspace of a factorisation, within qr_workspace_doubles(n).
struct QrWs {
    double *T, *tau, *ypart, *Y, *part, *Z;
};
constexpr int kMaxCols = 2048;  // columns of C taken at once
QrWs qr_carve(double *ws, int64_t n) {
    const int64_t panels = (n + kQB - 1) / kQB, cols = std::min<int64_t>(n, kMaxCols);
    QrWs q;
    q.T = ws;
    q.tau = q.T + (size_t)panels * kQB * kQB;
    q.ypart = q.tau + n;
    q.Y = q.ypart + (size_t)kMaxSplit * kQB * kQB;
    q.part = q.Y + kQB * kQB;
    q.Z = q.part + (size_t)kMaxSplit * kQB * cols;
    return q;
}

// Applies H_panel^T (trans) or H_panel to columns c0 .. c0 + ncols - 1 of C, in
// chunks of kMaxCols columns; with build, V^T V is formed in the first launch
// and T from it.
cudaError_t apply_panel(double *A, int64_t lda, int64_t m, int j0, int w, double *T, bool build, int trans, double *C,
                        int64_t ldc, int c0, int ncols, const QrWs &q, cudaStream_t st, long long *launches) {
    const int64_t rows = m - j0;
    for (int cb = 0; cb < ncols || (build && cb == 0); cb += kMaxCols) {
        const int nc = std::max(0, std::min(kMaxCols, ncols - cb));
        const bool with_v = build && cb == 0;
        const int tiles = (nc + kVtcCols - 1) / kVtcCols + (with_v ? kQB / kVtcCols : 0);
        const int nsplit = qr_nsplit(rows);
        const int64_t rows_per = (rows + nsplit - 1) / nsplit;
        k_qr_vtc<<<dim3(tiles, nsplit), kVtcThreads, 0, st>>>(A, lda, m, j0, w, C, ldc, c0 + cb, nc, rows_per, q.part,
                                                               with_v ? q.ypart : nullptr);
        *launches += 1;
        if (with_v) {
            k_qr_sum<<<kQB, kQB, 0, st>>>(q.ypart, nsplit, q.Y);
            k_qr_tbuild<<<1, kQB * kQB, 0, st>>>(q.Y, w, q.tau + j0, T);
            *launches += 2;
        }
        if (nc > 0) {
            k_qr_tz<<<(nc + kTzCols - 1) / kTzCols, kQB * kTzCols, 0, st>>>(q.part, nsplit, w, nc, T, trans, q.Z);
            const dim3 g2((unsigned)((rows + 63) / 64), (nc + kQB - 1) / kQB);
            k_qr_update<<<g2, 256, 0, st>>>(C, ldc, m, c0 + cb, nc, A, lda, j0, w, q.Z);
            *launches += 2;
        }
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

size_t qr_workspace_doubles(int64_t n) {
    const int64_t panels = (n + kQB - 1) / kQB, cols = std::min<int64_t>(n, kMaxCols);
    // T of every panel, tau, the partials of V^T V and their sum, the partials of V^T C, Z
    return (size_t)panels * kQB * kQB + (size_t)n + (size_t)(kMaxSplit + 1) * kQB * kQB +
           (size_t)(kMaxSplit + 1) * kQB * cols;
}

namespace {
// R (n x n, ldr) <- the upper triangle of A, zeros below; U (m x n, ldu) <-
// [U_R; 0] from U_R (n x n, ldur), or [I; 0]
__global__ void k_qr_extract_r(const double *__restrict__ A, int64_t lda, int64_t n, double *__restrict__ R,
                               int64_t ldr) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * n) return;
    const int64_t i = e % n, j = e / n;
    R[i + j * ldr] = i <= j ? A[i + j * lda] : 0.0;
}
__global__ void k_qr_embed_u(const double *__restrict__ UR, int64_t ldur, int64_t m, int64_t n,
                             double *__restrict__ U, int64_t ldu) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= m * n) return;
    const int64_t i = e % m, j = e / m;
    U[i + j * ldu] = i >= n ? 0.0 : (UR ? UR[i + j * ldur] : (i == j ? 1.0 : 0.0));  // no U_R: the identity
}
}  // namespace

cudaError_t qr_extract_r(const double *A, int64_t lda, int64_t n, double *R, int64_t ldr, cudaStream_t st) {
    const int64_t total = n * n;
    k_qr_extract_r<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(A, lda, n, R, ldr);
    return cudaGetLastError();
}

cudaError_t qr_embed_u(const double *UR, int64_t ldur, int64_t m, int64_t n, double *U, int64_t ldu,
                       cudaStream_t st) {
    const int64_t total = m * n;
    k_qr_embed_u<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(UR, ldur, m, n, U, ldu);
    return cudaGetLastError();
}

// A (m x n, lda) <- R in the upper triangle and the reflectors below it; T of
// every panel into ws.  m >= n.
cudaError_t qr_factor(double *A, int64_t lda, int64_t m, int64_t n, double *ws, cudaStream_t st,
                      long long *launches) {
    const int64_t panels = (n + kQB - 1) / kQB;
    const QrWs q = qr_carve(ws, n);
    for (int64_t p = 0; p < panels; ++p) {
        const int j0 = (int)(p * kQB), w = (int)std::min<int64_t>(kQB, n - j0);
        if (panel_cluster(A, lda, m, j0, w, q.tau, st) != cudaSuccess) {
            cudaGetLastError();  // clear a refused cluster launch; the one-CTA kernel does the panel
            k_qr_panel<<<1, kPanelThreads, 0, st>>>(A, lda, m, j0, w, q.tau);
        }
        *launches += 1;
        const cudaError_t e = apply_panel(A, lda, m, j0, w, q.T + (size_t)p * kQB * kQB, true, 1, A, lda, j0 + w,
                                          (int)(n - j0 - w), q, st, launches);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// U (m x ncols, ldu; ncols = 0: n) holds [U_R; 0] on entry; U <- Q U with the
// reflectors in A and the T factors in ws (as left by qr_factor).  The
// workspace holds partials for min(n, 2048) columns, so U is taken in chunks
// of that many columns.  With `identity` U holds [I; 0]: a panel's reflectors,
// zero above row j0, leave the columns before j0 as they are.
cudaError_t qr_apply_q(double *A, int64_t lda, int64_t m, int64_t n, double *ws, double *U, int64_t ldu,
                       cudaStream_t st, long long *launches, int64_t ncols, bool identity) {
    const int64_t panels = (n + kQB - 1) / kQB;
    const QrWs q = qr_carve(ws, n);
    const int64_t wcols = std::min<int64_t>(n, kMaxCols);
    if (ncols <= 0) ncols = n;
    for (int64_t c0 = 0; c0 < ncols; c0 += wcols) {
        const int nc = (int)std::min<int64_t>(wcols, ncols - c0);
        for (int64_t p = panels - 1; p >= 0; --p) {
            const int j0 = (int)(p * kQB), w = (int)std::min<int64_t>(kQB, n - j0);
            const int skip = identity ? (int)std::min<int64_t>(nc, std::max<int64_t>(0, j0 - c0)) : 0;
            if (skip == nc) continue;
            const cudaError_t e = apply_panel(A, lda, m, j0, w, q.T + (size_t)p * kQB * kQB, false, 0, U, ldu,
                                              (int)c0 + skip, nc - skip, q, st, launches);
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

}  // namespace hsvd
