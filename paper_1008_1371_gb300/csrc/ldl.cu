// ldl.cu -- the symmetric indefinite factorisation that turns an eigenproblem
// of a symmetric M into an HSVD (Sec. 1): M = P L D L^T P^T with complete
// (Bunch-Parlett) pivoting, D block diagonal with 1 x 1 and 2 x 2 blocks, and
// then G = P L B, J = diag(sign), B = diag(sqrt|d|) on 1 x 1 blocks and
// Q sqrt|Lambda| on a 2 x 2 block D_k = Q Lambda Q^T, so that M = G J G^T.
// The HSVD G V = U Sigma then gives M = U (Sigma^2 J) U^T: the eigenvalues of
// M are sigma_j^2 J_jj with eigenvectors u_j.
//
// Pivoting (Bunch and Parlett): with alpha = (1 + sqrt(17)) / 8,
// mu0 = max |a_ij| and mu1 = max |a_ii| over the trailing matrix, a 1 x 1 pivot
// on the largest diagonal entry if mu1 >= alpha mu0, else a 2 x 2 pivot on the
// rows and columns (r, q) of the largest off-diagonal entry.
//
// Unblocked and right-looking on the full trailing matrix.  Complete pivoting
// makes every step wait for the maximum of the step before over the whole
// matrix, so a step costs its latencies, not its arithmetic (two operations an
// entry): up to n = kPersistMaxN one cooperative launch does all the steps
// (k_ldl_persist), beyond that three kernels a step:
//   k_ldl_pivot   one CTA: reduces the per-CTA maxima of the last update,
//                 chooses the pivot, swaps it into place (rows and columns of
//                 the trailing matrix) and records the D block;
//   k_ldl_update  the rank-1 or rank-2 update of the trailing matrix, with the
//                 maxima of the updated entries per CTA for the next pivot;
//   k_ldl_lstore  the pivot column(s) below the block become L = W D^-1, and
//                 the position moves on.
// Both keep L in the output G, column k's entries in the rows of the original
// indices, so that no finished row is ever swapped; k_ldl_form_g turns it into
// G in place.  For the three kernels the position k and the step size live on
// the device; the host launches n rounds and the ones past the end return at
// once.
#include <cuda_runtime.h>

#include <algorithm>
#include <functional>
#include <type_traits>
#include <vector>

#include "hsvd_internal.cuh"

namespace hsvd {
namespace {

constexpr int kPivThreads = 1024;
constexpr int kUpdThreads = 256;

struct LdlState {
    int k;       // first column of the current step
    int s;       // its size (1 or 2; 0 once k reaches n)
    int bad;     // a non-finite entry (or no pivot found): HSVD_ERR_RANK
    int rank;    // columns factored: n, or the step at which the trailing matrix was zero
    double d[4];  // the step's D block, row-major
};

// per-CTA maxima of the trailing matrix: |diagonal| with its index, |off-diagonal| with (r, q)
struct LdlMax {
    double dmax, omax;
    int di, r, q, pad;
};

__device__ __forceinline__ void max_merge(LdlMax &a, const LdlMax &b) {
    // larger magnitude first, ties to the smaller index
    if (b.dmax > a.dmax || (b.dmax == a.dmax && b.di < a.di)) {
        a.dmax = b.dmax;
        a.di = b.di;
    }
    if (b.omax > a.omax || (b.omax == a.omax && (b.r < a.r || (b.r == a.r && b.q < a.q)))) {
        a.omax = b.omax;
        a.r = b.r;
        a.q = b.q;
    }
}

__device__ __forceinline__ LdlMax max_none() {
    LdlMax m;
    m.dmax = -1.0;
    m.omax = -1.0;
    m.di = m.r = m.q = 0x7fffffff;
    m.pad = 0;
    return m;
}

// swaps index a and b (both >= k) of the trailing symmetric matrix
__device__ void sym_swap(double *M, int64_t ld, int n, int k, int a, int b) {
    if (a == b) return;
    const int tid = threadIdx.x;
    // rows a, b in every trailing column
    for (int j = k + tid; j < n; j += blockDim.x) {
        if (j == a || j == b) continue;
        double *c = M + (int64_t)j * ld;
        const double t = c[a];
        c[a] = c[b];
        c[b] = t;
    }
    __syncthreads();
    // columns a, b in the trailing rows (the matrix is kept whole and symmetric)
    for (int i = k + tid; i < n; i += blockDim.x) {
        if (i == a || i == b) continue;
        double *ca = M + (int64_t)a * ld, *cb = M + (int64_t)b * ld;
        const double t = ca[i];
        ca[i] = cb[i];
        cb[i] = t;
    }
    if (tid == 0) {
        double *ca = M + (int64_t)a * ld, *cb = M + (int64_t)b * ld;
        const double t = ca[a];  // the two diagonal entries
        ca[a] = cb[b];
        cb[b] = t;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(kPivThreads)
k_ldl_pivot(double *__restrict__ M, int64_t ld, int n, LdlState *__restrict__ st, const LdlMax *__restrict__ mx,
            int nmx, int *__restrict__ perm, double *__restrict__ Dblk, int8_t *__restrict__ bsize) {
    __shared__ LdlMax red[kPivThreads / 32];
    __shared__ int s_choice[4];  // s, first, second
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int k = st->k;
    if (k >= n || st->bad) {  // done, or stopped at a zero pivot
        if (tid == 0) {
            st->s = 0;
            st->k = n;
        }
        return;
    }
    LdlMax a = max_none();
    for (int i = tid; i < nmx; i += kPivThreads) max_merge(a, mx[i]);
    for (int o = 16; o > 0; o >>= 1) {
        LdlMax b;
        b.dmax = __shfl_xor_sync(0xffffffffu, a.dmax, o);
        b.omax = __shfl_xor_sync(0xffffffffu, a.omax, o);
        b.di = __shfl_xor_sync(0xffffffffu, a.di, o);
        b.r = __shfl_xor_sync(0xffffffffu, a.r, o);
        b.q = __shfl_xor_sync(0xffffffffu, a.q, o);
        max_merge(a, b);
    }
    if (lane == 0) red[warp] = a;
    __syncthreads();
    if (tid == 0) {
        LdlMax t = red[0];
        for (int w = 1; w < kPivThreads / 32; ++w) max_merge(t, red[w]);
        const double alpha = (1.0 + sqrt(17.0)) / 8.0;
        const double mu0 = fmax(t.dmax, t.omax), mu1 = t.dmax;
        if (t.di >= k && t.di < n && mu0 == 0.0) {
            // the trailing matrix is zero: M has rank k (the postprocessing of a
            // singular M keeps the k columns found so far)
            s_choice[0] = -1;
        } else if (k == n - 1 || t.omax <= 0.0 || mu1 >= alpha * mu0) {
            s_choice[0] = 1;
            s_choice[1] = t.di;
        } else {
            s_choice[0] = 2;
            s_choice[1] = t.r < t.q ? t.r : t.q;
            s_choice[2] = t.r < t.q ? t.q : t.r;
        }
        // no valid pivot (NaN or Inf in the trailing matrix): stop with an error
        const bool valid = s_choice[0] == -1 ||
                           (s_choice[0] == 1 ? (s_choice[1] >= k && s_choice[1] < n)
                                             : (s_choice[1] >= k && s_choice[2] < n && s_choice[1] < s_choice[2]));
        if (!valid) s_choice[0] = 0;
    }
    __syncthreads();
    const int s = s_choice[0];
    if (s == -1) {
        if (tid == 0) {
            st->rank = k;
            st->s = 0;
            st->k = n;
        }
        return;
    }
    if (s == 0) {
        if (tid == 0) {
            st->bad = 1;
            st->s = 0;
            st->k = n;
        }
        return;
    }
    if (s == 1) {
        const int p = s_choice[1];
        sym_swap(M, ld, n, k, k, p);
        if (tid == 0) {
            const int t = perm[k];
            perm[k] = perm[p];
            perm[p] = t;
        }
    } else {
        const int r = s_choice[1], q = s_choice[2];  // r < q, both >= k
        // r -> k, then q -> k + 1 (q cannot be k: r < q and r >= k)
        sym_swap(M, ld, n, k, k, r);
        if (tid == 0) {
            const int t = perm[k];
            perm[k] = perm[r];
            perm[r] = t;
        }
        __syncthreads();
        const int q2 = (q == k) ? r : q;  // where q's index went after the first swap
        sym_swap(M, ld, n, k, k + 1, q2);
        if (tid == 0) {
            const int t = perm[k + 1];
            perm[k + 1] = perm[q2];
            perm[q2] = t;
        }
    }
    __syncthreads();
    // the D block; the pivot columns below it stay unscaled (W) for the update
    // and become L in k_ldl_lstore
    double *ck = M + (int64_t)k * ld;
    if (s == 1) {
        const double d = ck[k];
        if (tid == 0) {
            st->s = 1;
            st->d[0] = d;
            if (d == 0.0) st->bad = 1;
            Dblk[4 * k] = d;
            bsize[k] = 1;
        }
    } else {
        double *ck1 = M + (int64_t)(k + 1) * ld;
        const double d00 = ck[k], d01 = ck[k + 1], d11 = ck1[k + 1];
        if (tid == 0) {
            st->s = 2;
            st->d[0] = d00;
            st->d[1] = d01;
            st->d[2] = d01;
            st->d[3] = d11;
            if (fma(d00, d11, -d01 * d01) == 0.0) st->bad = 1;
            Dblk[4 * k] = d00;
            Dblk[4 * k + 1] = d01;
            Dblk[4 * k + 2] = d01;
            Dblk[4 * k + 3] = d11;
            bsize[k] = 2;
            bsize[k + 1] = 0;
        }
    }
}

// The trailing update for the step just pivoted: a_ij -= W_i D^-1 W_j^T for
// i, j >= k + s, W_i = (a_ik [, a_i,k+1]) the unscaled pivot columns.  The
// pivot columns become L = W D^-1 afterwards (k_ldl_lstore), once every CTA
// of this kernel has read them.
__global__ void __launch_bounds__(kUpdThreads)
k_ldl_update(double *__restrict__ M, int64_t ld, int n, const LdlState *__restrict__ st, LdlMax *__restrict__ mx) {
    __shared__ LdlMax red[kUpdThreads / 32];
    const int k = st->k, s = st->s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    LdlMax a = max_none();
    if (s > 0 && k < n && !st->bad) {
        const int t0 = k + s, nt = n - t0;
        const double *ck = M + (int64_t)k * ld, *ck1 = M + (int64_t)(k + 1) * ld;
        // D^-1 (1 x 1 or 2 x 2)
        double i00, i01 = 0.0, i11 = 0.0;
        if (s == 1) {
            i00 = 1.0 / st->d[0];
        } else {
            const double det = fma(st->d[0], st->d[3], -st->d[1] * st->d[1]);
            i00 = st->d[3] / det;
            i01 = -st->d[1] / det;
            i11 = st->d[0] / det;
        }
        const int64_t total = (int64_t)nt * nt;
        for (int64_t e = (int64_t)blockIdx.x * kUpdThreads + tid; e < total; e += (int64_t)gridDim.x * kUpdThreads) {
            const int i = t0 + (int)(e % nt), j = t0 + (int)(e / nt);
            double v;
            if (s == 1) {
                const double li = ck[i] * i00;
                v = fma(-li, ck[j], M[i + (int64_t)j * ld]);
            } else {
                const double wi0 = ck[i], wi1 = ck1[i];
                const double li0 = fma(wi0, i00, wi1 * i01), li1 = fma(wi0, i01, wi1 * i11);
                v = fma(-li0, ck[j], fma(-li1, ck1[j], M[i + (int64_t)j * ld]));
            }
            M[i + (int64_t)j * ld] = v;
            const double av = fabs(v);
            if (i == j) {
                if (av > a.dmax || (av == a.dmax && i < a.di)) {
                    a.dmax = av;
                    a.di = i;
                }
            } else if (i > j) {  // the lower triangle stands for both
                if (av > a.omax || (av == a.omax && (j < a.r || (j == a.r && i < a.q)))) {
                    a.omax = av;
                    a.r = j;
                    a.q = i;
                }
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        LdlMax b;
        b.dmax = __shfl_xor_sync(0xffffffffu, a.dmax, o);
        b.omax = __shfl_xor_sync(0xffffffffu, a.omax, o);
        b.di = __shfl_xor_sync(0xffffffffu, a.di, o);
        b.r = __shfl_xor_sync(0xffffffffu, a.r, o);
        b.q = __shfl_xor_sync(0xffffffffu, a.q, o);
        max_merge(a, b);
    }
    if (lane == 0) red[warp] = a;
    __syncthreads();
    if (tid == 0) {
        LdlMax t = red[0];
        for (int w = 1; w < kUpdThreads / 32; ++w) max_merge(t, red[w]);
        mx[blockIdx.x] = t;
    }
}

// After the update: the pivot column(s) below the block become L = W D^-1 (in
// G, by original row), and the state moves to the next step.
__global__ void k_ldl_lstore(const double *__restrict__ M, int64_t ld, int n, LdlState *__restrict__ st,
                             const int *__restrict__ perm, double *__restrict__ G, int64_t ldg) {
    const int k = st->k, s = st->s;
    if (s == 0 || k >= n) return;
    const double *ck = M + (int64_t)k * ld, *ck1 = M + (int64_t)(k + 1) * ld;
    if (!st->bad) {
        double i00, i01 = 0.0, i11 = 0.0;
        if (s == 1) {
            i00 = 1.0 / st->d[0];
        } else {
            const double det = fma(st->d[0], st->d[3], -st->d[1] * st->d[1]);
            i00 = st->d[3] / det;
            i01 = -st->d[1] / det;
            i11 = st->d[0] / det;
        }
        for (int i = k + s + (int)threadIdx.x; i < n; i += blockDim.x) {
            double *g = G + perm[i] + (int64_t)k * ldg;
            if (s == 1) {
                *g = ck[i] * i00;
            } else {
                const double wi0 = ck[i], wi1 = ck1[i];
                g[0] = fma(wi0, i00, wi1 * i01);
                g[ldg] = fma(wi0, i01, wi1 * i11);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) st->k = k + s;
}

// maxima of the whole matrix before the first pivot
__global__ void __launch_bounds__(kUpdThreads)
k_ldl_max0(const double *__restrict__ M, int64_t ld, int n, LdlMax *__restrict__ mx, LdlState *__restrict__ st) {
    __shared__ LdlMax red[kUpdThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    LdlMax a = max_none();
    const int64_t total = (int64_t)n * n;
    for (int64_t e = (int64_t)blockIdx.x * kUpdThreads + tid; e < total; e += (int64_t)gridDim.x * kUpdThreads) {
        const int i = (int)(e % n), j = (int)(e / n);
        const double av = fabs(M[i + (int64_t)j * ld]);
        if (!(av <= 1.7976931348623157e308)) atomicExch(&st->bad, 1);  // NaN or Inf in M
        if (i == j) {
            if (av > a.dmax || (av == a.dmax && i < a.di)) {
                a.dmax = av;
                a.di = i;
            }
        } else if (i > j) {
            if (av > a.omax || (av == a.omax && (j < a.r || (j == a.r && i < a.q)))) {
                a.omax = av;
                a.r = j;
                a.q = i;
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        LdlMax b;
        b.dmax = __shfl_xor_sync(0xffffffffu, a.dmax, o);
        b.omax = __shfl_xor_sync(0xffffffffu, a.omax, o);
        b.di = __shfl_xor_sync(0xffffffffu, a.di, o);
        b.r = __shfl_xor_sync(0xffffffffu, a.r, o);
        b.q = __shfl_xor_sync(0xffffffffu, a.q, o);
        max_merge(a, b);
    }
    if (lane == 0) red[warp] = a;
    __syncthreads();
    if (tid == 0) {
        LdlMax t = red[0];
        for (int w = 1; w < kUpdThreads / 32; ++w) max_merge(t, red[w]);
        mx[blockIdx.x] = t;
    }
}

// The two coefficients (per column of L) of a column of G, and its sign: a 1 x 1
// block scales by sqrt|d|, a 2 x 2 block D = Q diag(l1, l2) Q^T (Jacobi
// rotation, l1 > 0 > l2 for a 2 x 2 pivot) maps its two columns by
// Q diag(sqrt|l1|, sqrt|l2|).
struct GCol {
    double c0, c1;
    int8_t sgn;
};
__device__ __forceinline__ void g_columns(const double *d, int size, GCol &x, GCol &y) {
    if (size == 1) {
        x.c0 = sqrt(fabs(d[0]));
        x.c1 = 0.0;
        x.sgn = d[0] > 0.0 ? 1 : -1;
        return;
    }
    const double a = d[0], b = d[1], c = d[3];
    // the symmetric 2 x 2 Schur decomposition (a Jacobi rotation, t = tan phi
    // the smaller root): with Q = [cs sn; -sn cs], Q^T D Q = diag(a - t b, c + t b)
    double t = 0.0;
    if (b != 0.0) {
        const double zeta = (c - a) / (2.0 * b);
        t = (zeta >= 0.0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(fma(zeta, zeta, 1.0)));
    }
    const double cs = 1.0 / sqrt(fma(t, t, 1.0)), sn = t * cs;
    const double l1 = fma(-t, b, a), l2 = fma(t, b, c);
    // columns: q1 = (cs, -sn), q2 = (sn, cs)
    x.c0 = cs * sqrt(fabs(l1));
    x.c1 = -sn * sqrt(fabs(l1));
    x.sgn = l1 > 0.0 ? 1 : -1;
    y.c0 = sn * sqrt(fabs(l2));
    y.c1 = cs * sqrt(fabs(l2));
    y.sgn = l2 > 0.0 ? 1 : -1;
}

// G = P L B in place (column-major n x n) and J.  On entry column j of G holds
// column j of L below its block, by original row, zeros elsewhere; the row of
// position i is perm[i].  One CTA per block of D.
__global__ void k_ldl_form_g(int n, const int *__restrict__ perm, const double *__restrict__ Dblk,
                             const int8_t *__restrict__ bsize, double *__restrict__ G, int64_t ldg,
                             int8_t *__restrict__ J, const LdlState *__restrict__ st) {
    const int j = blockIdx.x;
    if (j >= st->rank) {  // past the rank of a singular M: no column (zeros), no sign
        if (threadIdx.x == 0) J[j] = 0;
        return;
    }
    const int size = bsize[j];
    if (size == 0) return;  // the second column of a 2 x 2 block
    GCol x = {}, y = {};
    g_columns(Dblk + 4 * (int64_t)j, size, x, y);
    const int p0 = perm[j], p1 = size == 2 ? perm[j + 1] : -1;
    double *g0 = G + (int64_t)j * ldg, *g1 = g0 + ldg;
    for (int o = threadIdx.x; o < n; o += blockDim.x) {
        // L is 1 on the diagonal, 0 above
        const double l0 = o == p0 ? 1.0 : g0[o], l1 = size == 2 ? (o == p1 ? 1.0 : g1[o]) : 0.0;
        g0[o] = fma(x.c0, l0, x.c1 * l1);
        if (size == 2) g1[o] = fma(y.c0, l0, y.c1 * l1);
    }
    if (threadIdx.x == 0) {
        J[j] = x.sgn;
        if (size == 2) J[j + 1] = y.sgn;
    }
}

// ---- all the steps in one launch ---------------------------------------------

constexpr int kPT = 1024;             // threads per CTA, one CTA per SM
constexpr int kPU = 8;                // columns of a row that a thread loads at once
constexpr int kPersistMaxN = 4096;    // the pivot columns and tables in shared memory; indices in 16 bits
constexpr unsigned kPollLimit = 1u << 22;

// A CTA's maxima of its part of the trailing matrix after step e - 1, as two
// 16-byte words that each carry the step number e, written and read whole:
// {key, e << 32 | bad << 31 | i << 1 | v < 0} for the diagonal and
// {key, e << 32 | r << 16 | q} below it, key = bits of |v| plus one, 0 for none (a
// NaN is none).
struct LdlSlot {
    unsigned long long dk, di, ok, oi;
};
__device__ __forceinline__ void put16(void *p, unsigned long long a, unsigned long long b) {
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
                 "l"(a), "l"(b)
                 : "memory");
}
__device__ __forceinline__ void get16(const void *p, unsigned long long &a, unsigned long long &b) {
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(a), "=l"(b)
                 : "l"(p)
                 : "memory");
}

// maximum key over the warp with the smallest index among equals, in every lane
__device__ __forceinline__ void warp_best(unsigned long long &key, unsigned &idx) {
    const unsigned hi = (unsigned)(key >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned lo = hi == mh ? (unsigned)key : 0u, ml = __reduce_max_sync(0xffffffffu, lo);
    idx = __reduce_min_sync(0xffffffffu, hi == mh && lo == ml ? idx : 0xffffffffu);
    key = ((unsigned long long)mh << 32) | ml;
}
struct LdlBest {
    unsigned long long dk, ok;
    unsigned di, oi;
    __device__ __forceinline__ void diag(unsigned long long k, unsigned i) {  // i: index << 1 | sign
        if (k > dk || (k == dk && i < di)) dk = k, di = i;
    }
    __device__ __forceinline__ void off(unsigned long long k, unsigned i) {
        if (k > ok || (k == ok && i < oi)) ok = k, oi = i;
    }
    // the value v at row i, column j (positions): the lower triangle stands for both
    __device__ __forceinline__ void see(double v, int i, int j) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
        const unsigned long long k = b <= 0x7FF0000000000000ull ? b + 1 : 0;
        if (i == j) diag(k, ((unsigned)i << 1) | (unsigned)(__double2hiint(v) < 0));
        else if (i > j) off(k, ((unsigned)j << 16) | (unsigned)i);
    }
    __device__ __forceinline__ void warp_reduce() {
        warp_best(dk, di);
        warp_best(ok, oi);
    }
};

// All the steps.  The matrix W (a copy of M) stays in L2; CTA b updates the
// trailing columns t0 + b, t0 + b + grid, ...; every CTA keeps the same two
// tables: perm (original index of a position) and slot (the column of W that
// holds a position's column).  A step:
//   - the CTAs' maxima of the last update, published with the step number, are
//     the grid barrier: every CTA polls all of them, a thread each, and takes
//     the same pivot decision;
//   - the pivot columns are read into shared memory.  The symmetric swap of
//     k_ldl_pivot needs no pass of its own: columns change places in `slot`,
//     and the one row that moves (row k into the pivot's place) is read from
//     where it was by the update.  The two entries a swap leaves unmoved,
//     (a, b) and (b, a), are read from there too: the same bits as swapping.
//     A column that moved is written into a free slot (W has two more than
//     columns), since other CTAs may still read the step's pivot columns and
//     the kept entries where they were;
//   - the update, the maxima of the new entries, and L's column (one CTA, by
//     turns) into G.
// A step reads W's slots only after every CTA published the step before it, and
// publishes into the half of the slots that step number's parity names, so no
// CTA can overwrite what another still reads.  A poll that runs out (2^22
// turns) sets state->bad = 2 and leaves.
// What bounds it is the chain of a step: about 1,700 cycles to reduce and
// publish, 4,000 for the slowest CTA's maxima to arrive, 3,000 for the decision,
// 2,300 for the loads, and the update (n = 1001: 4,500 on average, 2048: 15,000).
// Measured (N(0,1) symmetric, whole call, against the three kernels a step):
// n = 64: 0.48 against 2.37 ms, 300: 1.7 against 10.1, 1001: 8.9 against 37.7,
// 2048: 25.8 against 101, 4096: 124 against 358.
__global__ void __launch_bounds__(kPT, 1)
k_ldl_persist(const double *__restrict__ M, int64_t ldm, double *__restrict__ W, int n, double *__restrict__ G,
              int64_t ldg, int *__restrict__ perm_out, double *__restrict__ Dblk, int8_t *__restrict__ bsize,
              LdlState *__restrict__ st, LdlSlot *__restrict__ slots) {
    extern __shared__ __align__(16) double sm[];
    double *c0 = sm, *c1 = c0 + n;                     // the pivot columns, by position after the swap
    int *perm = reinterpret_cast<int *>(c1 + n), *slot = perm + n;
    __shared__ LdlBest red[kPT / 32];
    __shared__ int s_bad, s_late, s_sing, s_s, s_r, s_q;
    __shared__ int s_old[4], s_free[2];                // the slots of r, q, k, k + 1 before the swap; unused slots
    __shared__ double s_inv[3], s_d;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, grid = gridDim.x, cta = blockIdx.x;
    const double alpha = (1.0 + sqrt(17.0)) / 8.0;

    // copy M, with the maxima before the first step
    if (tid == 0) {
        s_bad = s_late = s_sing = 0;
        s_free[0] = n;
        s_free[1] = n + 1;
    }
    __syncthreads();
    LdlBest best = {0, 0, 0xffffffffu, 0xffffffffu};
    int bad = 0;
    for (int i = tid; i < n; i += kPT) perm[i] = slot[i] = i;
    for (int j = cta; j < n; j += grid)
        for (int i = tid; i < n; i += kPT) {
            const double v = M[i + (int64_t)j * ldm];
            bad |= !isfinite(v);
            __stcg(W + i + (int64_t)j * n, v);
            best.see(v, i, j);
        }
    if (bad) atomicOr(&s_bad, 1);

    int k = 0, rank = n, failed = 0;
    for (unsigned e = 1;; ++e) {
        // publish this CTA's maxima
        best.warp_reduce();
        if (lane == 0) red[warp] = best;
        __syncthreads();
        if (warp == 0) {
            LdlBest b = red[lane];
            b.warp_reduce();
            LdlSlot *mine = slots + (size_t)(e & 1) * grid;
            const unsigned long long tag = (unsigned long long)e << 32;
            if (lane == 0) {
                __threadfence();
                put16(&mine[cta].dk, b.dk, tag | ((unsigned)(s_bad != 0) << 31) | (b.di & 0x1ffffu));
                put16(&mine[cta].ok, b.ok, tag | b.oi);
            }
            __syncwarp();
        }
        __syncthreads();  // red is free again
        // every CTA's, one thread each
        {
            LdlBest t = {0, 0, 0xffffffffu, 0xffffffffu};
            if (warp * 32 < grid) {
                if (tid < grid) {
                    const LdlSlot *x = slots + (size_t)(e & 1) * grid + tid;
                    unsigned long long a, ia, o, io;
                    unsigned turns = 0;
                    do {
                        get16(&x->dk, a, ia);
                        get16(&x->ok, o, io);
                    } while (((unsigned)(ia >> 32) != e || (unsigned)(io >> 32) != e) && ++turns < kPollLimit);
                    if (turns >= kPollLimit) s_late = 1;
                    if ((unsigned)ia & 0x80000000u) s_bad = 1;
                    if (a) t.diag(a, (unsigned)ia & 0x1ffffu);
                    if (o) t.off(o, (unsigned)io);
                }
                t.warp_reduce();
                if (lane == 0) red[warp] = t;
            }
            __threadfence();  // what the others wrote before publishing is seen after this
        }
        __syncthreads();
        if (warp == 0) {
            LdlBest t = {0, 0, 0xffffffffu, 0xffffffffu};
            if (lane * 32 < grid) t = red[lane];
            t.warp_reduce();
            if (lane == 0) {
                const double dmax = t.dk ? __longlong_as_double((long long)(t.dk - 1)) : -1.0;
                const double omax = t.ok ? __longlong_as_double((long long)(t.ok - 1)) : -1.0;
                const double mu0 = fmax(dmax, omax);
                int s = 0, r = 0, q = 0;  // s: 0 no valid pivot, -1 the trailing matrix is zero, -2 a lost poll
                if (s_late) {
                    s = -2;
                } else if (s_bad) {
                    s = 0;
                } else if (t.dk && mu0 == 0.0) {
                    s = -1;
                } else if (k == n - 1 || omax <= 0.0 || dmax >= alpha * mu0) {
                    s = t.dk ? 1 : 0;
                    r = (int)(t.di >> 1);
                } else {
                    s = 2;
                    r = (int)(t.oi >> 16);
                    q = (int)(t.oi & 0xffffu);
                }
                if (e > 1) {  // the last step's moved columns, and the slots it gave up
                    const int r0 = s_r, q0 = s_q;
                    if (r0 >= k) slot[r0] = s_free[0];
                    if (s_s == 2 && q0 >= k) slot[q0] = s_free[1];
                    s_free[0] = s_old[0];
                    if (s_s == 2) s_free[1] = s_old[1];
                }
                if (s > 0) {
                    s_old[0] = slot[r];
                    s_old[1] = slot[q];
                    s_old[2] = slot[k];
                    s_old[3] = slot[min(k + 1, n - 1)];
                    auto swap = [](int *a, int x, int y) {
                        const int z = a[x];
                        a[x] = a[y];
                        a[y] = z;
                    };
                    swap(perm, k, r);
                    swap(slot, k, r);
                    if (s == 2) {
                        swap(perm, k + 1, q);
                        swap(slot, k + 1, q);
                    }
                }
                s_s = s;
                s_r = r;
                s_q = q;
                s_d = (t.di & 1) ? -dmax : dmax;  // the diagonal's largest: the pivot of a 1 x 1 step
            }
        }
        __syncthreads();
        const int s = s_s, r = s_r, q = s_q;
        if (s <= 0) {
            if (s == -1) rank = k;
            else failed = s == -2 ? 2 : 1;
            break;
        }
        const double *wr = W + (int64_t)s_old[0] * n, *wq = W + (int64_t)s_old[1] * n,
                     *wk = W + (int64_t)s_old[2] * n, *wk1 = W + (int64_t)s_old[3] * n;
        const int t0 = k + s;
        const int f0 = s_free[0], f1 = s_free[1];
        auto source = [&](int i) {  // where row i was before the swap
            const int x = s == 2 && i == q ? k + 1 : i;
            return x == r ? k : x;
        };
        // the pivot columns below the block into shared memory, and the thread's
        // first row of trailing entries into registers behind the same latency
        double old[kPU];
        const int row = t0 + tid, src = source(row);
#pragma unroll
        for (int u = 0; u < kPU; ++u) {
            const int j = t0 + cta + u * grid;
            if (row < n && j < n) old[u] = __ldcg(W + src + (int64_t)slot[j] * n);
        }
        for (int i = t0 + tid; i < n; i += kPT) {
            if (s == 1) {
                c0[i] = __ldcg(i == r ? wk + r : wr + i);
            } else {
                const int x = i == q ? k + 1 : i;
                c0[i] = __ldcg(r != k && x == r ? wk + r : wr + x);
                const bool kept = q != k + 1 && i == q;
                c1[i] = __ldcg(kept ? (r == k + 1 ? wk : wk1) + q : wq + (i == r && r != k ? k : i));
            }
        }
        if (warp == kPT / 32 - 1) {  // D and its inverse, the three quotients in three lanes
            const double d00 = s == 1 ? s_d : __ldcg(wr + r);
            const double d01 = s == 2 ? __ldcg(wr + q) : 0.0, d11 = s == 2 ? __ldcg(wq + q) : 0.0;
            const double det = s == 2 ? fma(d00, d11, -d01 * d01) : d00;
            const double num = s == 1 ? 1.0 : (lane == 0 ? d11 : (lane == 1 ? -d01 : d00));
            const double v = num / det;
            if (lane < 3) s_inv[lane] = v;
            if (lane == 0) {
                if (det == 0.0) s_sing = 1;  // no inverse
                if (cta == 0) {
                    double *d = Dblk + 4 * (int64_t)k;
                    d[0] = d00;
                    if (s == 2) {
                        d[1] = d01;
                        d[2] = d01;
                        d[3] = d11;
                    }
                    bsize[k] = (int8_t)s;
                    if (s == 2) bsize[k + 1] = 0;
                }
            }
        }
        __syncthreads();
        if (s_sing) {  // the same D everywhere: every CTA leaves here
            failed = 1;
            break;
        }
        const double i00 = s_inv[0], i01 = s_inv[1], i11 = s_inv[2];
        best = {0, 0, 0xffffffffu, 0xffffffffu};
        const bool store_l = cta == k % grid;
        // (the step's size is a template argument, the columns past n a branch: an
        // FP64 instruction that is predicated off occupies the pipe like any other)
        auto update = [&](auto size) {
            constexpr int S = decltype(size)::value;
            for (int i = row; i < n; i += kPT) {
                const int si = source(i);
                const double w0 = c0[i];
                double l0, l1 = 0.0;
                if constexpr (S == 1) {
                    l0 = w0 * i00;
                } else {
                    const double w1 = c1[i];
                    l0 = fma(w0, i00, w1 * i01);
                    l1 = fma(w0, i01, w1 * i11);
                }
                if (store_l) {
                    double *g = G + perm[i] + (int64_t)k * ldg;
                    g[0] = l0;
                    if (S == 2) g[ldg] = l1;
                }
                for (int j0 = t0 + cta; j0 < n; j0 += kPU * grid) {
                    if (i != row || j0 != t0 + cta) {
#pragma unroll
                        for (int u = 0; u < kPU; ++u) {
                            const int j = j0 + u * grid;
                            if (j < n) old[u] = __ldcg(W + si + (int64_t)slot[j] * n);
                        }
                    }
#pragma unroll
                    for (int u = 0; u < kPU; ++u) {
                        const int j = j0 + u * grid;
                        if (j >= n) break;
                        const int to = j == r ? f0 : (S == 2 && j == q ? f1 : slot[j]);
                        double v = old[u];
                        if constexpr (S == 2) v = fma(-l1, c1[j], v);
                        v = fma(-l0, c0[j], v);
                        __stcg(W + i + (int64_t)to * n, v);
                        best.see(v, i, j);
                    }
                }
            }
        };
        if (s == 1) update(std::integral_constant<int, 1>{});
        else update(std::integral_constant<int, 2>{});
        k = t0;
        if (k >= n) break;
    }
    if (cta == 0) {
        __syncthreads();
        for (int i = tid; i < n; i += kPT) perm_out[i] = perm[i];
        if (tid == 0) {
            st->rank = rank;
            st->bad = failed;
        }
    }
}

constexpr int kUpdGrid = 608;

// dynamic shared memory of k_ldl_persist: two pivot columns and two tables
constexpr size_t persist_smem(int64_t n) { return (size_t)n * (2 * sizeof(double) + 2 * sizeof(int)); }

}  // namespace

// M (n x n, ldm, device, symmetric; read-only) -> G (n x n, ldg, device) and
// J (n, device) with M = G J G^T.  A singular M stops once the trailing matrix
// is zero: *rank (may be NULL) receives the columns factored, and G's columns
// and J's entries past it are zero.  Returns HSVD_OK or HSVD_ERR_RANK (a
// non-finite entry).
int ldl_factor(const double *M, int64_t n, int64_t ldm, double *G, int64_t ldg, int8_t *J, cudaStream_t st,
               long long *launches, int64_t *rank) {
    double *W = nullptr, *Dblk = nullptr;
    int *perm = nullptr;
    int8_t *bsize = nullptr;
    LdlState *state = nullptr;
    LdlMax *mx = nullptr;
    LdlSlot *slots = nullptr;
    int rc = HSVD_OK;
    auto ok = [&](cudaError_t e) {
        if (e != cudaSuccess && rc == HSVD_OK) rc = HSVD_ERR_CUDA;
        return e == cudaSuccess;
    };
    // one launch while the pivot columns fit shared memory: a CTA for every six
    // columns, at most one per SM that the stream may use
    bool persist = n <= kPersistMaxN;
    const int grid = (int)std::min<int64_t>(stream_limits(st).sms, std::max<int64_t>(1, n / 6));
    const size_t nslots = persist ? 2 * (size_t)grid : 0;
    const double *m_end = M + (n - 1) * ldm + n, *g_end = G + (n - 1) * ldg + n;
    const bool overlap = persist && std::less<const double *>()(M, g_end) && std::less<const double *>()(G, m_end);
    double *Mc = nullptr;
    if ((overlap && !ok(scratch_alloc((void **)&Mc, sizeof(double) * n * n, st))) ||
        !ok(scratch_alloc((void **)&W, sizeof(double) * n * (n + 2), st)) ||
        !ok(scratch_alloc((void **)&Dblk, sizeof(double) * 4 * n, st)) ||
        !ok(scratch_alloc((void **)&perm, sizeof(int) * n, st)) ||
        !ok(scratch_alloc((void **)&bsize, (size_t)n, st)) ||
        !ok(scratch_alloc((void **)&state, sizeof(LdlState), st)) ||
        !ok(scratch_alloc((void **)&mx, sizeof(LdlMax) * kUpdGrid, st)) ||
        !ok(scratch_alloc((void **)&slots, sizeof(LdlSlot) * (nslots + 1), st))) {
        rc = HSVD_ERR_NOMEM;
    }
    if (rc == HSVD_OK) {
        LdlState s0 = {};
        s0.rank = (int)n;
        std::vector<int> p;
        ok(cudaMemcpyAsync(state, &s0, sizeof s0, cudaMemcpyHostToDevice, st));
        ok(cudaMemsetAsync(bsize, 1, (size_t)n, st));
        // L starts as zeros in G, which may lie in M's memory: M is copied first
        auto zero_g = [&]() { ok(cudaMemset2DAsync(G, sizeof(double) * ldg, 0, sizeof(double) * n, n, st)); };
        if (persist) {
            if (Mc) {
                ok(cudaMemcpy2DAsync(Mc, sizeof(double) * n, M, sizeof(double) * ldm, sizeof(double) * n, n,
                                     cudaMemcpyDeviceToDevice, st));
                M = Mc;
                ldm = n;
            }
            zero_g();
            const size_t smem = persist_smem(n);
            ok(cudaMemsetAsync(slots, 0, sizeof(LdlSlot) * nslots, st));
            // the limit for every n: it belongs to the function, not to this launch
            ok(cudaFuncSetAttribute(k_ldl_persist, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)persist_smem(kPersistMaxN)));
            int n_int = (int)n;
            void *args[] = {(void *)&M, &ldm, &W, &n_int, &G, &ldg, &perm, &Dblk, &bsize, &state, &slots};
            const cudaError_t e =
                cudaLaunchCooperativeKernel((const void *)k_ldl_persist, dim3(grid), dim3(kPT), args, smem, st);
            if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
                cudaGetLastError();  // refused: the three kernels need no CTAs at the same time
                persist = false;
            } else {
                ok(e);
            }
        }
        if (!persist) {
            p.resize((size_t)n);
            for (int64_t i = 0; i < n; ++i) p[(size_t)i] = (int)i;
            ok(cudaMemcpy2DAsync(W, sizeof(double) * n, M, sizeof(double) * ldm, sizeof(double) * n, n,
                                 cudaMemcpyDeviceToDevice, st));
            zero_g();
            ok(cudaMemcpyAsync(perm, p.data(), sizeof(int) * n, cudaMemcpyHostToDevice, st));
            k_ldl_max0<<<kUpdGrid, kUpdThreads, 0, st>>>(W, n, (int)n, mx, state);
            ok(cudaGetLastError());
            // every step takes one or two columns: n (pivot, update, store) rounds
            // cover the worst case, rounds past the end return at once
            for (int64_t t = 0; t < n && rc == HSVD_OK; ++t) {
                k_ldl_pivot<<<1, kPivThreads, 0, st>>>(W, n, (int)n, state, mx, kUpdGrid, perm, Dblk, bsize);
                k_ldl_update<<<kUpdGrid, kUpdThreads, 0, st>>>(W, n, (int)n, state, mx);
                k_ldl_lstore<<<1, 256, 0, st>>>(W, n, (int)n, state, perm, G, ldg);
                ok(cudaGetLastError());
            }
        }
        k_ldl_form_g<<<(unsigned)n, 256, 0, st>>>((int)n, perm, Dblk, bsize, G, ldg, J, state);
        ok(cudaGetLastError());
        LdlState fin = {};
        if (ok(cudaMemcpyAsync(&fin, state, sizeof fin, cudaMemcpyDeviceToHost, st)) &&
            ok(cudaStreamSynchronize(st)) && fin.bad)
            rc = fin.bad == 2 ? HSVD_ERR_CUDA : HSVD_ERR_RANK;
        if (rank) *rank = fin.rank;
        if (launches) *launches += persist ? 2 : 2 + 3 * n;
    }
    if (Mc) cudaFreeAsync(Mc, st);
    if (W) cudaFreeAsync(W, st);
    if (Dblk) cudaFreeAsync(Dblk, st);
    if (perm) cudaFreeAsync(perm, st);
    if (bsize) cudaFreeAsync(bsize, st);
    if (state) cudaFreeAsync(state, st);
    if (mx) cudaFreeAsync(mx, st);
    if (slots) cudaFreeAsync(slots, st);
    return rc;
}

}  // namespace hsvd
