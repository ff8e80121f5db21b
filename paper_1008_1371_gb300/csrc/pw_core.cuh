// pw_core.cuh -- the pointwise one-sided hyperbolic Jacobi method (Sec. 2,
// Alg. 4.5): the pieces shared by the single-factor kernels (pointwise.cu) and
// the persistent batched kernel (batched.cu), and pw_solve, the body that a
// group of NT threads (a whole CTA, or an aligned part of one that synchronises
// on its own named barrier `bar`) runs for one factor and all of its sweeps.
//
// G (column-major, rows padded to a multiple of 32) and the accumulated
// transformation W (the paper's V^{-T}, Eq. 2.1; formed only when V is asked
// for) sit in shared memory as far as they fit, the rest in global memory.
// For each pair a_ii, a_jj, a_ij come from the current columns, then the test
// of Eq. 2.3, (t, c), and the FMA form of Alg. 4.5 on the columns of G and W.
// The FP64 pipe of the SM (about 2 lanes' FMAs a clock) is the bound.  A
// column's dot with itself is kept until a rotation changes the column (the
// same bits as forming it again): the last sweeps, where nearly every pair
// passes, cost m operations a pair instead of 3 m.
//
// A step of the modified modulus strategy (Sec. 2) has n'/2 disjoint pairs.
// The dots: lane l of a warp sums rows l, l + 32, ..., then a butterfly over
// the lanes (xor 16, 8, 4, 2, 1), so every kernel forms the same bits.  The
// convergence check is the bit-or reduction of Eq. 4.2 held in two shared
// words: the sweep's rotation count (code (00)_2 when it is zero) and, with
// the tangent threshold T on, a flag set by any rotation with |t| > T (code
// (11)_2); a sweep that rotated without setting it is code (01)_2 and also
// ends the iteration.  No host round trip is needed between sweeps.
//
// In pw_solve columns are never moved: positions map to columns through pos[]
// (Sec. 4).  Before the first sweep positions are grouped J+ then J- (Alg. 4.2
// assumes J = diag(I_p, -I_{n-p})); with sorting on they are then ordered by
// d = ||g||^2, decreasing in the J+ part and increasing in the J- part, ties in
// current order (Sec. 4, Sort_Diagonal), again after every sweep.  An odd n is
// bordered with one unit column in a fresh row (Eq. 4.1).
#pragma once

#include "hsvd_internal.cuh"

namespace hsvd {

// The factor's working arrays.  G (m_pad x n_pad) and W (n_pad x n_pad): the
// first gs (ws) columns in shared memory at Gs (Ws), the others at column
// offset j in global memory at Gg (Wg).  Per column: its dot with itself
// (negative: to be formed), position maps and the sign.  Per pair of a step:
// a_pq (then c), t, the columns p | q << 16 and whether it rotates (0: no, -1: a
// trigonometric, 1: a hyperbolic rotation).
struct PwArrays {
    double *Gs, *Gg, *Ws, *Wg;
    int gs, ws;
    double *d;
    double *apq, *t;  // a_pq, then c; t
    int *pos, *newpos, *sg, *pq, *hyp;
    __device__ __forceinline__ double *g(int j, int m_pad) const {
        return (j < gs ? Gs : Gg) + (size_t)j * m_pad;
    }
    __device__ __forceinline__ double *w(int j, int n_pad) const {
        return (j < ws ? Ws : Wg) + (size_t)j * n_pad;
    }
};

// bytes of the per-column and per-pair arrays
__host__ __device__ inline size_t pw_aux_bytes(int64_t n_pad) {
    return (size_t)n_pad * (sizeof(double) + 3 * sizeof(int)) +
           (size_t)(n_pad / 2) * (2 * sizeof(double) + 2 * sizeof(int));
}

__device__ __forceinline__ void pw_carve(PwArrays &a, void *aux, int n_pad) {
    const int half = n_pad / 2;
    a.d = reinterpret_cast<double *>(aux);
    a.apq = a.d + n_pad;
    a.t = a.apq + half;
    a.pos = reinterpret_cast<int *>(a.t + half);
    a.newpos = a.pos + n_pad;
    a.sg = a.newpos + n_pad;
    a.pq = a.sg + n_pad;
    a.hyp = a.pq + half;
}

// lane l's part of the dots of columns gp, gq (length len, a multiple of 32):
// rows l, l + 32, ... in order; the products asked for are formed, four loads
// issued ahead of their FMAs so that columns in global memory stream
template <bool PP, bool QQ>
__device__ __forceinline__ void pw_dots(const double *__restrict__ gp, const double *__restrict__ gq, int len,
                                        int lane, double &app, double &aqq, double &apq) {
    constexpr int U = 4;
    app = aqq = apq = 0.0;
    int i = lane;
    for (; i + (U - 1) * kWarp < len; i += U * kWarp) {
        double x[U], y[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            x[u] = gp[i + u * kWarp];
            y[u] = gq[i + u * kWarp];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (PP) app = fma(x[u], x[u], app);
            if (QQ) aqq = fma(y[u], y[u], aqq);
            apq = fma(x[u], y[u], apq);
        }
    }
    for (; i < len; i += kWarp) {
        const double x = gp[i], y = gq[i];
        if (PP) app = fma(x, x, app);
        if (QQ) aqq = fma(y, y, aqq);
        apq = fma(x, y, apq);
    }
}

__device__ __forceinline__ void pw_dots_sel(bool pp, bool qq, const double *gp, const double *gq, int len, int lane,
                                            double &app, double &aqq, double &apq) {
    if (pp && qq) pw_dots<true, true>(gp, gq, len, lane, app, aqq, apq);
    else if (pp) pw_dots<true, false>(gp, gq, len, lane, app, aqq, apq);
    else if (qq) pw_dots<false, true>(gp, gq, len, lane, app, aqq, apq);
    else pw_dots<false, false>(gp, gq, len, lane, app, aqq, apq);
}

// one level of a butterfly over the lanes that halves the values a lane
// carries: lanes with bit `o` set keep b, the others a
__device__ __forceinline__ double pw_fold(double a, double b, int o, bool set) {
    const double send = set ? a : b;
    return (set ? b : a) + __shfl_xor_sync(0xffffffffu, send, o);
}
__device__ __forceinline__ double pw_xor_add(double a, int o) { return a + __shfl_xor_sync(0xffffffffu, a, o); }

// the column update of Alg. 4.5 from (xp, xq) to (yp, yq), which may be the
// same columns, four loads issued ahead
__device__ __forceinline__ void pw_rotate(const double *xp, const double *xq, double *yp, double *yq, int len,
                                          int lane, double ht, double t, double c) {
    constexpr int U = 4;
    int i = lane;
    for (; i + (U - 1) * kWarp < len; i += U * kWarp) {
        double x[U], y[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            x[u] = xp[i + u * kWarp];
            y[u] = xq[i + u * kWarp];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            yp[i + u * kWarp] = fma(ht, y[u], x[u]) * c;
            yq[i + u * kWarp] = fma(t, x[u], y[u]) * c;
        }
    }
    for (; i < len; i += kWarp) {
        const double x = xp[i], y = xq[i];
        yp[i] = fma(ht, y, x) * c;
        yq[i] = fma(t, x, y) * c;
    }
}

// Comparisons on bit patterns: an FP64 comparison would take one of the
// warp's 64-cycle turns on the FP64 pipe.
__device__ __forceinline__ unsigned long long pw_abs_bits(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}
constexpr unsigned long long kPwInf = 0x7FF0000000000000ull, kPwOne = 0x3FF0000000000000ull;
__device__ __forceinline__ bool pw_larger(double x, double bound) {  // |x| > bound >= 0, false for a NaN
    const unsigned long long a = pw_abs_bits(x);
    return a > pw_abs_bits(bound) && a <= kPwInf;
}
// a kept dot is missing when its sign bit is set
__device__ __forceinline__ bool pw_missing(double d) { return __double2hiint(d) < 0; }

// The test of Eq. 2.3, then for a pair that fails it the rotation of Sec. 2 by
// the formulas of rotation_params, bit for bit (a tangent threshold of Eq. 4.2
// then stops these kernels at the oracle's sweep).  Returns 0 (the pair
// passes), 1 (rotate with t, c) or 2 (rank deficient).
__device__ __forceinline__ int pw_decision(double aii, double ajj, double aij, int hyp, double tol, double &t,
                                           double &c) {
    if (pair_passes(aii, ajj, aij, tol)) return 0;
    const bool trig = hyp < 0;
    const double zeta = (trig ? ajj - aii : neg_bits(aii + ajj)) / (2.0 * aij);
    if (!trig && !pw_larger(zeta, 1.0)) return 2;
    const double az = fabs(zeta);
    double tt = 1.0 / (az + sqrt(trig ? az * az + 1.0 : az * az - 1.0));
    if (__double2hiint(zeta) < 0 && pw_abs_bits(zeta) != 0) tt = neg_bits(tt);
    const double q0 = sqrt(trig ? 1.0 + tt * tt : (1.0 - tt) * (1.0 + tt));
    t = tt;
    c = cosine_step(tt, hyp, 1.0 / q0);
    return 1;
}

// sort order (Sec. 4): keys between +0 and +inf compare as their bit patterns
// (an FP64 comparison issues at the FP64 rate), others as numbers
__device__ __forceinline__ bool pw_before(double kb, double key, int grp, bool b_first) {
    const unsigned long long x = (unsigned long long)__double_as_longlong(kb),
                             y = (unsigned long long)__double_as_longlong(key);
    if (x <= kPwInf && y <= kPwInf) return (grp > 0 ? x > y : x < y) || (x == y && b_first);
    return (grp > 0 ? kb > key : kb < key) || (kb == key && b_first);
}

// barrier of a group of NT threads (NT a multiple of 32; id 0 with NT equal
// to the CTA size is __syncthreads)
template <int NT>
__device__ __forceinline__ void grp_sync(int bar) {
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(NT) : "memory");
}

// shared scalars of a group
struct PwScalars {
    int rot, err, bad, big;
    unsigned long long total;
};

// positions by d = ||g||^2
template <int NT>
__device__ void pw_reorder(const PwArrays &sh, int m_pad, int n_pad, int bar) {
    constexpr int kW = NT / kWarp;
    const int tid = threadIdx.x & (NT - 1), lane = tid & 31, warp = tid >> 5;
    for (int j = warp; j < n_pad; j += kW) {
        double s = sh.d[j];
        if (pw_missing(s)) {
            const double *g = sh.g(j, m_pad);
            s = 0.0;
            for (int i = lane; i < m_pad; i += kWarp) s = fma(g[i], g[i], s);
            s = warp_sum(s);
        }
        __syncwarp();
        if (lane == 0) sh.d[j] = s;
    }
    grp_sync<NT>(bar);
    int nplus = 0;
    for (int a = 0; a < n_pad; ++a) nplus += sh.sg[sh.pos[a]] > 0;
    for (int a = tid; a < n_pad; a += NT) {
        const int col = sh.pos[a];
        const int grp = sh.sg[col];
        const double key = sh.d[col];
        int rank = 0;
        for (int b = 0; b < n_pad; ++b) {
            const int cb = sh.pos[b];
            if (sh.sg[cb] == grp && b != a && pw_before(sh.d[cb], key, grp, b < a)) ++rank;
        }
        sh.newpos[(grp > 0 ? 0 : nplus) + rank] = col;
    }
    grp_sync<NT>(bar);
    for (int a = tid; a < n_pad; a += NT) sh.pos[a] = sh.newpos[a];
    grp_sync<NT>(bar);
}

// One column's outputs (Sec. 2): sigma = ||g||, u = g / sigma, v = w; one warp.
// Returns an error code or 0 (lane 0).
__device__ __forceinline__ int pw_finish_column(const double *g, const double *w, int m, int n, int j, int lane,
                                                double *__restrict__ sigma, double *__restrict__ U, int64_t ldu,
                                                double *__restrict__ V, int64_t ldv) {
    double mx = 0.0;
    for (int i = lane; i < m; i += kWarp) mx = fmax(mx, fabs(g[i]));
    mx = warp_max(mx);
    int e;
    const double scl = pow2_scale_for(mx, e);
    double ss = 0.0;
    for (int i = lane; i < m; i += kWarp) {
        const double v = g[i] * scl;
        ss = fma(v, v, ss);
    }
    ss = warp_sum(ss);
    const double sj = ldexp(sqrt(ss), e);
    int err = 0;
    if (lane == 0) {
        sigma[j] = sj;
        if (!(sj > 0.0)) err = HSVD_ERR_RANK;
        if (!isfinite(sj)) err = HSVD_ERR_NONFINITE;
    }
    if (U)
        for (int i = lane; i < m; i += kWarp) U[i + (int64_t)j * ldu] = g[i] / sj;
    if (V)
        for (int i = lane; i < n; i += kWarp) V[i + (int64_t)j * ldv] = w[i];
    return err;
}

// The dots of step s for the group's pairs, PER pairs of a warp at a time, reduced
// together: a lane ends with one of the sums, z = a_pq of pair u in the lanes whose
// `part` is PART_Z, and where a pair's kept dots are missing x = a_pp and y = a_qq in
// two others.
template <int NT, int PER>
__device__ __forceinline__ void pw_step_dots(const PwArrays &sh, int m_pad, int n_pad, int s) {
    constexpr int kW = NT / kWarp;
    const int tid = threadIdx.x & (NT - 1), lane = tid & 31, warp = tid >> 5, half = n_pad / 2;
    for (int k0 = PER * warp; k0 < half; k0 += PER * kW) {
        const int nb = min(PER, half - k0);
        int my_p = 0, my_q = 0, my_need = 0;
        if (lane < nb) {
            int a, b;
            modulus_pair(n_pad, s, k0 + lane, a, b);
            my_p = sh.pos[a];
            my_q = sh.pos[b];
            sh.pq[k0 + lane] = my_p | (my_q << 16);
            my_need = (pw_missing(sh.d[my_p]) ? 1 : 0) | (pw_missing(sh.d[my_q]) ? 2 : 0);
        }
        const bool any = __any_sync(0xffffffffu, my_need);
        double v[PER][3];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            v[u][0] = v[u][1] = v[u][2] = 0.0;
            if (u < nb) {
                const int p = __shfl_sync(0xffffffffu, my_p, u), q = __shfl_sync(0xffffffffu, my_q, u);
                const int need = __shfl_sync(0xffffffffu, my_need, u);
                pw_dots_sel(need & 1, need & 2, sh.g(p, m_pad), sh.g(q, m_pad), m_pad, lane, v[u][0], v[u][1],
                            v[u][2]);
            }
        }
        const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4, h2 = lane & 2;
        constexpr int PART_X = 0, PART_Y = PER == 4 ? 4 : 8, PART_Z = PER == 4 ? 2 : (PER == 2 ? 4 : 16);
        double z;
        int u, part;
        if constexpr (PER == 4) {  // lanes with bits 4, 3 = u hold pair u's sums from the second level on
            z = pw_fold(pw_fold(v[0][2], v[2][2], 16, h16), pw_fold(v[1][2], v[3][2], 16, h16), 8, h8);
            if (any) {
                const double x = pw_fold(pw_fold(v[0][0], v[2][0], 16, h16), pw_fold(v[1][0], v[3][0], 16, h16),
                                         8, h8);
                const double y = pw_fold(pw_fold(v[0][1], v[2][1], 16, h16), pw_fold(v[1][1], v[3][1], 16, h16),
                                         8, h8);
                // bit 1 set: z, else bit 2 clear: x, set: y
                z = pw_fold(pw_fold(x, y, 4, h4), pw_xor_add(z, 4), 2, h2);
            } else {
                z = pw_xor_add(pw_xor_add(z, 4), 2);
            }
            u = (lane >> 3) & 3;
            part = lane & 7;
        } else if constexpr (PER == 2) {  // bit 4 = u
            z = pw_xor_add(pw_fold(v[0][2], v[1][2], 16, h16), 8);
            if (any) {
                const double x = pw_fold(v[0][0], v[1][0], 16, h16), y = pw_fold(v[0][1], v[1][1], 16, h16);
                // bit 2 set: z, else bit 3 clear: x, set: y
                z = pw_fold(pw_fold(x, y, 8, h8), z, 4, h4);
            } else {
                z = pw_xor_add(z, 4);
            }
            z = pw_xor_add(z, 2);
            u = lane >> 4;
            part = lane & 15;
        } else {
            z = v[0][2];
            if (any) {  // bit 4 set: z, else bit 3 clear: x, set: y
                const double x = pw_fold(v[0][0], z, 16, h16), y = pw_xor_add(v[0][1], 16);
                z = pw_fold(x, h16 ? x : y, 8, h8);
            } else {
                z = pw_xor_add(pw_xor_add(z, 16), 8);
            }
            z = pw_xor_add(pw_xor_add(z, 4), 2);
            u = 0;
            part = lane;
        }
        z = pw_xor_add(z, 1);
        const int p = __shfl_sync(0xffffffffu, my_p, u), q = __shfl_sync(0xffffffffu, my_q, u);
        const int need = __shfl_sync(0xffffffffu, my_need, u);
        if (u < nb) {
            if (part == PART_Z) sh.apq[k0 + u] = z;
            if (part == PART_X && (need & 1)) sh.d[p] = z;
            if (part == PART_Y && (need & 2)) sh.d[q] = z;
        }
    }
}

// Solves one factor; every thread of the group calls it.  Writes status, sweeps,
// the rotation count and the stop rule (HSVD_STOP_*) through out_status /
// out_sweeps / out_rot / out_rule (thread 0; out_rule may be null).  tstop > 0
// is the tangent threshold of the early stop (Sec. 2), 0 turns it off.  W is
// formed only when V is asked for.
//
// A step has three phases with a group barrier after each: the dots of every
// pair by its warp (up to four pairs at a time), the rotations one pair per lane,
// and the column updates.  The rotation's chain of about 50 FP64 instructions
// costs a warp the same for 1 or 32 pairs (64 cycles of its quarter of the
// SM's FP64 pipe per instruction), so the pairs are packed into as few warps
// as hold them, warp `first` on; groups of one SM start at different warps so
// that they do not share a quarter.  Measured (600 factors, n in [16, 256]):
// 457 ms with a rotation per warp and every dot formed anew, 275 ms so.
//
// FEW is for factors of at most kPwFew columns, whose pairs are too few to come four
// to a warp: one or two a warp instead, on eight warps (two a quarter of the SM)
// where there are that many.  With four, 110 factors of 2048 x 16 took 5.9 ms, 3.5
// so (3.8 with every pair on a warp of its own from dots to update), 304 of n = 8
// 0.41 and 0.29 (0.38), 600 of n = 24 2.08 and 1.95 ms (4.65).  It is a template
// argument because either form costs the other's registers (1 % of a batch of
// large factors).
constexpr int kPwFew = 32;
template <int NT, bool FEW>
__device__ void pw_solve(const double *__restrict__ G, int64_t ldg, int m, int n, const int8_t *__restrict__ J,
                         int m_pad, int n_pad, double tol, double tstop, int max_sweeps, int sort,
                         const PwArrays &sh, PwScalars &sc, double *__restrict__ sigma, double *__restrict__ U,
                         int64_t ldu, double *__restrict__ V, int64_t ldv, int *out_status, int *out_sweeps,
                         long long *out_rot, int *out_rule, int bar, int first) {
    constexpr int kW = NT / kWarp;
    const int tid = threadIdx.x & (NT - 1), lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        sc.rot = 0;
        sc.err = 0;
        sc.bad = 0;
        sc.big = 0;
        sc.total = 0;
    }
    grp_sync<NT>(bar);

    // load and border (Eq. 4.1): pad columns are unit vectors in fresh rows
    int bad = 0;
    for (int j = warp; j < n_pad; j += kW) {
        double *g = sh.g(j, m_pad);
        for (int i = lane; i < m_pad; i += kWarp) {
            double v = 0.0;
            if (j < n) {
                if (i < m) v = G[i + (int64_t)j * ldg];
            } else if (i == m + (j - n)) {
                v = 1.0;
            }
            bad |= !isfinite(v);
            g[i] = v;
        }
        if (V) {
            double *w = sh.w(j, n_pad);
            for (int i = lane; i < n_pad; i += kWarp) w[i] = (i == j) ? 1.0 : 0.0;
        }
    }
    if (bad) atomicOr(&sc.bad, 1);
    for (int j = tid; j < n_pad; j += NT) {
        const int sj = (j < n) ? (int)J[j] : 1;
        sh.sg[j] = sj > 0 ? 1 : -1;
        if (sj != 1 && sj != -1) atomicOr(&sc.bad, 2);
        sh.d[j] = -1.0;
    }
    grp_sync<NT>(bar);
    if (sc.bad) {
        const int b = sc.bad;
        grp_sync<NT>(bar);
        if (tid == 0) {
            *out_status = (b & 2) ? HSVD_ERR_ARG : HSVD_ERR_NONFINITE;
            *out_sweeps = 0;
            *out_rot = 0;
            if (out_rule) *out_rule = HSVD_STOP_NONE;
        }
        return;
    }
    // initial positions: J+ columns in index order, then J- columns
    for (int j = tid; j < n_pad; j += NT) {
        int before = 0;
        for (int i = 0; i < j; ++i) before += (sh.sg[i] > 0) == (sh.sg[j] > 0);
        int nplus = 0;
        if (sh.sg[j] < 0)
            for (int i = 0; i < n_pad; ++i) nplus += sh.sg[i] > 0;
        sh.pos[(sh.sg[j] > 0 ? 0 : nplus) + before] = j;
    }
    grp_sync<NT>(bar);
    if (sort) pw_reorder<NT>(sh, m_pad, n_pad, bar);

    long long rot_total = 0;
    int sweep = 0, status = HSVD_NOT_CONVERGED, rule = HSVD_STOP_NONE;
    const int half = n_pad / 2;
    const int pwarp = (warp - first) & (kW - 1);  // which 32 pairs this warp rotates
    for (sweep = 1; sweep <= max_sweeps; ++sweep) {
        for (int s = 0; s < n_pad; ++s) {
            if constexpr (FEW) {
                if (half <= 8) pw_step_dots<NT, 1>(sh, m_pad, n_pad, s);
                else pw_step_dots<NT, 2>(sh, m_pad, n_pad, s);
            } else {
                pw_step_dots<NT, 4>(sh, m_pad, n_pad, s);
            }
            grp_sync<NT>(bar);
            // the rotations, one pair per lane
            for (int k0 = 32 * pwarp; k0 < half; k0 += 32 * kW) {
                const int k = k0 + lane;
                int rot = 0;
                bool large = false;
                if (k < half) {
                    const int p = sh.pq[k] & 0xffff, q = sh.pq[k] >> 16;
                    const int hyp = (sh.sg[p] == sh.sg[q]) ? -1 : 1;
                    double t, c;
                    const int d = pw_decision(sh.d[p], sh.d[q], sh.apq[k], hyp, tol, t, c);
                    rot = d == 1;
                    if (d == 2) atomicExch(&sc.err, HSVD_ERR_RANK);
                    if (rot) {
                        sh.apq[k] = c;
                        sh.t[k] = t;
                        sh.d[p] = -1.0;
                        sh.d[q] = -1.0;
                        large = tstop > 0.0 && pw_larger(t, tstop);
                    }
                    sh.hyp[k] = rot ? hyp : 0;
                }
                const unsigned rmask = __ballot_sync(0xffffffffu, rot);
                if (tstop > 0.0 && __any_sync(0xffffffffu, large) && lane == 0) sc.big = 1;
                if (lane == 0 && rmask) {
                    atomicAdd(&sc.rot, __popc(rmask));
                    rot_total += __popc(rmask);
                }
            }
            grp_sync<NT>(bar);
            if (sc.err) break;
            // the column updates
            for (int k = warp; k < half; k += kW) {
                const int hyp = sh.hyp[k];
                if (!hyp) continue;
                const int p = sh.pq[k] & 0xffff, q = sh.pq[k] >> 16;
                const double c = sh.apq[k], t = sh.t[k], ht = hyp < 0 ? -t : t;
                double *gp = sh.g(p, m_pad), *gq = sh.g(q, m_pad);
                pw_rotate(gp, gq, gp, gq, m_pad, lane, ht, t, c);
                if (V) {
                    double *wp = sh.w(p, n_pad), *wq = sh.w(q, n_pad);
                    pw_rotate(wp, wq, wp, wq, n_pad, lane, ht, t, c);
                }
            }
            grp_sync<NT>(bar);
        }
        if (sc.err) {
            status = sc.err;
            break;
        }
        const int nrot = sc.rot, big = sc.big;
        grp_sync<NT>(bar);
        if (tid == 0) {
            sc.rot = 0;
            sc.big = 0;
        }
        if (nrot == 0 || (tstop > 0.0 && !big)) {  // (00)_2 or (01)_2 of Eq. 4.2
            status = HSVD_OK;
            rule = nrot == 0 ? HSVD_STOP_ORTHO : HSVD_STOP_TANGENT;
            break;
        }
        if (sort) pw_reorder<NT>(sh, m_pad, n_pad, bar);
        else grp_sync<NT>(bar);
    }
    if (sweep > max_sweeps) sweep = max_sweeps;
    grp_sync<NT>(bar);

    if (status == HSVD_OK || status == HSVD_NOT_CONVERGED) {
        for (int j = warp; j < n; j += kW) {
            const int e = pw_finish_column(sh.g(j, m_pad), V ? sh.w(j, n_pad) : nullptr, m, n, j, lane, sigma, U, ldu, V, ldv);
            if (e) atomicExch(&sc.err, e);
        }
        grp_sync<NT>(bar);
        if (sc.err) status = sc.err;
    }
    if (lane == 0 && rot_total) atomicAdd(&sc.total, (unsigned long long)rot_total);
    grp_sync<NT>(bar);
    if (tid == 0) {
        *out_status = status;
        *out_sweeps = sweep;
        *out_rot = (long long)sc.total;
        if (out_rule) *out_rule = status == HSVD_OK ? rule : HSVD_STOP_NONE;
    }
    grp_sync<NT>(bar);
}

// Where position x sits at step `s` of the modified modulus strategy on r
// indices: slot 2 k for the smaller index of pair k, 2 k + 1 for the larger
// (the inverse of modulus_pair).
__host__ __device__ __forceinline__ int modulus_slot(int r, int s, int x) {
    const int c = (r - 1 + (s % r)) % r;
    const int low = (c + 1) / 2;  // pairs with a sum of c; an even c has the pair (c/2, c/2 + r/2) next
    if (!(c & 1)) {
        if (x == c / 2) return 2 * low;
        if (x == c / 2 + r / 2) return 2 * low + 1;
    }
    if (x <= c) return x < c - x ? 2 * x : 2 * (c - x) + 1;
    const int y = c + r - x, k = low + ((c & 1) ? 0 : 1) - (c + 1);
    return x < y ? 2 * (k + x) : 2 * (k + y) + 1;
}

// rows of G's working copy: m plus the bordering row of an odd n, rounded up to 32
__host__ __device__ inline int pw_rows_pad(int64_t m, int64_t n) {
    const int64_t n_pad = n + (n & 1);
    const int64_t rows = m + (n_pad - n);
    return (int)((rows + 31) / 32 * 32);
}

}  // namespace hsvd
