// pw_cluster.cuh -- one factor of the pointwise method on a thread-block
// cluster: the body of the single-factor kernel (pointwise.cu) and of the
// batched kernel for a few factors (batched.cu).
#pragma once

#include <cooperative_groups.h>

#include "pw_core.cuh"

namespace hsvd {

namespace cg = cooperative_groups;

constexpr int kMaxCl = 16;       // CTAs of a cluster at most (16 is beyond the portable 8)
constexpr int kMaxClPairs = 16;  // pairs (warps) per CTA at most
// Dynamic shared memory of a CTA at most.  The kernels' limit is set to it, whatever
// a call needs: the limit belongs to the function, so a call that lowered it to
// its own size would fail another host thread's launch.
constexpr size_t kClSmemMax = 220 * 1024;

// dynamic shared memory of a CTA with P pairs
__host__ __device__ inline size_t pw_cluster_smem(int64_t m_pad, int64_t n_pad, int64_t P, bool has_v) {
    const size_t S = 2 * (size_t)P, L = (size_t)m_pad + (has_v ? n_pad : 0);
    return 2 * S * L * sizeof(double) + 2 * S * (sizeof(double) + sizeof(int)) +
           (size_t)n_pad * (sizeof(double) + sizeof(int)) + (size_t)P * n_pad * 2 * sizeof(int);
}

// One factor on a cluster of C CTAs; CTA r owns the slots of pairs [r P, r P + P),
// one warp per pair.  A slot holds a column (its rows of G, then of W) with
// its dot with itself (negative: to be formed) and its number and sign.
// In a step a warp forms its pair's dots, every lane the rotation, and the
// updated columns go straight into the slots, local or of another CTA, where
// the next step of the modulus strategy wants them, in the other of two slot
// buffers: one cluster barrier per step, and every load is local.
//
// The bound is the chain of FP64 instructions of one warp (one per 64 cycles
// whatever the lanes do): 3 m / 32 for the dots, 6 to sum them (the three sums
// folded together), about 50 for the rotation, 4 (m + n) / 32 for the update.
// Hence one pair per quarter of an SM's FP64 pipe: P <= 4 up to n = 128.
// Measured (N(0,1), whole call, against the one-CTA kernel before it): n = 24:
// 0.96 against 1.93 ms (0.84 with the scratch pool), n = 64: 2.39 against 13.2 ms,
// n = 128: 5.7 against 52.5 ms (4.4 us a step, where one SM's FP64 rate made it 40 us).  The arithmetic is
// pw_solve's, so the bits are those of the batched form.
// out: status, sweeps, stop rule.
static __device__ __forceinline__ void pw_cluster_solve(
    double *smem, const double *__restrict__ G, int64_t ldg, int m, int n, const int8_t *__restrict__ J, int P,
    double tol, double tstop, int max_sweeps, int sort, double *__restrict__ sigma, double *__restrict__ U,
    int64_t ldu, double *__restrict__ V, int64_t ldv, int *__restrict__ out, long long *__restrict__ rot_out) {
    const int n_pad = n + (n & 1), m_pad = pw_rows_pad(m, n);
    __shared__ int s_bad, s_err[2], s_fin;
    __shared__ int cnt[kMaxCl], cbig[kMaxCl], cbad[kMaxCl];  // every CTA's word, in every CTA
    __shared__ int wcnt[kMaxClPairs], wbig[kMaxClPairs];
    __shared__ unsigned long long s_total;
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x;
    const int half = n_pad / 2, L = m_pad + (V ? n_pad : 0), S = 2 * P;
    double *cols = smem;                              // [2][S][L]
    double *dots = cols + (size_t)2 * S * L;          // [2][S] dots of the columns with themselves
    double *key = dots + 2 * S;                       // [n_pad] sort keys by position
    int *id = reinterpret_cast<int *>(key + n_pad);   // [2][S] column * 2 + (sign > 0)
    int *ksg = id + 2 * S;                            // [n_pad] signs by position
    int2 *to_tab = reinterpret_cast<int2 *>(ksg + n_pad);  // [P][n_pad] slots a step's two columns go to
    int *colat = reinterpret_cast<int *>(key);        // [n_pad] columns by position (start only)
    auto col = [&](int b, int sl) { return cols + ((size_t)b * S + sl) * L; };

    if (tid == 0) {
        s_bad = 0;
        s_err[0] = s_err[1] = 0;
        s_fin = 0;
        s_total = 0;
    }
    int bad = 0;
    for (int j = tid; j < n_pad; j += nthr) {
        const int sj = (j < n) ? (int)J[j] : 1;
        ksg[j] = sj > 0 ? 1 : -1;
        if (sj != 1 && sj != -1) bad |= 2;
    }
    __syncthreads();
    // initial positions: J+ columns in index order, then J- columns
    for (int j = tid; j < n_pad; j += nthr) {
        int before = 0, nplus = 0;
        for (int i = 0; i < n_pad; ++i) {
            nplus += ksg[i] > 0;
            before += i < j && ksg[i] == ksg[j];
        }
        colat[(ksg[j] > 0 ? 0 : nplus) + before] = j;
    }
    __syncthreads();
    const int k = rank * P + warp;  // this warp's pair
    const bool act = warp < P && k < half;
    if (act) {
        int a, b;
        // where step s sends them: the positions' slots at step s + 1
        for (int s = lane; s < n_pad; s += kWarp) {
            modulus_pair(n_pad, s, k, a, b);
            to_tab[warp * n_pad + s] = make_int2(modulus_slot(n_pad, s + 1, a), modulus_slot(n_pad, s + 1, b));
        }
        modulus_pair(n_pad, 0, k, a, b);
        for (int u = 0; u < 2; ++u) {
            const int j = colat[u ? b : a], sl = 2 * warp + u;
            double *x = col(0, sl);
            // border (Eq. 4.1): pad columns are unit vectors in fresh rows
            for (int i = lane; i < m_pad; i += kWarp) {
                double v = 0.0;
                if (j < n) {
                    if (i < m) v = G[i + (int64_t)j * ldg];
                } else if (i == m + (j - n)) {
                    v = 1.0;
                }
                if (!isfinite(v)) bad |= 1;
                x[i] = v;
            }
            for (int i = m_pad + lane; i < L; i += kWarp) x[i] = (i - m_pad == j) ? 1.0 : 0.0;
            if (lane == 0) {
                dots[sl] = -1.0;
                id[sl] = 2 * j + (ksg[j] > 0);
            }
        }
    }
    if (bad) atomicOr(&s_bad, bad);
    cluster.sync();  // every CTA loaded and running before any remote write
    if (tid < C) *cluster.map_shared_rank(&cbad[rank], tid) = s_bad;
    cluster.sync();
    bad = 0;
    for (int r = 0; r < C; ++r) bad |= cbad[r];
    if (bad) {
        if (rank == 0 && tid == 0) {
            out[0] = (bad & 2) ? HSVD_ERR_ARG : HSVD_ERR_NONFINITE;
            out[1] = 0;
            out[2] = HSVD_STOP_NONE;
            *rot_out = 0;
        }
        cluster.sync();  // no CTA leaves while another may still write its word into it
        return;
    }

    int cur = 0;  // the slot buffer that holds the columns
    // slot `to` (of all the cluster's) in the other buffer: its column; its words (one lane)
    auto dst_col = [&](int to) {
        return cluster.map_shared_rank(cols, to / S) + ((size_t)(cur ^ 1) * S + to % S) * L;
    };
    auto put_words = [&](int to, double d, int c) {
        cluster.map_shared_rank(dots, to / S)[(cur ^ 1) * S + to % S] = d;
        cluster.map_shared_rank(id, to / S)[(cur ^ 1) * S + to % S] = c;
    };
    // diagonal sorting (Sec. 4): the keys of every position into every CTA,
    // then each column to its new position's slot at step 0
    auto reorder = [&]() {
        int pos[2] = {0, 0};
        double dd[2] = {0.0, 0.0};
        if (act) {
            modulus_pair(n_pad, 0, k, pos[0], pos[1]);
            for (int u = 0; u < 2; ++u) {
                const int sl = 2 * warp + u;
                const double *x = col(cur, sl);
                double d = dots[cur * S + sl];
                if (pw_missing(d)) {
                    d = 0.0;
                    for (int i = lane; i < m_pad; i += kWarp) d = fma(x[i], x[i], d);
                    d = warp_sum(d);
                }
                dd[u] = d;
                if (lane < C) {
                    cluster.map_shared_rank(key, lane)[pos[u]] = d;
                    cluster.map_shared_rank(ksg, lane)[pos[u]] = (id[cur * S + sl] & 1) ? 1 : -1;
                }
            }
        }
        cluster.sync();
        if (act) {
            for (int u = 0; u < 2; ++u) {
                const int sl = 2 * warp + u, a = pos[u], grp = ksg[a];
                const double ka = key[a];
                int rk = 0, nplus = 0;
                for (int b = lane; b < n_pad; b += kWarp) {
                    nplus += ksg[b] > 0;
                    if (ksg[b] == grp && b != a && pw_before(key[b], ka, grp, b < a)) ++rk;
                }
                rk = __reduce_add_sync(0xffffffffu, rk);
                nplus = __reduce_add_sync(0xffffffffu, nplus);
                const int to = modulus_slot(n_pad, 0, (grp > 0 ? 0 : nplus) + rk);
                const double *x = col(cur, sl);
                double *y = dst_col(to);
                for (int i = lane; i < L; i += kWarp) y[i] = x[i];
                if (lane == 0) put_words(to, dd[u], id[cur * S + sl]);
            }
        }
        cluster.sync();
        cur ^= 1;
    };
    if (sort) reorder();

    long long rot_total = 0;
    int sweep = 0, status = HSVD_NOT_CONVERGED, rule = HSVD_STOP_NONE;
    for (sweep = 1; sweep <= max_sweeps; ++sweep) {
        int rots = 0, big = 0, err = 0;
        for (int s = 0; s < n_pad; ++s) {
            if (act) {
                const int slp = 2 * warp, slq = slp + 1;
                const double *gp = col(cur, slp), *gq = col(cur, slq);
                const double kp = dots[cur * S + slp], kq = dots[cur * S + slq];
                const int ip = id[cur * S + slp], iq = id[cur * S + slq];
                const bool np = pw_missing(kp), nq = pw_missing(kq);
                double x, y, z;
                pw_dots_sel(np, nq, gp, gq, m_pad, lane, x, y, z);
                // sums of x, y, z: lanes 0-7, 8-15 and 16-31 end with one each
                const bool h16 = lane & 16, h8 = lane & 8;
                double v;
                if (np || nq) {
                    x = pw_fold(x, z, 16, h16);
                    y = pw_xor_add(y, 16);
                    if (h16) y = x;
                    v = pw_fold(x, y, 8, h8);
                } else {
                    v = pw_xor_add(pw_xor_add(z, 16), 8);
                }
                v = pw_xor_add(pw_xor_add(pw_xor_add(v, 4), 2), 1);
                const double app = np ? __shfl_sync(0xffffffffu, v, 0) : kp;
                const double aqq = nq ? __shfl_sync(0xffffffffu, v, 8) : kq;
                const double apq = __shfl_sync(0xffffffffu, v, 16);
                const int2 to = to_tab[warp * n_pad + s];
                double *yp = dst_col(to.x), *yq = dst_col(to.y);
                const int hyp = ((ip ^ iq) & 1) ? 1 : -1;
                double t, c;
                const int dec = pw_decision(app, aqq, apq, hyp, tol, t, c);
                if (dec == 2 && lane < C) *cluster.map_shared_rank(&s_err[cur], lane) = HSVD_ERR_RANK;
                if (dec == 1) {
                    ++rots;
                    big |= tstop > 0.0 && pw_larger(t, tstop);
                    pw_rotate(gp, gq, yp, yq, L, lane, hyp < 0 ? -t : t, t, c);
                } else {
                    for (int i = lane; i < L; i += kWarp) {
                        const double u = gp[i], w = gq[i];
                        yp[i] = u;
                        yq[i] = w;
                    }
                }
                if ((lane & 15) == 0) put_words(h16 ? to.y : to.x, dec == 1 ? -1.0 : (h16 ? aqq : app), h16 ? iq : ip);
            }
            cluster.sync();
            err = s_err[cur];  // written before the barrier only: every CTA decides alike
            cur ^= 1;
            if (err) break;
        }
        rot_total += rots;
        if (err) {
            status = err;
            break;
        }
        if (lane == 0) {
            wcnt[warp] = rots;
            wbig[warp] = big;
        }
        __syncthreads();
        if (tid < C) {
            int r = 0, g = 0;
            for (int w = 0; w < nthr / 32; ++w) {
                r += wcnt[w];
                g |= wbig[w];
            }
            *cluster.map_shared_rank(&cnt[rank], tid) = r;
            *cluster.map_shared_rank(&cbig[rank], tid) = g;
        }
        cluster.sync();
        int nrot = 0;
        big = 0;
        for (int r = 0; r < C; ++r) {
            nrot += cnt[r];
            big |= cbig[r];
        }
        if (nrot == 0 || (tstop > 0.0 && !big)) {  // (00)_2 or (01)_2 of Eq. 4.2
            status = HSVD_OK;
            rule = nrot == 0 ? HSVD_STOP_ORTHO : HSVD_STOP_TANGENT;
            break;
        }
        if (sort) reorder();
    }
    if (sweep > max_sweeps) sweep = max_sweeps;
    if (act && (status == HSVD_OK || status == HSVD_NOT_CONVERGED)) {
        for (int u = 0; u < 2; ++u) {
            const int sl = 2 * warp + u, j = id[cur * S + sl] >> 1;
            if (j >= n) continue;
            const double *x = col(cur, sl);
            const int e = pw_finish_column(x, x + m_pad, m, n, j, lane, sigma, U, ldu, V, ldv);
            if (e) atomicExch(cluster.map_shared_rank(&s_fin, 0), e);
        }
    }
    if (act && lane == 0 && rot_total)
        atomicAdd(cluster.map_shared_rank(&s_total, 0), (unsigned long long)rot_total);
    cluster.sync();  // no CTA leaves while another may still write into it
    if (rank == 0 && tid == 0) {
        if (s_fin) status = s_fin;
        out[0] = status;
        out[1] = sweep;
        out[2] = status == HSVD_OK ? rule : HSVD_STOP_NONE;
        *rot_out = (long long)s_total;
    }
}

}  // namespace hsvd
