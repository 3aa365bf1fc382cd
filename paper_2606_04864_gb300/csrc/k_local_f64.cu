// FP64 local solves (Section 3.2: z_f = sum_i R_i^T A_i^{-1} R_i r', and the
// restriction r_c = R_0 r' of Section 3.1 fused in): the FP64 preconditioner,
// and the shift-invert solves of the eigenproblems.  One thread block per
// subdomain, block rows of 32, band Cholesky factor tiles with inverted
// diagonal blocks (ams_internal.h).
//
// Forward, K = 0 .. nb-1:
//   t = r'_K - sum_d L_{K,K-c+d} y_{K-c+d},  y_K = L_KK^{-1} t
// Backward (right-looking), K = nb-1 .. 0:
//   w = y_K - pending_K,  x_K = L_KK^{-T} w,  pending_{K-c+d} += L_{K,K-c+d}^T x_K
//
// What bounds it: the FP64 pipe, about two lanes a clock and SM, so 17 clocks
// a warp instruction whatever its lanes do.  A task is a pair of rows (a,
// 31 - a) of one right-hand side: the two rows of the triangular tiles
// together take 33 multiply-adds, so no lane runs masked ones (a lane per
// row with masks runs 64 a tile pair), the columns past the last right-hand
// side have no task, and the coefficients are broadcasts.  The backward sweep
// frees a ring slot as soon as its row is done (see k_local_mma.cu).
// A lane per row with masks: 16 columns on 512 subdomains of 8^3 (c = 2) 1.54
// ms a launch, on 256 of 32^2 (c = 1, then 32 columns) 2.30; 5 columns on 343 of
// 8^3 530 us.  This: 1.17 ms, 0.71 (16 columns) and 400-415 us, the last with
// three blocks on some SMs and two on others.
#include <cstdint>

#include "ams_internal.h"
#include "kernels.cuh"
#include "launch.h"

namespace ams {

// Sum over the S neighbouring lanes that share a task.
template <int S>
__device__ __forceinline__ double lane_sum(double v) {
#pragma unroll
    for (int o = 1; o < S; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// NT tasks per thread (1: up to 16 right-hand sides, 2: up to 32); S lanes
// per task, each taking every S-th term of its dot products.  A warp's
// multiply-adds run on its own quarter of the SM at a quarter of the rate, so
// S fills the last warp and gives a block at least four.  PAD: there are
// columns between the right-hand sides and ld; they have no task, but the
// coarse products and the prolongation read them, so they get zeros.
template <int NT, int MM, int S, bool PAD>
__global__ void __launch_bounds__(256)
k_local_f64(const SubInfo* __restrict__ subs, const double* __restrict__ fac, const double* __restrict__ rin,
            const double* __restrict__ qin, const CgScalars* __restrict__ csc, const double* __restrict__ rowscale,
            double* __restrict__ zf, const double* __restrict__ psi, double* __restrict__ rc, int ld, int ncols,
            int cmax, int depth, const SolveState* st) {
    pdl_wait();
    if (st != nullptr && st->done) return;
    extern __shared__ __align__(16) double sm64[];
    const SubInfo sub = subs[blockIdx.x];
    const int c = sub.c, nb = sub.nb, n = sub.n, m = sub.m;
    const int part = (int)threadIdx.x % S;                     // which terms of a dot product
    const int D = depth, nbuf = D + 1;
    const int64_t brs = blockrow_elems(c), brs_max = blockrow_elems(cmax);
    const int blk = 32 * ncols;                                // one block row of the right-hand sides
    double* bufs = sm64;                                       // nbuf * brs_max
    double* tmp = bufs + nbuf * brs_max;                       // t, then w
    double* ring = tmp + blk;                                  // c blocks: y; backward: block 0 holds x ...
    double* pnd = ring + (int64_t)cmax * blk;                  // ... and c blocks of pending sums, by their own tasks
    const double* F = fac + sub.fac_off;
    const int ntask = 16 * ncols;
    int col[NT], ra[NT], rb[NT];
    bool on[NT], upd[NT];
    double al[NT];
#pragma unroll
    for (int k = 0; k < NT; ++k) {
        const int task = ((int)threadIdx.x + k * (int)blockDim.x) / S;
        on[k] = task < ntask;
        col[k] = on[k] ? task % ncols : 0;
        ra[k] = on[k] ? task / ncols : 0;
        rb[k] = 31 - ra[k];
        // r' = r - alpha q for (system, rhs) pairs still iterating (see ResidIn)
        al[k] = 0.0;
        upd[k] = false;
        if (qin != nullptr && on[k]) {
            const CgScalars cs = csc[(int64_t)sub.seg * ld + col[k]];
            upd[k] = cs.active != 0;
            if (upd[k]) al[k] = cs.alpha;
        }
    }
    double racc[NT][MM];
#pragma unroll
    for (int k = 0; k < NT; ++k)
#pragma unroll
        for (int i = 0; i < MM; ++i) racc[k][i] = 0.0;

    auto copy_row = [&](int K) {
        block_copy_async(bufs + (int64_t)(K % nbuf) * brs_max, F + (int64_t)K * brs, brs * sizeof(double));
    };
    // r' of the next block row is loaded while the current one is computed
    double rn[NT][2], qn[NT][2];
    auto load_in = [&](int K) {
#pragma unroll
        for (int k = 0; k < NT; ++k)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = K * 32 + (h ? rb[k] : ra[k]);
                rn[k][h] = 0.0;
                qn[k][h] = 0.0;
                if (on[k] && K < nb && row < n) {
                    const int64_t e = (sub.row0 + row) * ld + col[k];
                    rn[k][h] = rin[e];
                    if (upd[k]) qn[k][h] = qin[e];
                }
            }
    };
    for (int j = 0; j < D; ++j) {
        if (j < nb) copy_row(j);
        cp_async_commit();
    }
    load_in(0);
    cp_async_wait_n(D - 1);
    __syncthreads();
    // ---------------- forward ----------------
#pragma unroll 1
    for (int K = 0; K < nb; ++K) {
        const double* B = bufs + (int64_t)(K % nbuf) * brs_max;
        double v[NT][2];
#pragma unroll
        for (int k = 0; k < NT; ++k)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                v[k][h] = upd[k] ? fma(-al[k], qn[k][h], rn[k][h]) : rn[k][h];
                const int row = K * 32 + (h ? rb[k] : ra[k]);
                if (on[k] && row < n) {
                    if (rowscale != nullptr) v[k][h] *= rowscale[sub.row0 + row];
                    if (rc != nullptr && part == 0) {
                        const double* pr = psi + sub.psi_off + (int64_t)row * m;
#pragma unroll
                        for (int i = 0; i < MM; ++i)
                            if (i < m) racc[k][i] = fma(pr[i], v[k][h], racc[k][i]);
                    }
                }
            }
        load_in(K + 1);
#pragma unroll
        for (int k = 0; k < NT; ++k) {
            double a = part == 0 ? v[k][0] : 0.0, b = part == 0 ? v[k][1] : 0.0;
            if (on[k] && K >= c) {   // L_{K,K-c}: columns q >= row of M
                const double* y = ring + (int64_t)(K % c) * blk + col[k];
                int q = ra[k] + part;
                for (; q < rb[k]; q += S) a = fma(-B[tile_idx(ra[k], q)], y[q * ncols], a);
                for (; q < 32; q += S) {
                    const double yq = y[q * ncols];
                    a = fma(-B[tile_idx(ra[k], q)], yq, a);
                    b = fma(-B[tile_idx(rb[k], q)], yq, b);
                }
            }
            for (int d = 1; d < c; ++d) {
                const int src = K - c + d;
                if (src < 0 || !on[k]) continue;
                const double* y = ring + (int64_t)(src % c) * blk + col[k];
                const double* T = B + d * 1024;
#pragma unroll 4
                for (int q = part; q < 32; q += S) {
                    const double yq = y[q * ncols];
                    a = fma(-T[tile_idx(ra[k], q)], yq, a);
                    b = fma(-T[tile_idx(rb[k], q)], yq, b);
                }
            }
            v[k][0] = a = lane_sum<S>(a);
            v[k][1] = b = lane_sum<S>(b);
            if (on[k] && part == 0) {
                tmp[ra[k] * ncols + col[k]] = a;
                tmp[rb[k] * ncols + col[k]] = b;
            }
        }
        __syncthreads();                       // t complete; every thread is past block row K - 1
        if (K + D < nb) copy_row(K + D);       // into its slot
        cp_async_commit();
#pragma unroll
        for (int k = 0; k < NT; ++k) {
            const double* t = tmp + col[k];
            double a = part == 0 ? B[c * 1024 + ra[k]] * v[k][0] : 0.0;
            double b = part == 0 ? B[c * 1024 + rb[k]] * v[k][1] : 0.0;
            if (on[k]) {
                int q = part;
                for (; q < ra[k]; q += S) {
                    const double tq = t[q * ncols];
                    a = fma(B[tile_idx(ra[k], q)], tq, a);
                    b = fma(B[tile_idx(rb[k], q)], tq, b);
                }
                for (; q < rb[k]; q += S) b = fma(B[tile_idx(rb[k], q)], t[q * ncols], b);
            }
            a = lane_sum<S>(a);
            b = lane_sum<S>(b);
            if (!on[k] || part != 0) continue;
            double* y = ring + (int64_t)(K % c) * blk + col[k];
            y[ra[k] * ncols] = a;
            y[rb[k] * ncols] = b;
            const int64_t e = (sub.row0 + K * 32) * ld + col[k];
            if (K * 32 + ra[k] < n) zf[e + (int64_t)ra[k] * ld] = a;
            if (K * 32 + rb[k] < n) zf[e + (int64_t)rb[k] * ld] = b;
        }
        cp_async_wait_n(D - 1);                // block row K + 1 has landed
        __syncthreads();
    }
    if (rc != nullptr) {   // the row pairs' sums, in order
#pragma unroll 1
        for (int i = 0; i < m; ++i) {
#pragma unroll
            for (int k = 0; k < NT; ++k)
#pragma unroll
                for (int j = 0; j < MM; ++j)
                    if (j == i && on[k] && part == 0) tmp[ra[k] * ncols + col[k]] = racc[k][j];
            __syncthreads();
            for (int cc = threadIdx.x; cc < ncols; cc += blockDim.x) {
                double s = 0.0;
                for (int a = 0; a < 16; ++a) s += tmp[a * ncols + cc];
                rc[(sub.coff + i) * ld + cc] = s;
            }
            __syncthreads();
        }
    }
    pdl_trigger();
    // ---------------- backward ----------------
    // block rows nb - nbuf .. nb - 1 are still in the ring
    cp_async_wait_all();
    const int Rres = nb > nbuf ? nb - nbuf : 0;
    double yn[NT][2];
    auto load_y = [&](int K) {
#pragma unroll
        for (int k = 0; k < NT; ++k)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = K * 32 + (h ? rb[k] : ra[k]);
                yn[k][h] = (on[k] && K >= 0 && row < n) ? zf[(sub.row0 + row) * ld + col[k]] : 0.0;
            }
    };
#pragma unroll
    for (int k = 0; k < NT; ++k)
        if (on[k] && part == 0)
            for (int d = 0; d < c; ++d) {
                pnd[d * blk + ra[k] * ncols + col[k]] = 0.0;
                pnd[d * blk + rb[k] * ncols + col[k]] = 0.0;
            }
    load_y(nb - 1);
#pragma unroll 1
    for (int K = nb - 1; K >= 0; --K) {
        const double* B = bufs + (int64_t)(K % nbuf) * brs_max;
        double v[NT][2];
#pragma unroll
        for (int k = 0; k < NT; ++k) {
            if (!on[k] || part != 0) continue;
            double* p = pnd + (K % c) * blk + col[k];
            v[k][0] = yn[k][0] - p[ra[k] * ncols];
            v[k][1] = yn[k][1] - p[rb[k] * ncols];
            p[ra[k] * ncols] = 0.0;
            p[rb[k] * ncols] = 0.0;
            tmp[ra[k] * ncols + col[k]] = v[k][0];
            tmp[rb[k] * ncols + col[k]] = v[k][1];
        }
        load_y(K - 1);
        __syncthreads();                       // w complete; every thread is past block row K + 1
        if (K - D >= 0 && K - D < Rres) copy_row(K - D);
        cp_async_commit();
#pragma unroll
        for (int k = 0; k < NT; ++k) {
            const double* t = tmp + col[k];
            double a = 0.0, b = 0.0;
            if (on[k] && part == 0) {
                a = B[c * 1024 + ra[k]] * v[k][0];
                b = B[c * 1024 + rb[k]] * v[k][1];
            }
            if (on[k]) {
                int r = ra[k] + 1 + part;
                for (; r <= rb[k]; r += S) a = fma(B[tile_idx(r, ra[k])], t[r * ncols], a);
                for (; r < 32; r += S) {
                    const double tr = t[r * ncols];
                    a = fma(B[tile_idx(r, ra[k])], tr, a);
                    b = fma(B[tile_idx(r, rb[k])], tr, b);
                }
            }
            a = lane_sum<S>(a);
            b = lane_sum<S>(b);
            if (!on[k] || part != 0) continue;
            double* x = ring + col[k];
            x[ra[k] * ncols] = a;
            x[rb[k] * ncols] = b;
            const int64_t e = (sub.row0 + K * 32) * ld + col[k];
            if (K * 32 + ra[k] < n) zf[e + (int64_t)ra[k] * ld] = a;
            if (K * 32 + rb[k] < n) zf[e + (int64_t)rb[k] * ld] = b;
        }
        __syncthreads();                       // x_K complete
#pragma unroll
        for (int k = 0; k < NT; ++k) {
            const double* x = ring + col[k];
            for (int d = c - 1; d >= 0; --d) {
                const int dst = K - c + d;
                if (dst < 0) break;
                const double* T = B + d * 1024;
                double a = 0.0, b = 0.0;
                if (on[k] && d > 0) {
#pragma unroll 4
                    for (int r = part; r < 32; r += S) {
                        const double xr = x[r * ncols];
                        a = fma(T[tile_idx(r, ra[k])], xr, a);
                        b = fma(T[tile_idx(r, rb[k])], xr, b);
                    }
                } else if (on[k]) {   // L_{K,K-c}: rows r <= column of M
                    int r = part;
                    for (; r <= ra[k]; r += S) {
                        const double xr = x[r * ncols];
                        a = fma(T[tile_idx(r, ra[k])], xr, a);
                        b = fma(T[tile_idx(r, rb[k])], xr, b);
                    }
                    for (; r <= rb[k]; r += S) b = fma(T[tile_idx(r, rb[k])], x[r * ncols], b);
                }
                a = lane_sum<S>(a);
                b = lane_sum<S>(b);
                if (on[k] && part == 0) {
                    double* p = pnd + (dst % c) * blk + col[k];
                    p[ra[k] * ncols] += a;
                    p[rb[k] * ncols] += b;
                }
            }
        }
        cp_async_wait_n(D - 1);                // block row K - 1 has landed (the next barrier shows it to all)
    }
    if constexpr (PAD) {
        const int npad = ld - ncols;
        for (int i = threadIdx.x; i < n * npad; i += blockDim.x)
            zf[(sub.row0 + i / npad) * ld + ncols + i % npad] = 0.0;
        if (rc != nullptr)
            for (int i = threadIdx.x; i < m * npad; i += blockDim.x)
                rc[(sub.coff + i / npad) * ld + ncols + i % npad] = 0.0;
    }
}

// One to four right-hand sides on many subdomains of one tile a block row: a
// lane per row (forward) or column (backward), NR columns a warp, with the
// triangles' other halves masked.  64 multiply-adds a lane and tile pair where
// row pairs take 33, but no lane idles and no partial sums are added up across
// lanes, which with few columns and one tile costs more FP64 instructions than
// the masks.  Left-looking in both sweeps: step K of the backward one needs
// block rows K .. K + c.
template <int NR, int MM>
__global__ void k_local_f64_rows(const SubInfo* __restrict__ subs, const double* __restrict__ fac,
                              const double* __restrict__ rin, const double* __restrict__ qin,
                              const CgScalars* __restrict__ csc, const double* __restrict__ rowscale,
                              double* __restrict__ zf, const double* __restrict__ psi, double* __restrict__ rc,
                              int ld, int cmax, int depth, const SolveState* st) {
    pdl_wait();
    if (st != nullptr && st->done) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const SubInfo S = subs[blockIdx.x];
    const int c = S.c, nb = S.nb, n = S.n;
    const int D = depth;                                       // block rows in flight
    const int nbuf = c + D + 1;
    const int64_t brs = blockrow_elems(c);
    const int64_t brs_max = blockrow_elems(cmax);
    double* bufs = (double*)smem_raw;                                  // (cmax+D+1) * brs_max
    double* ring = bufs + (int64_t)(cmax + D + 1) * brs_max;       // (cmax+1) * 32 * ld
    double* tmp = ring + (int64_t)(cmax + 1) * 32 * ld;            // 32 * ld
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int rhs0 = warp * NR;
    const double* F = fac + S.fac_off;
    const int m = S.m;

    double racc[MM][NR];
#pragma unroll
    for (int k = 0; k < MM; ++k)
#pragma unroll
        for (int j = 0; j < NR; ++j) racc[k][j] = 0.0;

    // r' = r - alpha q for (system, rhs) pairs still iterating (see ResidIn)
    double al[NR];
    bool upd[NR];
#pragma unroll
    for (int j = 0; j < NR; ++j) {
        al[j] = 0.0;
        upd[j] = false;
        if (qin != nullptr) {
            const CgScalars cj = csc[(int64_t)S.seg * ld + rhs0 + j];
            upd[j] = cj.active != 0;
            if (upd[j]) al[j] = cj.alpha;
        }
    }
    // Inputs of block row K (r and q rows, basis rows, row scale) are
    // loaded two block rows ahead into alternating register buffers and
    // kept in their loaded type until the step that uses them, so their
    // global-memory latency overlaps the substitution of earlier rows.
    auto load_fwd = [&](int K, double (&rv)[NR], double (&qv)[NR], double (&pv)[MM], double& scv) {
        const int row = K * 32 + lane;
        const bool valid = K < nb && row < n;
        const int64_t grow = S.row0 + row;
        scv = 1.0;
#pragma unroll
        for (int j = 0; j < NR; ++j) {
            rv[j] = 0.0;
            qv[j] = 0.0;
        }
#pragma unroll
        for (int k = 0; k < MM; ++k) pv[k] = 0.0;
        if (valid) {
            if (rowscale != nullptr) scv = rowscale[grow];
#pragma unroll
            for (int j = 0; j < NR; ++j) {
                rv[j] = rin[grow * ld + rhs0 + j];
                if (upd[j]) qv[j] = qin[grow * ld + rhs0 + j];
            }
            if (rc != nullptr) {
#pragma unroll
                for (int k = 0; k < MM; ++k)
                    if (k < m) pv[k] = psi[S.psi_off + (int64_t)row * m + k];
            }
        }
    };
    double rb[2][NR], qb[2][NR], sb[2];
    double pb[2][MM];
    load_fwd(0, rb[0], qb[0], pb[0], sb[0]);
    load_fwd(1, rb[1], qb[1], pb[1], sb[1]);

    // ---------------- forward ----------------
    // one commit group per block row; row K+D is requested at step K
    for (int j = 0; j < D; ++j) {
        if (j < nb) block_copy_async(bufs + (int64_t)(j % nbuf) * brs_max, F + (int64_t)j * brs, brs * sizeof(double));
        cp_async_commit();
    }
    auto fwd_step = [&](int K, double (&rv)[NR], double (&qv)[NR], double (&pb_)[MM], double& scv) {
        if (K + D < nb)
            block_copy_async(bufs + (int64_t)((K + D) % nbuf) * brs_max, F + (int64_t)(K + D) * brs,
                             brs * sizeof(double));
        cp_async_commit();
        double t[NR], pv[MM];
#pragma unroll
        for (int j = 0; j < NR; ++j) t[j] = ((upd[j] ? fma(-al[j], qv[j], rv[j]) : rv[j]) * scv);
#pragma unroll
        for (int k = 0; k < MM; ++k) pv[k] = pb_[k];
        load_fwd(K + 2, rv, qv, pb_, scv);
        cp_async_wait_n(D);
        __syncthreads();
        const double* B = bufs + (int64_t)(K % nbuf) * brs_max;
        const int row = K * 32 + lane;
        const bool valid = row < n;
        const int64_t grow = S.row0 + row;
        if (rc != nullptr) {
#pragma unroll
            for (int k = 0; k < MM; ++k)
#pragma unroll
                for (int j = 0; j < NR; ++j) racc[k][j] += pv[k] * t[j];
        }
        for (int d = 0; d < c; ++d) {
            const int src = K - c + d;
            if (src < 0) continue;
            const double* T = B + d * 1024;
            const double* ys = ring + (int64_t)(src % (c + 1)) * 32 * ld + rhs0;
#pragma unroll 8
            for (int q = 0; q < 32; ++q) {
                double coef = T[tile_idx(lane, q)];
                if (d == 0 && q < lane) coef = 0.0;
#pragma unroll
                for (int j = 0; j < NR; ++j) t[j] -= coef * ys[q * ld + j];
            }
        }
#pragma unroll
        for (int j = 0; j < NR; ++j) tmp[lane * ld + rhs0 + j] = t[j];
        __syncwarp();
        const double piv = B[c * 1024 + lane];
        double y[NR];
#pragma unroll
        for (int j = 0; j < NR; ++j) y[j] = piv * t[j];
#pragma unroll 8
        for (int q = 0; q < 32; ++q) {
            const double coef = q < lane ? B[tile_idx(lane, q)] : 0.0;
#pragma unroll
            for (int j = 0; j < NR; ++j) y[j] += coef * tmp[q * ld + rhs0 + j];
        }
        double* yr = ring + (int64_t)(K % (c + 1)) * 32 * ld + rhs0;
#pragma unroll
        for (int j = 0; j < NR; ++j) yr[lane * ld + j] = y[j];
        if (valid) {
#pragma unroll
            for (int j = 0; j < NR; ++j) zf[grow * ld + rhs0 + j] = y[j];
        }
        __syncthreads();
    };
#pragma unroll 1
    for (int K = 0; K < nb; K += 2) {
        fwd_step(K, rb[0], qb[0], pb[0], sb[0]);
        if (K + 1 < nb) fwd_step(K + 1, rb[1], qb[1], pb[1], sb[1]);
    }
    pdl_trigger();
    // restriction: reduce over lanes, lane 0 writes r_c rows of this subdomain
    if (rc != nullptr) {
#pragma unroll
        for (int k = 0; k < MM; ++k) {
#pragma unroll
            for (int j = 0; j < NR; ++j) {
                double v = racc[k][j];
                for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
                if (lane == 0 && k < m) rc[(S.coff + k) * ld + rhs0 + j] = v;
            }
        }
    }
    // ---------------- backward ----------------
    // step K needs block rows K..K+c; row K-D is requested at step K
    cp_async_wait_all();
    __syncthreads();
    for (int j = 0; j < D; ++j) {
        const int r = nb - 1 - j;
        if (r >= 0) block_copy_async(bufs + (int64_t)(r % nbuf) * brs_max, F + (int64_t)r * brs, brs * sizeof(double));
        cp_async_commit();
    }
    auto load_bwd = [&](int K, double (&wv)[NR]) {
        const int row = K * 32 + lane;
        const bool valid = K >= 0 && row < n;
        const int64_t grow = S.row0 + row;
#pragma unroll
        for (int j = 0; j < NR; ++j) wv[j] = 0.0;
        if (valid) {
#pragma unroll
            for (int j = 0; j < NR; ++j) wv[j] = zf[grow * ld + rhs0 + j];
        }
    };
    double wb[2][NR];
    load_bwd(nb - 1, wb[0]);
    load_bwd(nb - 2, wb[1]);
    auto bwd_step = [&](int K, double (&wv)[NR]) {
        if (K - D >= 0)
            block_copy_async(bufs + (int64_t)((K - D) % nbuf) * brs_max, F + (int64_t)(K - D) * brs,
                             brs * sizeof(double));
        cp_async_commit();
        double w[NR];
#pragma unroll
        for (int j = 0; j < NR; ++j) w[j] = wv[j];
        load_bwd(K - 2, wv);
        cp_async_wait_n(D);
        __syncthreads();
        const int row = K * 32 + lane;
        const bool valid = row < n;
        const int64_t grow = S.row0 + row;
        for (int d = 1; d <= c; ++d) {
            const int src = K + d;
            if (src >= nb) break;
            const double* Bs = bufs + (int64_t)(src % nbuf) * brs_max;
            const double* T = (d < c) ? Bs + (c - d) * 1024 : Bs;
            const double* xs = ring + (int64_t)(src % (c + 1)) * 32 * ld + rhs0;
#pragma unroll 8
            for (int r = 0; r < 32; ++r) {
                double coef = T[tile_idx(r, lane)];
                if (d == c && r > lane) coef = 0.0;
#pragma unroll
                for (int j = 0; j < NR; ++j) w[j] -= coef * xs[r * ld + j];
            }
        }
#pragma unroll
        for (int j = 0; j < NR; ++j) tmp[lane * ld + rhs0 + j] = w[j];
        __syncwarp();
        const double* B = bufs + (int64_t)(K % nbuf) * brs_max;
        const double piv = B[c * 1024 + lane];
        double x[NR];
#pragma unroll
        for (int j = 0; j < NR; ++j) x[j] = piv * w[j];
#pragma unroll 8
        for (int r = 0; r < 32; ++r) {
            const double coef = r > lane ? B[tile_idx(r, lane)] : 0.0;
#pragma unroll
            for (int j = 0; j < NR; ++j) x[j] += coef * tmp[r * ld + rhs0 + j];
        }
        double* xr = ring + (int64_t)(K % (c + 1)) * 32 * ld + rhs0;
#pragma unroll
        for (int j = 0; j < NR; ++j) xr[lane * ld + j] = x[j];
        if (valid) {
#pragma unroll
            for (int j = 0; j < NR; ++j) zf[grow * ld + rhs0 + j] = x[j];
        }
        __syncthreads();
    };
#pragma unroll 1
    for (int K = nb - 1; K >= 0; K -= 2) {
        bwd_step(K, wb[0]);
        if (K - 1 >= 0) bwd_step(K - 1, wb[1]);
    }
}

// Shared memory that a setup or a launch shape is checked against: the
// staging of c + depth + 1 block rows (what the lane-per-row kernel uses, an upper
// bound for the other).
size_t local_solve_smem(int cmax, int ld, size_t tf_bytes, int depth) {
    return ((size_t)(cmax + depth + 1) * blockrow_elems(cmax) + (size_t)(cmax + 1) * 32 * ld + 32 * ld) *
           tf_bytes;
}
static size_t local_f64_smem(int cmax, int ncols, int depth) {
    return ((size_t)(depth + 1) * blockrow_elems(cmax) + (size_t)(2 * cmax + 1) * 32 * ncols) * sizeof(double);
}

template <int NT, int MM, int S, bool PAD>
static cudaError_t local_f64_pad(const LocalSolveArgs& a, const double* fac, const double* psi, double* zf, double* rc) {
    // two block rows in flight hide the copies behind the FP64 pipe, and leave room for several blocks
    int depth = a.depth > 0 ? a.depth : 2;
    while (depth > 1 && local_f64_smem(a.cmax, a.ncols, depth) > 200 * 1024) --depth;
    const size_t smem = local_f64_smem(a.cmax, a.ncols, depth);
    auto kern = k_local_f64<NT, MM, S, PAD>;
    static size_t smem_set = 0;           // per template instance
    if (smem > smem_set) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        smem_set = smem;
    }
    const int threads = ((16 * a.ncols * S / NT + 31) / 32) * 32;
    return launch_kernel(a.pdl, kern, dim3(a.nsub), dim3(threads), smem, a.stream, a.subs, fac, a.in.r, a.in.q,
                         a.in.sc, a.rowscale, zf, psi, rc, a.ld, a.ncols, a.cmax, depth, a.st);
}

template <int NT, int MM, int S>
static cudaError_t local_f64(const LocalSolveArgs& a, const double* fac, const double* psi, double* zf, double* rc) {
    return a.ncols < a.ld ? local_f64_pad<NT, MM, S, true>(a, fac, psi, zf, rc)
                          : local_f64_pad<NT, MM, S, false>(a, fac, psi, zf, rc);
}

template <int NR, int MM>
static cudaError_t local_f64_rows(const LocalSolveArgs& a, const double* fac, const double* psi, double* zf, double* rc) {
    int depth = a.depth > 0 ? a.depth : 4;
    while (depth > 1 && local_solve_smem(a.cmax, a.ld, 8, depth) > (a.depth > 0 ? 200 : 100) * 1024) --depth;
    const size_t smem = local_solve_smem(a.cmax, a.ld, 8, depth);
    auto kern = k_local_f64_rows<NR, MM>;
    static size_t smem_set = 0;           // per template instance
    if (smem > smem_set) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        smem_set = smem;
    }
    return launch_kernel(a.pdl, kern, dim3(a.nsub), dim3(a.ld / NR * 32), smem, a.stream, a.subs, fac, a.in.r, a.in.q,
                         a.in.sc, a.rowscale, zf, psi, rc, a.ld, a.cmax, depth, a.st);
}

// A lane per row where the FP64 pipe is full: one tile a block row and enough
// subdomains.  Lane per row / row pairs, us a launch at 1, 2, 3, 4 columns, the
// subdomains an SM in brackets, the better ring depth of each:
//   up to 8 modes
//     256 of 16^2 (1.7)    62 / 62   112 / 79   194 / 102  174 / 95
//     441 of 16^2 (2.9)    65 / 81   106 / 94   178 / 120  199 / 139
//     484 of 32^2 (3.2)   262 / 376  444 / 462  778 / 666  778 / 699
//     529 of 16^2 (3.5)    65 / 96   112 / 122  198 / 172  199 / 176
//     625 of 16^2 (4.1)    69 / 151  118 / 145  194 / 250  194 / 201
//     1024 of 32^2 (6.7)  286 / 711  512 / 860  967 / 1123 967 / 1303
//   more
//     121 of 32^2 (0.8)   274 / 233  429 / 255  427 / 277  427 / 343
//     196 of 32^2 (1.3)   274 / 286  453 / 332  452 / 449  452 / 444
//     361 of 12^2 (2.4)    47 / 61    77 / 75    87 / 146   82 / 92
//     625 of 16^2 (4.1)    75 / 180  112 / 195  223 / 296  238 / 282
// With two tiles a block row the pairs are the faster at any number (1728 of 8^3,
// 11 an SM: 395 / 379, 1230 / 884, 2156 / 1305, 2156 / 1403).
static bool f64_by_rows(const LocalSolveArgs& a) {
    if (a.cmax != 1 || a.ld > 4) return false;
    const bool big = a.mmax > 8;
    const int per_sm = a.ld == 1 ? (big ? 1 : 2) : a.ld == 2 ? 3 : big ? 2 : 4;
    return a.nsub > per_sm * a.sms;
}

// Ring depths worth trying, and what one takes: the left-looking kernel gains
// from up to six (480^2 in 16^2 blocks, 12 modes x 3: 290 us at three, 233 at five),
// the other one from a few.
int local_solve_max_depth(const LocalSolveArgs& a) { return f64_by_rows(a) ? 6 : 3; }
size_t local_solve_launch_smem(const LocalSolveArgs& a, int depth) {
    return f64_by_rows(a) ? local_solve_smem(a.cmax, a.ld, 8, depth) : local_f64_smem(a.cmax, a.ncols, depth);
}

template <int MM>
static cudaError_t local_f64_mm(const LocalSolveArgs& a, const double* fac, const double* psi, double* zf, double* rc) {
    constexpr int R4 = MM > 8 ? 2 : 4;   // columns a warp (registers)
    if (f64_by_rows(a)) {
        if (a.ld == 1) return local_f64_rows<1, MM>(a, fac, psi, zf, rc);
        if (a.ld == 2) return local_f64_rows<2, MM>(a, fac, psi, zf, rc);
        return local_f64_rows<R4, MM>(a, fac, psi, zf, rc);
    }
    if (a.ncols > 16) return local_f64<2, MM, 1>(a, fac, psi, zf, rc);
    // lanes per task: at least four warps, and no half-empty one where twice the lanes still fit a block
    int s = 1;
    while (16 * a.ncols * s < 128) s *= 2;
    if (16 * a.ncols * s % 32 != 0 && 32 * a.ncols * s <= 256) s *= 2;
    switch (s) {
        case 1: return local_f64<1, MM, 1>(a, fac, psi, zf, rc);
        case 2: return local_f64<1, MM, 2>(a, fac, psi, zf, rc);
        case 4: return local_f64<1, MM, 4>(a, fac, psi, zf, rc);
        default: return local_f64<1, MM, 8>(a, fac, psi, zf, rc);
    }
}

cudaError_t launch_local_solve(const LocalSolveArgs& a, const double* fac, const double* psi, double* zf,
                               double* rc) {
    return a.mmax > 8 ? local_f64_mm<16>(a, fac, psi, zf, rc) : local_f64_mm<8>(a, fac, psi, zf, rc);
}

}  // namespace ams
