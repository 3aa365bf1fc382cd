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
// S fills the last warp and gives a block at least four.
template <int NT, int MM, int S>
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
}

// Shared memory that a setup or a launch shape is checked against: the
// staging of c + depth + 1 block rows (an upper bound of what is used).
size_t local_solve_smem(int cmax, int ld, size_t tf_bytes, int depth) {
    return ((size_t)(cmax + depth + 1) * blockrow_elems(cmax) + (size_t)(cmax + 1) * 32 * ld + 32 * ld) *
           tf_bytes;
}
static size_t local_f64_smem(int cmax, int ncols, int depth) {
    return ((size_t)(depth + 1) * blockrow_elems(cmax) + (size_t)(2 * cmax + 1) * 32 * ncols) * sizeof(double);
}

template <int NT, int MM, int S>
static cudaError_t local_f64(const LocalSolveArgs& a, const double* fac, const double* psi, double* zf, double* rc) {
    // two block rows in flight hide the copies behind the FP64 pipe, and leave room for several blocks
    int depth = a.depth > 0 ? a.depth : 2;
    while (depth > 1 && local_f64_smem(a.cmax, a.ncols, depth) > 200 * 1024) --depth;
    const size_t smem = local_f64_smem(a.cmax, a.ncols, depth);
    auto kern = k_local_f64<NT, MM, S>;
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

template <int MM>
static cudaError_t local_f64_mm(const LocalSolveArgs& a, const double* fac, const double* psi, double* zf, double* rc) {
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
