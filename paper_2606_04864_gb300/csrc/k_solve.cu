// Solve-phase kernels of the AMS-preconditioned CG (one GPU, sm_103a).
//
// One CG iteration (Section 3.1 preconditioner inside CG) is five kernels:
//   k_dir_update      p = z + beta p_old
//   k_spmv_dot        q = A p and p.q                          (SELL-32 SpMV)
//   k_local_*         z_f = sum_i R_i^T A_i^{-1} R_i r'  and  r_c = R_0 r',
//                     r' = r - alpha q formed on the fly       (alpha = rho/pq)
//   k_coarse_*        y = L_c^{-1} r_c  (k_coarse.cu)          (A_0 = L_c L_c^T)
//   k_prolong_update  e_c = L_c^{-T} y, z = z_f + R_0^T e_c, r = r',
//                     x += alpha p, r.z, r.r, z.q, convergence test, beta
#include <cstdint>
#include <cstdio>
#include <type_traits>

#include "ams_internal.h"
#include "kernels.cuh"
#include "launch.h"
#include "mma_tf32.cuh"

namespace ams {

// ===========================================================================
// a1: SpMV q = A p and the dot p.q per (system, rhs) (SELL-32: slice s =
// rows 32s..32s+31, entry j of lane l at sell_ptr[s] + 32 j + l; padded
// entries have value 0 and a valid column).  One element (row, rhs) per
// thread per step; the first JU entries of the row are loaded before any
// product, so their loads and then their gathers are in flight together.
// FP64 arithmetic is scarce on this GPU (about 1/64 of the FP32 rate), so
// the direction update p = z + beta p_old runs as its own streaming pass
// (k_dir_update) rather than being recomputed for every gathered entry.
// with_dot = 0: plain product (no dot, no solve state).
// ===========================================================================
template <int LD, int JU>
__global__ void __launch_bounds__(kRedThreads)
k_spmv_dot(const int64_t* __restrict__ sell_ptr, const int32_t* __restrict__ sell_col,
           const double* __restrict__ sell_val, const double* __restrict__ p, double* __restrict__ q,
           RedLayout R, CgScalars* sc, SolveState* st, int with_dot) {
    __shared__ double s_out[kRedMaxNV * kMaxLd];
    __shared__ double s_scr[kRedThreads];
    const int rhs = threadIdx.x % LD;                // kRedThreads is a multiple of LD
    const int64_t lo = R.blk_lo[blockIdx.x], hi = R.blk_lo[blockIdx.x + 1];
    int64_t b0 = 0;
    int w = 0, lane = 0;
    int col[JU];
    double val[JU];
    // matrix entries of one element (setup data: may be read before pdl_wait)
    auto load_row = [&](int64_t e) {
        const int64_t row = e / LD;
        const int64_t sl = row >> 5;
        lane = (int)(row & 31);
        b0 = __ldg(sell_ptr + sl);
        w = (int)((__ldg(sell_ptr + sl + 1) - b0) >> 5);
#pragma unroll
        for (int j = 0; j < JU; ++j) {
            col[j] = 0;
            val[j] = 0.0;
            if (j < w) {
                col[j] = __ldg(sell_col + b0 + 32 * j + lane);
                val[j] = __ldg(sell_val + b0 + 32 * j + lane);
            }
        }
    };
    int64_t e = lo + threadIdx.x;
    if (e < hi) load_row(e);
    pdl_wait();
    if (st != nullptr && st->done) return;
    double dot[1] = {0.0};
    while (e < hi) {
        double xv[JU];
#pragma unroll
        for (int j = 0; j < JU; ++j) {
            xv[j] = 0.0;
            if (j < w && AMS_ROW_OK(col[j], 1)) xv[j] = __ldg(p + (int64_t)col[j] * LD + rhs);
        }
        double acc = 0.0;
#pragma unroll
        for (int j = 0; j < JU; ++j)
            if (j < w) acc = fma(val[j], xv[j], acc);
        for (int j = JU; j < w; ++j) {
            const int64_t o = b0 + 32 * j + lane;
            const int cj = __ldg(sell_col + o);
            if (AMS_ROW_OK(cj, 1)) acc = fma(__ldg(sell_val + o), __ldg(p + (int64_t)cj * LD + rhs), acc);
        }
        q[e] = acc;
        if (with_dot) dot[0] = fma(__ldg(p + e), acc, dot[0]);
        e += kRedThreads;
        if (e < hi) load_row(e);
    }
    pdl_trigger();
    if (!with_dot) return;
    int seg;
    if (!seg_reduce<1>(dot, LD, R, s_out, s_scr, seg)) return;
    if (threadIdx.x < LD) {
        CgScalars& c = sc[seg * LD + threadIdx.x];
        c.pq = s_out[threadIdx.x];
        // the iteration's step length, divided once here: a division in every
        // warp of the local solves cost 800 cycles of this GPU's FP64 pipe a
        // warp (8 uneven systems x 8 right-hand sides: 273 to 262 us a launch)
        if (c.active) c.alpha = c.rho / c.pq;
        if (c.active && !(c.pq > 0.0 && isfinite(c.pq))) {
            st->status = AMS_ERR_BREAKDOWN;
            st->done = 1;
        }
    }
}

// a7: p_new = z + beta p_old per (system, rhs); p_old and p_new are
// different buffers (successive iterations alternate them).  XUPD: this
// launch also applies the previous iteration's x += alpha p_old (from 8
// right-hand sides, where the prolongation leaves it); without it the
// kernel is the bare direction update.
template <int LD, typename ZT, bool XUPD>
__global__ void __launch_bounds__(kRedThreads)
k_dir_update(const ZT* __restrict__ z, const double* __restrict__ p_old, double* __restrict__ p_new,
             double* __restrict__ x, RedLayout R, const CgScalars* sc, SolveState* st) {
    pdl_wait();
    if (st->done) return;
    pdl_trigger();
    const CgScalars& c = sc[R.blk_seg[blockIdx.x] * LD + threadIdx.x % LD];
    const int64_t lo = R.blk_lo[blockIdx.x], hi = R.blk_lo[blockIdx.x + 1];
    if constexpr (!XUPD) {
        const double beta = c.beta;
#pragma unroll 4
        for (int64_t e = lo + threadIdx.x; e < hi; e += kRedThreads) p_new[e] = fma(beta, p_old[e], widen(z[e]));
    } else {
        if (blockIdx.x == 0 && threadIdx.x == 0) st->xdone_it = st->it;
        const double beta = c.beta, alpha = c.alpha;
        const bool xupd = c.xpend != 0;
#pragma unroll 4
        for (int64_t e = lo + threadIdx.x; e < hi; e += kRedThreads) {
            const double po = p_old[e];
            p_new[e] = fma(beta, po, widen(z[e]));
            if (xupd) x[e] = fma(alpha, po, x[e]);   // the previous iteration's x += alpha p
        }
    }
}

// After the loop: the last iteration's x += alpha p, unless a direction
// update ran after it (a breakdown found by the next SpMV ends the loop
// after that update).  Its direction is the one that iteration computed:
// iteration k writes p2 when k is even, p when it is odd.
template <int LD>
__global__ void __launch_bounds__(kRedThreads)
k_x_flush(const double* __restrict__ p, const double* __restrict__ p2, double* __restrict__ x, RedLayout R,
          const CgScalars* sc, const SolveState* st) {
    const int it = st->it;
    if (it == 0 || st->xdone_it == it) return;
    const CgScalars& c = sc[R.blk_seg[blockIdx.x] * LD + threadIdx.x % LD];
    if (!c.xpend) return;
    const double alpha = c.alpha;
    const double* pl = ((it - 1) % 2 == 0) ? p2 : p;
    const int64_t lo = R.blk_lo[blockIdx.x], hi = R.blk_lo[blockIdx.x + 1];
    for (int64_t e = lo + threadIdx.x; e < hi; e += kRedThreads) x[e] = fma(alpha, pl[e], x[e]);
}

// ===========================================================================
// a5 (backward substitution) + a6 + a2: e_c = L_c^{-T} y, z = z_f + R_0^T e_c,
// the CG update and the dots.  A thread block takes a range of consecutive
// subdomains of one system.  Per subdomain: its m_i rows of e_c are the
// product of its rows of the backward block of its nested-dissection node
// (L_c^{-T} restricted to the node's rows and the columns of the node and
// its ancestors) with y gathered at those columns; the block reduces them
// in a fixed order into shared memory, then prolongates over the
// subdomain's contiguous rows (basis rows by 16-byte loads).  With many
// right-hand sides the per-subdomain gathers of y cost more than a separate
// backward launch: then e_c comes in precomputed (ec != NULL).  Padded rows
// belong to no subdomain: their z stays 0 and r, q, x are 0.
//
// mode 0: z only (a plain preconditioner application).
// mode 1: first application of a solve: z and rho = r.z (beta = 0).
// mode 2: CG iteration.  For (system, rhs) pairs still iterating,
//         r <- r - alpha q and (up to four right-hand sides) x <- x + alpha p
//         with alpha = rho / pq (the local solves applied the same fused
//         multiply-add to r on the fly), then r.z, r.r and, for flexible CG,
//         z.q; the last block of a
//         system applies the convergence test and sets beta: rho'/rho (PCG)
//         or -(z.q)/(p.q) (flexible CG).
// ===========================================================================
// Basis row of `m` entries into registers: one 16-byte load per 16 bytes when
// the row is 16-byte aligned and m == MM (vec = 2), pairs of entries when m is
// even and pairs are aligned (vec = 1), else entry by entry.
template <typename TP, int MM>
__device__ __forceinline__ void load_basis_row(const TP* __restrict__ pr, int m, int vec, TP (&v)[MM]) {
    constexpr int PER = 16 / sizeof(TP);
    using P2 = typename std::conditional<sizeof(TP) == 2, uint32_t,
                                         typename std::conditional<sizeof(TP) == 4, uint2, uint4>::type>::type;
    if (vec == 1) {
#pragma unroll
        for (int k = 0; k < MM; k += 2) {
            P2 u{};
            if (k < m) u = __ldg(reinterpret_cast<const P2*>(pr + k));
            const TP* t = reinterpret_cast<const TP*>(&u);
            v[k] = t[0];
            v[k + 1] = t[1];
        }
    } else if (MM % PER == 0 && vec == 2) {
#pragma unroll
        for (int k = 0; k < MM; k += PER) {
            const uint4 u = __ldg(reinterpret_cast<const uint4*>(pr + k));
            const TP* t = reinterpret_cast<const TP*>(&u);
#pragma unroll
            for (int i = 0; i < PER; ++i) v[k + i] = t[i];
        }
    } else {
#pragma unroll
        for (int k = 0; k < MM; ++k) v[k] = (k < m) ? pr[k] : TP(0.f);
    }
}

// Basis row as raw 16-byte words, loaded as load_basis_row does.
template <typename TP, int MM>
struct RowWords {
    static constexpr int NW = (MM * (int)sizeof(TP) + 15) / 16;
    uint4 w[NW];
    __device__ __forceinline__ void load(const TP* __restrict__ pr, int m, int vec) {
        using P2 = typename std::conditional<sizeof(TP) == 2, uint32_t,
                                             typename std::conditional<sizeof(TP) == 4, uint2, uint4>::type>::type;
#pragma unroll
        for (int i = 0; i < NW; ++i) w[i] = make_uint4(0u, 0u, 0u, 0u);
        if (vec == 2) {
#pragma unroll
            for (int i = 0; i < NW; ++i) w[i] = __ldg(reinterpret_cast<const uint4*>(pr) + i);
        } else if (vec == 1) {
#pragma unroll
            for (int k = 0; k < MM / 2; ++k)
                if (2 * k < m) reinterpret_cast<P2*>(w)[k] = __ldg(reinterpret_cast<const P2*>(pr) + k);
        } else {
#pragma unroll
            for (int k = 0; k < MM; ++k)
                if (k < m) reinterpret_cast<TP*>(w)[k] = pr[k];
        }
    }
    __device__ __forceinline__ TP get(int k) const { return reinterpret_cast<const TP*>(w)[k]; }
};

// CH: from 8 right-hand sides (e_c comes from a launch of its own then) a block
// takes its subdomains kChunk at a time: their rows are consecutive, so one
// loop runs over all of them, with e_c and the basis offsets of the chunk in
// shared memory.  One subdomain at a time costs two barriers and a drained
// pipeline for each (8 uneven systems x 8, most of the subdomains 64 rows: 218 us
// a launch; in chunks 178); large subdomains have no use for it, see below.
//
// MODE: 0 and 1 as above, 2 an iteration of PCG, 3 of flexible CG.  Bound by the
// FP64 pipe (two thirds busy at 16 and more right-hand sides: r', three dots)
// and the latency of its streams: the four elements a thread has in flight need
// the loads free of branches (the mode as a run-time argument: 128^3 x 32 785
// us, 96x80x72 x 3 78; this 735 and 72) and 64 registers, four blocks per SM
// (two elements and six blocks 803 and 79, one and eight 834 and 79).
// Blocks per SM that the registers are cut for: three where four spill and that
// costs more than the fourth block gives.  us a launch at four / three: 96^3 with
// 10 modes x 1 86 / 71, x 4 195 / 170, but x 16 212 / 229; 480^2 with 12 modes in
// FP64 x 8 104 / 91; in chunks with an FP32 basis, 48^3 in 4^3 blocks x 32 138 / 122.
template <typename TF, typename TP, int LD, int MM, bool CH>
constexpr int prolong_blocks() {
    if (CH) return MM > 8 || sizeof(TP) == 4 ? 3 : 4;
    return MM > 8 && (sizeof(TF) == 8 || LD <= 4) ? 3 : 4;
}
template <typename TF, typename TP, int LD, int MM, int MODE, bool CH>
__global__ void __launch_bounds__(kRedThreads, prolong_blocks<TF, TP, LD, MM, CH>())
k_prolong_update(const SubInfo* __restrict__ subs, const TP* __restrict__ psi, const TF* __restrict__ ec,
                 const TF* __restrict__ yc, const TF* __restrict__ qmat, const CoarseRef* __restrict__ cref, const int32_t* __restrict__ gat,
                 const TF* __restrict__ zf, double* __restrict__ r, const double* __restrict__ q,
                 double* __restrict__ x, const double* __restrict__ p, TF* __restrict__ z, RedLayout R,
                 CgScalars* sc, SolveState* st, int nseg, const int32_t* __restrict__ sub_of_row) {
    constexpr bool ITER = MODE >= 2, FLEX = MODE == 3, XUPD = ITER && LD < kDeferXMinLd;
    constexpr bool FUSED = LD <= kFusedBackwardMaxLd;   // has the code and the scratch for qmat
    using AT = typename Acc<TF>::type;
    using V4 = typename std::conditional<sizeof(TF) == 4, float4, double4>::type;
    constexpr int NCG = kRedThreads / LD;            // column groups of the backward product
    constexpr int NW = kRedThreads / 32;
    __shared__ double s_out[kRedMaxNV * kMaxLd];
    __shared__ double s_scr[kRedThreads];
    // chunk of subdomains from 8 right-hand sides: as many e_c blocks as fit 16 KB, at most 16
    constexpr int CH0 = 16384 / (MM * LD * (int)sizeof(AT));
    constexpr int kChunk = !CH ? 1 : CH0 > 16 ? 16 : CH0;
    static_assert(kChunk >= 1, "one block of e_c fits");
    __shared__ AT s_ec[kChunk * MM * LD];
    __shared__ AT s_part[FUSED ? NW * MM * LD : 1];
    __shared__ int64_t s_psi[kChunk];                // basis offset of the subdomain's row 0, less row0 * m
    __shared__ int s_mv[kChunk];                     // modes, and how its basis rows load
    pdl_wait();
    if (st != nullptr && st->done) return;
    pdl_trigger();
    const int rhs = threadIdx.x % LD;
    const int cg = threadIdx.x / LD;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double alpha = 0.0;
    bool upd = false;
    if (ITER) {
        const CgScalars c = sc[(int64_t)R.blk_seg[blockIdx.x] * LD + rhs];
        upd = c.active != 0;
        if (upd) alpha = c.alpha;
    }
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    const int64_t s_lo = R.blk_lo[blockIdx.x], s_hi = R.blk_lo[blockIdx.x + 1];
    auto basis_vec = [&](int64_t off, int m) {
        const uintptr_t pa = reinterpret_cast<uintptr_t>(psi + off);
        return m == MM && (pa & 15) == 0 ? 2 : (m & 1) == 0 && (pa & (2 * sizeof(TP) - 1)) == 0 ? 1 : 0;
    };
    // z = z_f + pe, the CG update and the dots of one element
    auto finish = [&](int64_t e, AT zfv, AT pe, double rv, double qv) {
        const AT zs = zfv + pe;              // z in the apply precision, stored so
        const double zv = widen(zs);         // (FP32 widens exactly: the iterates do not change)
        z[e] = zs;
        if (MODE != 0) {
            if (ITER && upd) {
                rv = fma(-alpha, qv, rv);
                r[e] = rv;
                // x += alpha p here, or (from 8 right-hand sides) in the
                // next direction update, marked by xpend
                if (XUPD) x[e] = fma(alpha, p[e], x[e]);
            }
            v[0] = fma(rv, zv, v[0]);
            v[1] = fma(rv, rv, v[1]);
            if (FLEX) v[2] = fma(zv, qv, v[2]);
        }
    };
    if constexpr (CH) {
        using Row = RowWords<TP, MM>;
        constexpr int U = Row::NW * 4 > 16 ? 1 : Row::NW * 4 > 8 ? 2 : 4;   // elements in flight
        const bool coarse = ec != nullptr;
        for (int64_t c0 = s_lo; c0 < s_hi; c0 += kChunk) {
            const int nsub = (int)(s_hi - c0 < kChunk ? s_hi - c0 : kChunk);
            if (threadIdx.x < nsub) {
                const SubInfo S = subs[c0 + threadIdx.x];
                s_psi[threadIdx.x] = S.psi_off - S.row0 * S.m;
                s_mv[threadIdx.x] = S.m * 4 + basis_vec(S.psi_off, S.m);
            }
            if (coarse)
                for (int i = threadIdx.x; i < nsub * MM * LD; i += kRedThreads) {
                    const SubInfo* S = subs + c0 + i / (MM * LD);
                    const int k = i % (MM * LD);
                    s_ec[i] = k < S->m * LD ? (AT)ec[S->coff * LD + k] : AT(0);
                }
            const int64_t e0 = subs[c0].row0 * LD;
            const int64_t e1 = (subs[c0 + nsub - 1].row0 + subs[c0 + nsub - 1].n) * LD;
            __syncthreads();
            for (int64_t eb = e0 + threadIdx.x; eb < e1; eb += U * kRedThreads) {
                AT zv[U];
                double rv[U], qv[U];
                int si[U];
                Row row[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int64_t e = eb + u * kRedThreads;
                    zv[u] = AT(0);
                    rv[u] = qv[u] = 0.0;
                    si[u] = 0;
                    if (e < e1) {
                        if (coarse) si[u] = (int)(__ldg(sub_of_row + e / LD) - c0);
                        zv[u] = (AT)zf[e];
                        if (MODE != 0) rv[u] = r[e];
                        if (ITER) qv[u] = q[e];
                    }
                }
                if (coarse)
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int64_t e = eb + u * kRedThreads;
                        const int mv = s_mv[si[u]], m = mv >> 2;
                        if (e < e1) row[u].load(psi + s_psi[si[u]] + e / LD * m, m, mv & 3);
                    }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int64_t e = eb + u * kRedThreads;
                    if (e >= e1) break;
                    AT pe = AT(0);
                    if (coarse)
#pragma unroll
                        for (int k = 0; k < MM; ++k)
                            pe += (AT)to_d(row[u].get(k)) * s_ec[(si[u] * MM + k) * LD + rhs];
                    finish(e, zv[u], pe, rv[u], qv[u]);
                }
            }
            __syncthreads();                 // the chunk's tables are reused by the next
        }
    } else {
        for (int64_t si = s_lo; si < s_hi; ++si) {
            const SubInfo S = subs[si];
            const int m = S.m;
            const bool coarse = (ec != nullptr || (FUSED && qmat != nullptr)) && m > 0;
            if (coarse && ec != nullptr) {
                // e_c computed by a separate backward-substitution launch
                for (int i = threadIdx.x; i < MM * LD; i += kRedThreads)
                    s_ec[i] = (i < m * LD) ? (AT)ec[(int64_t)S.coff * LD + i] : AT(0);
            } else if (coarse) {
                if constexpr (FUSED) {
                    // e_c rows of this subdomain: acc[k] = sum_j Q[k][j] y[gat[j]] over this thread's columns
                    const CoarseRef cr = cref[si];
                    const TF* Q = qmat + cr.q_off;
                    const int32_t* G = gat + cr.gat_off;
                    AT acc[MM];
#pragma unroll
                    for (int k = 0; k < MM; ++k) acc[k] = AT(0);
                    for (int c4 = cg; 4 * c4 < cr.K; c4 += NCG) {
                        const int j0 = 4 * c4;
                        AT yv[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            yv[e] = AT(0);
                            if (j0 + e < cr.K) {
                                const int gi = __ldg(G + j0 + e);
                                if (AMS_COARSE_OK(gi, 2)) yv[e] = (AT)yc[(int64_t)gi * LD + rhs];
                            }
                        }
#pragma unroll
                        for (int k = 0; k < MM; ++k) {
                            if (k < m) {
                                const V4 qv = *reinterpret_cast<const V4*>(Q + (int64_t)k * cr.ldm + j0);
                                acc[k] += (AT)qv.x * yv[0] + (AT)qv.y * yv[1] + (AT)qv.z * yv[2] + (AT)qv.w * yv[3];
                            }
                        }
                    }
                    // sum over column groups: lanes of a warp with the same rhs, then warps in order
#pragma unroll
                    for (int k = 0; k < MM; ++k) {
                        AT a = acc[k];
                        for (int off = 16; off >= LD; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
                        if (lane < LD) s_part[(warp * MM + k) * LD + lane] = a;
                    }
                    __syncthreads();
                    for (int i = threadIdx.x; i < MM * LD; i += kRedThreads) {
                        AT a = AT(0);
                        for (int w = 0; w < NW; ++w) a += s_part[w * MM * LD + i];
                        s_ec[i] = a;
                    }
                }
            }
            __syncthreads();
            const int vec = basis_vec(S.psi_off, m);
            const int64_t ne = (int64_t)S.n * LD;
            const int64_t g0 = S.row0 * LD;
#pragma unroll 4
            for (int64_t le = threadIdx.x; le < ne; le += kRedThreads) {
                const int64_t e = g0 + le;
                AT acc = (AT)zf[e];
                AT pe = AT(0);
                if (coarse) {
                    TP pv[MM];
                    load_basis_row<TP, MM>(psi + S.psi_off + (le / LD) * m, m, vec, pv);
#pragma unroll
                    for (int k = 0; k < MM; ++k) pe += (AT)to_d(pv[k]) * s_ec[k * LD + rhs];
                }
                finish(e, acc, pe, MODE != 0 ? r[e] : 0.0, ITER ? q[e] : 0.0);
            }
            __syncthreads();                 // s_ec / s_part are reused by the next subdomain
        }
    }
    if (MODE == 0) return;
    int sg;
    if (!seg_reduce<4>(v, LD, R, s_out, s_scr, sg)) return;
    const int it = st->it;
    if (threadIdx.x < LD) {
        CgScalars& c = sc[sg * LD + threadIdx.x];
        const double rz = s_out[threadIdx.x];
        const double rr = s_out[LD + threadIdx.x];
        const double zq = s_out[2 * LD + threadIdx.x];
        if (MODE == 1) {
            c.rho = rz;
            c.beta = 0.0;
            c.zq = 0.0;
            if (c.active && !isfinite(rz)) {
                st->status = AMS_ERR_BREAKDOWN;
                st->done = 1;
            } else if (c.active && rr <= st->rtol2 * c.fnorm2) {   // x_0 already meets the target
                c.active = 0;
                c.rr = rr;
            } else if (c.active && !(rz > 0.0)) {   // r^T M^{-1} r <= 0: the preconditioner is not SPD
                st->status = AMS_ERR_BREAKDOWN;
                st->done = 1;
            }
        } else if (c.active) {
            c.xpend = 1;   // x += alpha p of this iteration: next direction update or the flush
            c.rr = rr;
            c.iters = it + 1;
            if (!isfinite(rr) || !isfinite(rz)) {
                st->status = AMS_ERR_BREAKDOWN;
                st->done = 1;
            } else if (rr <= st->rtol2 * c.fnorm2) {
                c.active = 0;
                c.beta = 0.0;
            } else if (!FLEX && !(rz > 0.0)) {
                // r^T M^{-1} r <= 0 in exact-arithmetic PCG: M is not SPD (the
                // flexible variant, whose M^{-1} is applied in FP32, is only
                // checked on its first residual, in mode 1)
                st->status = AMS_ERR_BREAKDOWN;
                st->done = 1;
            } else {
                c.beta = FLEX ? -zq / c.pq : rz / c.rho;
            }
            c.zq = zq;
            c.rho = rz;
        } else {
            c.xpend = 0;   // inactive this iteration: its update (if any) was applied
        }
    }
    if (!ITER) return;
    if (!last_system(R, nseg)) return;
    if (threadIdx.x == 0) {
        int nact = 0;
        double worst = 0.0;
        for (int i = 0; i < nseg * LD; ++i) {
            nact += sc[i].active;
            if (sc[i].active) worst = fmax(worst, sc[i].rr / sc[i].fnorm2);
        }
        st->nactive = nact;
        st->worst = worst;
        st->it = it + 1;
        if (nact == 0 || it + 1 >= st->maxit) st->done = 1;
    }
}

// End of one body of the device-resident loop: count it and set the while
// node's condition.  The body cap bounds the loop even if no kernel ever
// reported convergence or the iteration cap.
__global__ void k_loop_cond(cudaGraphConditionalHandle h, SolveState* st, int cap) {
    const int b = ++st->bodies;
    cudaGraphSetConditional(h, (!st->done && b < cap) ? 1u : 0u);
}

void launch_loop_cond(cudaStream_t s, cudaGraphConditionalHandle h, SolveState* st, int cap) {
    k_loop_cond<<<1, 1, 0, s>>>(h, st, cap);
}

// ||f||^2 per (system, rhs) and CG scalar initialisation
template <int LD>
__global__ void __launch_bounds__(kRedThreads)
k_init_norms(const double* __restrict__ r, RedLayout R, CgScalars* sc, SolveState* st, int nseg,
             int nrhs) {
    __shared__ double s_out[kRedMaxNV * kMaxLd];
    __shared__ double s_scr[kRedThreads];
    double v[1] = {0.0};
    for (int64_t e = R.blk_lo[blockIdx.x] + threadIdx.x; e < R.blk_lo[blockIdx.x + 1]; e += kRedThreads)
        v[0] = fma(r[e], r[e], v[0]);
    int sg;
    if (!seg_reduce<1>(v, LD, R, s_out, s_scr, sg)) return;
    if (threadIdx.x < LD) {
        CgScalars& c = sc[sg * LD + threadIdx.x];
        c.fnorm2 = s_out[threadIdx.x];
        c.rr = c.fnorm2;
        c.rho = 0.0;
        c.pq = 0.0;
        c.zq = 0.0;
        c.alpha = 0.0;
        c.beta = 0.0;
        c.iters = 0;
        c.xpend = 0;
        c.active = (threadIdx.x < nrhs && c.fnorm2 > 0.0) ? 1 : 0;
    }
    if (!last_system(R, nseg)) return;
    if (threadIdx.x == 0) {
        int nact = 0;
        for (int i = 0; i < nseg * LD; ++i) nact += sc[i].active;
        st->nactive = nact;
        st->it = 0;
        st->xdone_it = 0;
        st->status = 0;
        st->worst = 1.0;
        st->done = (nact == 0);
    }
}

// Caller order (column-major n x nrhs) <-> internal node-major rows, through a
// shared-memory tile of at most 256 rows and 2048 values: both sides move whole
// lines (a column of consecutive dofs, a row's LD values), where a thread per
// dof wrote or read 8 bytes of a different row per lane.  Bound by HBM (apply and
// product at 96^3 x 16, two permutes in and two out: 1.00 -> 0.85 ms).  One column
// has whole lines on both sides as it is and needs no tile: a row's index and
// its value load together, and 256 rows a block fill more SMs than 2048.
__host__ __device__ constexpr int perm_rows(int ld) { return ld < 8 ? 256 : 2048 / ld; }
template <int LD>
__global__ void __launch_bounds__(256)
k_permute_in(const double* __restrict__ f, int64_t n, int nrhs, const int64_t* __restrict__ int_row,
             double* __restrict__ r, double* __restrict__ x) {
    constexpr int ROWS = perm_rows(LD);
    if constexpr (LD == 1) {
        const int64_t i = (int64_t)blockIdx.x * ROWS + threadIdx.x;
        if (i >= n) return;
        const int64_t row = __ldg(int_row + i);
        if (!AMS_ROW_OK(row, 6)) return;
        r[row] = f[i];
        if (x != nullptr) x[row] = 0.0;
        return;
    }
    __shared__ double tile[ROWS * (LD + 1)];
    const int64_t i0 = (int64_t)blockIdx.x * ROWS;
    const int nr = (int)(n - i0 < ROWS ? n - i0 : ROWS);
#pragma unroll 4
    for (int e = threadIdx.x; e < ROWS * LD; e += 256) {
        const int i = e % ROWS, k = e / ROWS;
        tile[i * (LD + 1) + k] = i < nr && k < nrhs ? f[i0 + i + (int64_t)k * n] : 0.0;
    }
    __syncthreads();
#pragma unroll 4
    for (int e = threadIdx.x; e < nr * LD; e += 256) {
        const int i = e / LD, k = e % LD;
        const int64_t row = __ldg(int_row + i0 + i);
        if (!AMS_ROW_OK(row, 6)) continue;
        r[row * LD + k] = tile[i * (LD + 1) + k];
        if (x != nullptr) x[row * LD + k] = 0.0;
    }
}

template <int LD, typename XT>
__global__ void __launch_bounds__(256)
k_permute_out(const XT* __restrict__ x, int64_t n, int nrhs, const int64_t* __restrict__ int_row,
              double* __restrict__ u) {
    constexpr int ROWS = perm_rows(LD);
    if constexpr (LD == 1) {
        const int64_t i = (int64_t)blockIdx.x * ROWS + threadIdx.x;
        if (i >= n) return;
        const int64_t row = __ldg(int_row + i);
        u[i] = AMS_ROW_OK(row, 6) ? widen(x[row]) : 0.0;
        return;
    }
    __shared__ XT tile[ROWS * (LD + 1)];
    const int64_t i0 = (int64_t)blockIdx.x * ROWS;
    const int nr = (int)(n - i0 < ROWS ? n - i0 : ROWS);
#pragma unroll 4
    for (int e = threadIdx.x; e < nr * LD; e += 256) {
        const int i = e / LD, k = e % LD;
        const int64_t row = __ldg(int_row + i0 + i);
        tile[i * (LD + 1) + k] = AMS_ROW_OK(row, 6) ? x[row * LD + k] : XT(0);
    }
    __syncthreads();
#pragma unroll 4
    for (int e = threadIdx.x; e < nrhs * ROWS; e += 256) {
        const int i = e % ROWS, k = e / ROWS;
        if (i < nr) u[i0 + i + (int64_t)k * n] = widen(tile[i * (LD + 1) + k]);
    }
}

// u += u0 (caller order) for the right-hand sides with f != 0 (a warm
// start solves A e = f - A u0 from e = 0; a zero right-hand side keeps u = 0)
__global__ void k_add_initial_guess(double* __restrict__ u, const double* __restrict__ u0, int64_t n, int nrhs,
                                    const CgScalars* __restrict__ sc) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int k = 0; k < nrhs; ++k)
        if (sc[k].fnorm2 > 0.0) u[i + (int64_t)k * n] += u0[i + (int64_t)k * n];
}

void launch_add_initial_guess(cudaStream_t s, double* u, const double* u0, int64_t n, int nrhs,
                              const CgScalars* sc) {
    if (n > 0) k_add_initial_guess<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(u, u0, n, nrhs, sc);
}

// a8: dvals[e] = - sum_k lambda_k[row_e] u_k[col_e]  (caller CSR order)
__global__ void k_sddmm(const int64_t* __restrict__ rowptr, const int32_t* __restrict__ colind,
                        int64_t n, int nrhs, const double* __restrict__ lam,
                        const double* __restrict__ u, double* __restrict__ dvals) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    for (int64_t e = rowptr[i]; e < rowptr[i + 1]; ++e) {
        const int64_t j = colind[e];
        double s = 0.0;
        for (int k = 0; k < nrhs; ++k) s += lam[i + (int64_t)k * n] * u[j + (int64_t)k * n];
        dvals[e] = -s;
    }
}

// sell_val[pos[e]] = vals[e] (caller CSR entry e -> SELL slot)
__global__ void k_scatter_vals(const double* __restrict__ vals, const int64_t* __restrict__ pos, int64_t nnz,
                               double* __restrict__ sell_val) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e < nnz) sell_val[pos[e]] = vals[e];
}

__global__ void k_zero(double* __restrict__ a, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] = 0.0;
}

// ===========================================================================
// host launchers
// ===========================================================================
#define AMS_DISPATCH_LD(ld, F, ...)                     \
    switch (ld) {                                        \
        case 1: F<1>(__VA_ARGS__); break;                \
        case 2: F<2>(__VA_ARGS__); break;                \
        case 4: F<4>(__VA_ARGS__); break;                \
        case 8: F<8>(__VA_ARGS__); break;                \
        case 16: F<16>(__VA_ARGS__); break;              \
        default: F<32>(__VA_ARGS__); break;              \
    }

template <int LD>
static void spmv_ld(const LaunchCtx& L, const double* p, double* q, int with_dot) {
    launch_kernel(L.pdl, k_spmv_dot<LD, 8>, dim3((unsigned)L.nblk), dim3(kRedThreads), 0, L.stream, L.sell_ptr,
                  L.sell_col, L.sell_val, p, q, L.red, L.sc, with_dot ? L.st : nullptr, with_dot);
}
void launch_spmv_dot(const LaunchCtx& L, const double* p, double* q, int with_dot) {
    AMS_DISPATCH_LD(L.ld, spmv_ld, L, p, q, with_dot);
}

template <int LD>
static void dir_ld(const LaunchCtx& L, int prec, const void* z, const double* p_old, double* p_new, double* x) {
    const dim3 g((unsigned)L.nblk), b(kRedThreads);
    const CgScalars* sc = (const CgScalars*)L.sc;
    if (prec == AMS_PREC_FP64) {
        const double* zd = (const double*)z;
        if (x != nullptr)
            launch_kernel(L.pdl, k_dir_update<LD, double, true>, g, b, 0, L.stream, zd, p_old, p_new, x, L.red, sc, L.st);
        else
            launch_kernel(L.pdl, k_dir_update<LD, double, false>, g, b, 0, L.stream, zd, p_old, p_new, x, L.red, sc, L.st);
    } else {
        const float* zf = (const float*)z;
        if (x != nullptr)
            launch_kernel(L.pdl, k_dir_update<LD, float, true>, g, b, 0, L.stream, zf, p_old, p_new, x, L.red, sc, L.st);
        else
            launch_kernel(L.pdl, k_dir_update<LD, float, false>, g, b, 0, L.stream, zf, p_old, p_new, x, L.red, sc, L.st);
    }
}
void launch_dir_update(const LaunchCtx& L, int prec, const void* z, const double* p_old, double* p_new, double* x) {
    AMS_DISPATCH_LD(L.ld, dir_ld, L, prec, z, p_old, p_new, x);
}
template <int LD>
static void flush_ld(const LaunchCtx& L, const double* p, const double* p2, double* x) {
    k_x_flush<LD><<<(unsigned)L.nblk, kRedThreads, 0, L.stream>>>(p, p2, x, L.red, (const CgScalars*)L.sc,
                                                               (const SolveState*)L.st);
}
void launch_x_flush(const LaunchCtx& L, const double* p, const double* p2, double* x) {
    AMS_DISPATCH_LD(L.ld, flush_ld, L, p, p2, x);
}

template <int LD>
static void norms_ld(const LaunchCtx& L, const double* r, int nrhs) {
    k_init_norms<LD><<<L.nblk, kRedThreads, 0, L.stream>>>(r, L.red, L.sc, L.st, L.nseg, nrhs);
}
void launch_init_norms(const LaunchCtx& L, const double* r, int nrhs) {
    AMS_DISPATCH_LD(L.ld, norms_ld, L, r, nrhs);
}

template <typename TF, typename TP, int LD, int MM, bool CH>
static cudaError_t prolong_ch(const LaunchCtx& L, const ProlongArgs& a) {
    auto kern = a.mode == 0   ? k_prolong_update<TF, TP, LD, MM, 0, CH>
                : a.mode == 1 ? k_prolong_update<TF, TP, LD, MM, 1, CH>
                : a.flexible  ? k_prolong_update<TF, TP, LD, MM, 3, CH>
                              : k_prolong_update<TF, TP, LD, MM, 2, CH>;
    return launch_kernel(L.pdl, kern, dim3((unsigned)L.nblk_sub), dim3(kRedThreads), 0, L.stream, L.subs,
                         (const TP*)a.psi, (const TF*)a.ec, (const TF*)a.yc, (const TF*)a.qmat, a.cref, a.gat,
                         (const TF*)a.zf, a.r, a.q, a.x, a.p, (TF*)a.z, L.red_sub, L.sc, L.st, L.nseg, L.sub_of_row);
}
// In chunks up to 2048 elements a subdomain on average, two passes of a block
// over it.  One subdomain at a time / in chunks, us a launch: 1430 elements (the
// uneven systems) 218 / 178, 2048 (512^2 in 16 x 16 blocks x 8) 59 / 57.6; 3650
// (77^3 x 8) 84 / 86, 4096 (64^3 x 8) 53 / 55, 8192 (96^3 x 16) 200 / 204, where
// the row's subdomain is one more load before the basis.  FP64 62 / 65 at 2900.
template <typename TF, typename TP, int LD, int MM>
static cudaError_t prolong_mm(const LaunchCtx& L, const ProlongArgs& a) {
    if constexpr (LD >= 8 && sizeof(TF) == 4) {
        if (L.rows * LD <= 2048 * (int64_t)L.nsub) return prolong_ch<TF, TP, LD, MM, true>(L, a);
    }
    return prolong_ch<TF, TP, LD, MM, false>(L, a);
}
template <typename TF, typename TP, int LD>
static cudaError_t prolong_ld(const LaunchCtx& L, const ProlongArgs& a) {
    if (L.nsub == 0) return cudaSuccess;
    return a.mmax > 8 ? prolong_mm<TF, TP, LD, kMaxM>(L, a) : prolong_mm<TF, TP, LD, 8>(L, a);
}
template <typename TF, typename TP>
static cudaError_t prolong_tp(const LaunchCtx& L, const ProlongArgs& a) {
    switch (L.ld) {
        case 1: return prolong_ld<TF, TP, 1>(L, a);
        case 2: return prolong_ld<TF, TP, 2>(L, a);
        case 4: return prolong_ld<TF, TP, 4>(L, a);
        case 8: return prolong_ld<TF, TP, 8>(L, a);
        case 16: return prolong_ld<TF, TP, 16>(L, a);
        default: return prolong_ld<TF, TP, 32>(L, a);
    }
}
cudaError_t launch_prolong_update(const LaunchCtx& L, int prec, const ProlongArgs& a) {
    if (a.qmat != nullptr && L.ld > kFusedBackwardMaxLd) return cudaErrorInvalidValue;
    if (a.x == nullptr && a.mode == 2 && L.ld < kDeferXMinLd) return cudaErrorInvalidValue;
    if (prec == AMS_PREC_FP64) return prolong_tp<double, double>(L, a);
    if (prec == AMS_PREC_FP32) return prolong_tp<float, float>(L, a);
    return prolong_tp<float, __nv_bfloat16>(L, a);
}

static unsigned perm_blocks(int64_t n, int ld) { return (unsigned)((n + perm_rows(ld) - 1) / perm_rows(ld)); }
template <int LD>
static void perm_in_ld(cudaStream_t s, const double* f, int64_t n, int nrhs, const int64_t* int_row, double* r, double* x) {
    k_permute_in<LD><<<perm_blocks(n, LD), 256, 0, s>>>(f, n, nrhs, int_row, r, x);
}
void launch_permute_in(cudaStream_t s, const double* f, int64_t n, int nrhs, int ld, const int64_t* int_row, double* r,
                       double* x) {
    AMS_DISPATCH_LD(ld, perm_in_ld, s, f, n, nrhs, int_row, r, x);
}
template <int LD>
static void perm_out_ld(cudaStream_t s, const double* x, int64_t n, int nrhs, const int64_t* int_row, double* u) {
    k_permute_out<LD, double><<<perm_blocks(n, LD), 256, 0, s>>>(x, n, nrhs, int_row, u);
}
template <int LD>
static void perm_out32_ld(cudaStream_t s, const float* x, int64_t n, int nrhs, const int64_t* int_row, double* u) {
    k_permute_out<LD, float><<<perm_blocks(n, LD), 256, 0, s>>>(x, n, nrhs, int_row, u);
}
void launch_permute_out(cudaStream_t s, const double* x, int64_t n, int nrhs, int ld, const int64_t* int_row,
                        double* u) {
    AMS_DISPATCH_LD(ld, perm_out_ld, s, x, n, nrhs, int_row, u);
}
void launch_permute_out_f32(cudaStream_t s, const float* x, int64_t n, int nrhs, int ld, const int64_t* int_row,
                            double* u) {
    AMS_DISPATCH_LD(ld, perm_out32_ld, s, x, n, nrhs, int_row, u);
}
void launch_sddmm(cudaStream_t s, const int64_t* rowptr, const int32_t* colind, int64_t n, int nrhs,
                  const double* lam, const double* u, double* dvals) {
    k_sddmm<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(rowptr, colind, n, nrhs, lam, u, dvals);
}
void launch_scatter_vals(cudaStream_t s, const double* vals, const int64_t* pos, int64_t nnz, double* sell_val) {
    if (nnz > 0) k_scatter_vals<<<(unsigned)((nnz + 255) / 256), 256, 0, s>>>(vals, pos, nnz, sell_val);
}
void launch_zero(cudaStream_t s, double* a, int64_t n) {
    if (n > 0) k_zero<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, n);
}

// ---------------------------------------------------------------------------
// checking-build hooks and self-test (see kernels.cuh)
// ---------------------------------------------------------------------------
AMS_DEBUG_TU_HOOKS(solve)

__global__ void k_debug_selftest() { (void)AMS_ROW_OK(-1, 99); }
void launch_debug_selftest(cudaStream_t s) { k_debug_selftest<<<1, 1, 0, s>>>(); }

}  // namespace ams
