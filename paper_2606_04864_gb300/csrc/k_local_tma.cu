// Local solves of the reduced-precision preconditioner (Section 3.2 A_i,
// fine-level term sum_i R_i^T A_i^{-1} R_i r) with the factor tiles fed by
// the Tensor Memory Accelerator.
//
// Storage (FP32, one 32x32 tile = 4 KB, row-major inside a tile), block row
// K: [ M_K | L_{K,K-c+1} | ... | L_{K,K-1} ] with M_K[r][q] = L_{K,K-c}[r][q]
// (q >= r) and (L_KK^{-1})[r][q] (q < r), plus the reciprocal pivots
// 1/L_KK[r][r] in a per-row array.  The tiles are viewed as a 2-D tensor of
// 32-float rows; one TMA box is one tile, written to shared memory with the
// 128-byte swizzle (16-byte chunk j of tile row r lands at chunk
// j ^ (r mod 8)), so a lane that owns tile row r reads its 32 coefficients
// with eight conflict-free 128-bit loads.  Each ring slot has an mbarrier
// that the TMA completes (expect-tx); every wait is bounded and a timeout
// sets AMS_ERR_DEVICE_TIMEOUT.
//
// Forward sweep (lane = row r of block row K):
//   t = r_K - sum_d L_{K,K-c+d} y_{K-c+d} ;  y_K = L_KK^{-1} t
// Backward sweep (lane = column l of block column K):
//   w = y_K - sum_d L_{K+d,K}^T x_{K+d}   ;  x_K = L_KK^{-T} w
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include <cuda.h>
#include <cudaTypedefs.h>

#include "ams_internal.h"
#include "kernels.cuh"
#include "launch.h"
#include "tma.cuh"

namespace ams {

// ---------------------------------------------------------------------------
// One right-hand side: one warp per subdomain, forward tiles only.
//
// With a single vector each step is a chain of two dependent 32x32 products
// (the off-diagonal update, then L_KK^{-1}), so the kernel is bound by the
// latency of that chain and by the bytes of the factor, not by arithmetic.
// This variant trims both:
//   * the backward sweep reads the forward tiles by column (lane l reads
//     column l of a tile: element (r, l) lies in bank ((l/4) ^ (r mod 8))*4
//     + l mod 4 of row r, so the 32 lanes of a load hit 32 distinct banks),
//     so the transposed copy is never read and the block rows that the
//     forward sweep left in the ring are reused without a reload;
//   * y stays in shared memory between the sweeps and x overwrites it in
//     place (step K reads y_K and x_{K+1..K+c} only);
//   * the row of M_K is loaded once for both of its parts; the triangular
//     masks act per 4-column chunk (a 0/1 weight per chunk, plus the one
//     chunk that holds the diagonal), and each 32-term dot is summed as a
//     tree of eight 4-term dots.
// ---------------------------------------------------------------------------
// Packed FP32 pairs (FFMA2, sm_100 and later): a 32-term dot product in
// 16 two-wide fused multiply-adds on four independent accumulators.
__device__ __forceinline__ float2 lo2(const float4& v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4& v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float pdot16(const float2 (&a)[16], const float* v) {
    float2 s0 = make_float2(0.f, 0.f), s1 = s0, s2 = s0, s3 = s0;
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
        const float4 v0 = *reinterpret_cast<const float4*>(v + 4 * j);
        const float4 v1 = *reinterpret_cast<const float4*>(v + 4 * j + 4);
        s0 = __ffma2_rn(a[2 * j], lo2(v0), s0);
        s1 = __ffma2_rn(a[2 * j + 1], hi2(v0), s1);
        s2 = __ffma2_rn(a[2 * j + 2], lo2(v1), s2);
        s3 = __ffma2_rn(a[2 * j + 3], hi2(v1), s3);
    }
    const float2 s = __fadd2_rn(__fadd2_rn(s0, s1), __fadd2_rn(s2, s3));
    return s.x + s.y;
}
// Column `lane` of a swizzled tile as 16 row pairs (2i, 2i+1).
__device__ __forceinline__ void col_pairs(const float* T, const int (&csw)[8], float2 (&c)[16]) {
#pragma unroll
    for (int i = 0; i < 16; ++i)
        c[i] = make_float2(T[(2 * i) * 32 + csw[(2 * i) & 7]], T[(2 * i + 1) * 32 + csw[(2 * i + 1) & 7]]);
}

// Basis row of one subdomain row (m <= MM entries) as raw 16-byte words when
// the row is 16-byte aligned and m == MM, element by element otherwise.
template <typename TP, int MM>
struct BasisRow {
    static constexpr int PER = 16 / (int)sizeof(TP);
    static constexpr int NW = (MM * (int)sizeof(TP) + 15) / 16;
    uint4 w[NW];
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int i = 0; i < NW; ++i) w[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    __device__ __forceinline__ void load(const TP* __restrict__ pr, int m, bool vec) {
        if (MM % PER == 0 && vec) {
#pragma unroll
            for (int i = 0; i < NW; ++i) w[i] = __ldg(reinterpret_cast<const uint4*>(pr) + i);
        } else {
            TP* e = reinterpret_cast<TP*>(w);
#pragma unroll
            for (int k = 0; k < MM; ++k)
                if (k < m) e[k] = pr[k];
        }
    }
    __device__ __forceinline__ float get(int k) const { return to_f(reinterpret_cast<const TP*>(w)[k]); }
    // entries 2i and 2i+1 (a BF16 pair is widened with two integer operations)
    __device__ __forceinline__ float2 get2(int i) const {
        if constexpr (sizeof(TP) == 2) {
            const uint32_t u = reinterpret_cast<const uint32_t*>(w)[i];
            return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
        } else {
            return make_float2(get(2 * i), get(2 * i + 1));
        }
    }
};

// C1: every subdomain has c == 1 (one 32x32 tile per block row).  The
// backward sweep then keeps column `lane` of M_K in registers after step K
// and forms the step K-1 term sum_{r <= lane} M_K[r][lane] x_K[r] at once,
// so every tile column is read from shared memory once.
template <typename TP, int MM, bool C1>
__global__ void __launch_bounds__(32, 8)
k_local_tma1(const __grid_constant__ CUtensorMap tmF, const SubInfo* __restrict__ subs,
             const int64_t* __restrict__ tile_row0, const float* __restrict__ piv,
             const double* __restrict__ rin, const double* __restrict__ qin,
             const CgScalars* __restrict__ csc, float* __restrict__ zf, const TP* __restrict__ psi,
             float* __restrict__ rc, int cmax, int nbmax, int depth, int l2mode, int l2keep, int64_t budget,
             SolveState* st, int32_t* err, int probe) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = smem_align1024(smem_raw);
    const SubInfo S = subs[blockIdx.x];
    if (!AMS_ROW_OK(S.row0, 5) || !AMS_ROW_OK(S.row0 + S.n - 1, 5)) return;
    const int c = C1 ? 1 : S.c;
    const int nb = S.nb, n = S.n, m = S.m;
    const int D = depth;
    const int nbuf = cmax + D + 1;
    // Block rows nb-nbuf .. nb-1 stay in the ring from the forward sweep to
    // the backward one; rows below Rres are loaded twice.
    const int Rres = nb > nbuf ? nb - nbuf : 0;
    float* tiles = (float*)base;                                        // nbuf * cmax * 1024
    uint64_t* bars = (uint64_t*)(tiles + (size_t)nbuf * cmax * 1024);    // ring_bar_slots(nbuf)
    float* yv = (float*)(bars + ring_bar_slots(nbuf));                   // nbmax * 32: y, then x
    float* tmp = yv + (size_t)nbmax * 32;                                // 32
    const int lane = threadIdx.x;
    const int jr = lane >> 2, er = lane & 3;
    const int64_t trow = tile_row0[blockIdx.x];
    const uint32_t tile_bytes = 4096u * (uint32_t)c;
    const int slot_floats = cmax * 1024;
    // parity of each slot's next completion, and the slots with a copy in
    // flight; both change only when a wait succeeds, so the exit drain waits for every copy
    uint32_t phase = 0, pend = 0;
    bool ok = true;

    // per-lane offsets and masks, fixed for the whole kernel
    int rsw[8], csw[8];
    float2 mk[16], mg[16];                           // 1 where index >= lane / index > lane, pairs (2i, 2i+1)
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        rsw[j] = lane * 32 + ((j ^ (lane & 7)) << 2);   // chunk j of tile row `lane`
        csw[j] = ((jr ^ j) << 2) + er;                 // element (r, lane) sits at r*32 + csw[r & 7]
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        mk[i] = make_float2(2 * i >= lane ? 1.f : 0.f, 2 * i + 1 >= lane ? 1.f : 0.f);
        mg[i] = make_float2(2 * i > lane ? 1.f : 0.f, 2 * i + 1 > lane ? 1.f : 0.f);
    }
    const float2 neg1 = make_float2(-1.f, -1.f);

    if (lane == 0) {
        for (int i = 0; i <= nbuf; ++i) mbar_init(smem_u32(bars + i), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    __syncwarp();

    // ring slots are tracked incrementally (no division in the step loop)
    auto wrap_up = [&](int sl) { return sl >= nbuf ? sl - nbuf : sl; };
    auto wrap_dn = [&](int sl) { return sl < 0 ? sl + nbuf : sl; };
    // L2 priorities of the tile copies (l2mode > 0): a copy that reads a
    // block row for the last time (a resident row's forward load, a backward
    // reload, a forward load whose reload is far away) is evict-first; the
    // forward loads of the l2keep rows below Rres, which the backward sweep
    // reloads soonest, keep normal (l2mode 1) or evict-last (2) priority.
    uint64_t pol_dead = 0, pol_keep = 0;
    if (l2mode > 0 && lane == 0) {
        pol_dead = l2_policy_evict_first();
        pol_keep = l2mode == 2 ? l2_policy_evict_last() : l2_policy_evict_normal();
    }
    auto issue = [&](int K, int slot, bool reload) {
        if (lane == 0) {
            const uint32_t bar = smem_u32(bars + slot);
            mbar_expect_tx(bar, tile_bytes);
            const bool keep = !reload && K < Rres && K >= Rres - l2keep;
            const uint64_t pol = keep ? pol_keep : pol_dead;
            for (int d = 0; d < c; ++d) {
                const uint32_t dst = smem_u32(tiles + slot * slot_floats + d * 1024);
                const int32_t y = (int32_t)(trow + ((int64_t)K * c + d) * 32);
                if (l2mode > 0)
                    tma_load_2d_hint(dst, &tmF, 0, y, bar, pol);
                else
                    tma_load_2d(dst, &tmF, 0, y, bar);
            }
        }
        pend |= 1u << slot;
    };
    auto wait_slot = [&](int slot) {
        if (!mbar_wait(smem_u32(bars + slot), (phase >> slot) & 1u, budget)) {
            ok = false;
            return;
        }
        phase ^= 1u << slot;
        pend &= ~(1u << slot);
    };

    static_assert(MM % 2 == 0, "basis rows are accumulated in pairs");
    float2 racc[MM / 2];
#pragma unroll
    for (int k = 0; k < MM / 2; ++k) racc[k] = make_float2(0.f, 0.f);

    // Per-row inputs of block row K+PF are loaded while step K runs.  They
    // stay in the loaded type until the step that uses them: a conversion
    // or a select right after the load would wait for it there.  Basis rows
    // and pivots are setup data; r and q are written by the previous
    // kernels and are read only after pdl_wait().
    constexpr int PF = 4;
    const float* vp = piv + S.row0 + lane;
    const bool vec = (m == MM) && ((reinterpret_cast<uintptr_t>(psi + S.psi_off) & 15) == 0);
    const TP* pp = rc != nullptr ? psi + S.psi_off + (int64_t)lane * m : nullptr;
    double bt[PF], bq[PF];
    BasisRow<TP, MM> bp[PF];
    float bv[PF];
    auto load_static = [&](int K, BasisRow<TP, MM>& pv, float& pvt) {
        const int row = K * 32 + lane;
        pvt = 1.f;
        pv.clear();
        if (K < nb && row < n) {
            pvt = vp[K * 32];
            if (rc != nullptr) pv.load(pp + (int64_t)K * 32 * m, m, vec);
        }
    };
    // first block rows of the factor and their setup inputs, ahead of the wait
    for (int j = 0; j < D && j < nb; ++j) issue(j, j, false);
#pragma unroll
    for (int u = 0; u < PF; ++u) load_static(u, bp[u], bv[u]);
    pdl_wait();
    if (st != nullptr && st->done) {   // converged: leave once the first copies have landed
        drain_copies(bars, nbuf, pend, phase);
        return;
    }
    if (probe) {   // timeout test hook: a bounded wait on a barrier nothing completes
        if (!mbar_wait(smem_u32(bars + nbuf), 0u, budget)) ok = false;
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) {
            timeout_drain(bars, nbuf, pend, phase, err, st, lane == 0);
            return;
        }
    }
    // r' = r - alpha q when this subdomain's system is still iterating
    double alpha = 0.0;
    bool upd = false;
    if (qin != nullptr) {
        const CgScalars cs = csc[S.seg];
        upd = cs.active != 0;
        if (upd) alpha = cs.alpha;
    }
    const double* rp = rin + S.row0 + lane;
    const double* qp = upd ? qin + S.row0 + lane : nullptr;
    auto load_dyn = [&](int K, double& tv, double& qv) {
        const int row = K * 32 + lane;
        tv = 0.0;
        qv = 0.0;
        if (K < nb && row < n) {
            tv = rp[K * 32];
            if (upd) qv = qp[K * 32];
        }
    };
#pragma unroll
    for (int u = 0; u < PF; ++u) load_dyn(u, bt[u], bq[u]);

    int sK = 0;   // slot of block row K
    auto fwd_step = [&](int K, double& tb, double& qb, BasisRow<TP, MM>& pb, float& vb) {
        if (K + D < nb) issue(K + D, wrap_up(sK + D), false);
        // the FP64 pipe is nearly idle in this kernel: the hardware narrowing
        // is one instruction where the integer-pipe one is about a dozen
        float t = __double2float_rn(upd ? fma(-alpha, qb, tb) : tb);
        const float pvt = vb;
        if (rc != nullptr) {
            const float2 t2 = make_float2(t, t);
#pragma unroll
            for (int k = 0; k < MM / 2; ++k) racc[k] = __ffma2_rn(pb.get2(k), t2, racc[k]);
        }
        load_static(K + PF, pb, vb);
        load_dyn(K + PF, tb, qb);
        wait_slot(sK);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) return;
        const float* T = tiles + sK * slot_floats;
        // row `lane` of M_K split exactly into its two triangles: mu (q >= lane,
        // from L_{K,K-c}) and ml (q < lane, from L_KK^{-1})
        float2 mu[16], ml[16];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float4 m4 = *reinterpret_cast<const float4*>(T + rsw[j]);
            mu[2 * j] = __fmul2_rn(lo2(m4), mk[2 * j]);
            mu[2 * j + 1] = __fmul2_rn(hi2(m4), mk[2 * j + 1]);
            ml[2 * j] = __ffma2_rn(mu[2 * j], neg1, lo2(m4));
            ml[2 * j + 1] = __ffma2_rn(mu[2 * j + 1], neg1, hi2(m4));
        }
        // t = r_K - sum_d L_{K,K-c+d} y_{K-c+d}
        if (!C1) {
#pragma unroll 1
            for (int d = 1; d < c; ++d) {
                const int src = K - c + d;
                if (src < 0) continue;
                const float* Td = T + d * 1024;
                float2 dp[16];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float4 m4 = *reinterpret_cast<const float4*>(Td + rsw[j]);
                    dp[2 * j] = lo2(m4);
                    dp[2 * j + 1] = hi2(m4);
                }
                t -= pdot16(dp, yv + src * 32);
            }
        }
        if (K >= c) t -= pdot16(mu, yv + (K - c) * 32);
        tmp[lane] = t;
        __syncwarp();
        // y_K = L_KK^{-1} t: pivot times t plus the strict lower part of M_K
        const float y = fmaf(pvt, t, pdot16(ml, tmp));
        yv[K * 32 + lane] = y;
        sK = wrap_up(sK + 1);
        __syncwarp();
    };

    // ---------------- forward ----------------
#pragma unroll 1
    for (int K0 = 0; K0 < nb && ok; K0 += PF) {
#pragma unroll
        for (int u = 0; u < PF; ++u)
            if (K0 + u < nb && ok) fwd_step(K0 + u, bt[u], bq[u], bp[u], bv[u]);
    }
    pdl_trigger();
    if (rc != nullptr && ok) {
#pragma unroll
        for (int k = 0; k < MM; ++k) {
            float v = (k & 1) ? racc[k / 2].y : racc[k / 2].x;
            for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
            if (lane == 0 && k < m) rc[S.coff + k] = v;
        }
    }

    // ---------------- backward ----------------
    // Block rows Rres .. nb-1 are still in the ring; older ones are
    // reloaded D steps ahead of their use.
    auto load_bwd = [&](int K, float& pvt) {
        const int row = K * 32 + lane;
        pvt = 1.f;
        if (K >= 0 && row < n) pvt = vp[K * 32];
    };
    float ucarry = 0.f;   // C1: sum_{r <= lane} M_{K+1}[r][lane] x_{K+1}[r] for the next step
    sK = (nb - 1) % nbuf;
    auto bwd_step = [&](int K, float& vb) {
        if (K - D >= 0 && K - D < Rres) issue(K - D, wrap_dn(sK - D), true);
        const float pvt = vb;
        load_bwd(K - PF, vb);
        if (K < Rres) wait_slot(sK);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) return;
        float w = yv[K * 32 + lane];
        const float* Tm = tiles + sK * slot_floats;   // M_K
        if (C1) {
            w -= ucarry;
        } else {
            // w = y_K - sum_d L_{K+d,K}^T x_{K+d}
#pragma unroll 1
            for (int d = 1; d < c; ++d) {
                const int src = K + d;
                if (src >= nb) break;
                float2 cp[16];
                col_pairs(tiles + wrap_up(sK + d) * slot_floats + (c - d) * 1024, csw, cp);
                w -= pdot16(cp, yv + src * 32);
            }
            if (K + c < nb) {   // L_{K+c,K}: upper part of M_{K+c}, rows r <= lane of column lane
                const float* Tc = tiles + wrap_up(sK + c) * slot_floats;
                const float* v = yv + (K + c) * 32;
                float2 cp[16], cl[16];
                col_pairs(Tc, csw, cp);
#pragma unroll
                for (int i = 0; i < 16; ++i) cl[i] = __ffma2_rn(__fmul2_rn(cp[i], mg[i]), neg1, cp[i]);
                w -= pdot16(cl, v);
            }
        }
        tmp[lane] = w;
        __syncwarp();
        // x_K = L_KK^{-T} w: rows r > lane of column lane of M_K.  Column
        // `lane` splits exactly into au (rows r > lane, from L_KK^{-1}) and
        // al (rows r <= lane, from L_{K,K-c}).  (Reloading the transposed
        // tile instead, to read the column as a row, measured slower: the
        // reloads of the forward tiles find part of them still in L2, those
        // of a second array find nothing.)
        float2 au[16], al[16];
        col_pairs(Tm, csw, au);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float2 a2 = au[i];
            au[i] = __fmul2_rn(a2, mg[i]);
            al[i] = __ffma2_rn(au[i], neg1, a2);
        }
        const float x = fmaf(pvt, w, pdot16(au, tmp));
        yv[K * 32 + lane] = x;
        const int row = K * 32 + lane;
        if (row < n) zf[S.row0 + row] = x;
        __syncwarp();
        if (C1 && K > 0) {
            // term of step K-1: L_{K,K-1} is the upper part of M_K (rows r <= lane of column lane)
            ucarry = pdot16(al, yv + K * 32);
        }
        sK = wrap_dn(sK - 1);
    };
    if (ok) {
#pragma unroll
        for (int u = 0; u < PF; ++u) load_bwd(nb - 1 - u, bv[u]);
    }
#pragma unroll 1
    for (int K0 = nb - 1; K0 >= 0 && ok; K0 -= PF) {
#pragma unroll
        for (int u = 0; u < PF; ++u)
            if (K0 - u >= 0 && ok) bwd_step(K0 - u, bv[u]);
    }
    if (!ok) timeout_drain(bars, nbuf, pend, phase, err, st, lane == 0);
}

// ---------------------------------------------------------------------------
// Two to four right-hand sides, and one on a subdomain too long for the kernel
// above: W warps of NC columns each, lane = row (forward) or column (backward).
//
// All arithmetic is FP32 multiply-adds, each 32-term dot as four sums of packed
// pairs.  Bound by the chain of dependent steps and the factor's bytes.  What was
// there before: a lane per row with one sum a dot, forward and transposed tiles
// and a ring of c + depth + 1 block rows (A); the MMA kernel with empty columns
// (B), whose tensor cores truncate as they add up.  A / B / this, us a launch and
// the FP32 apply's relative distance from the FP64 one on N(0, 1):
//   1024^2 in 32^2 x 2  128 / 138 / 67    1.2e-7 / 2.7e-6 / 1.1e-7
//   512^2 in 16^2 x 3    46 / 39 / 27     1.4e-7 / 5.8e-7 / 1.1e-7
//   96x80x72 in 8^3 x 3 145 / 111 / 65    2.3e-7 / 6.8e-7 / 0.8e-7
//   24^3 in 8^3 x 4      66 / 49 / 32     2.6e-7 / 5.8e-7 / 0.8e-7
//   72^3 in 9^3 x 2     237 / 109 / 66    2.7e-7 / 1.1e-6 / 0.9e-7
//   64,000 rows x 1    2281 / 2475 / 1337 1.9e-7 / 2.6e-6 / 0.8e-7
// Four columns are one warp's or two warps' (a.nr): 65 / 67 us at 96x80x72, 41 / 33
// at 24^3, 86 / 96 at 1024^2, 167 / 146 at 110^3; the tuner picks.
//
// The warps of a block share the ring of factor tiles only.  The backward sweep
// is right-looking (see k_local_mma.cu): step K adds the transposes of its own
// block row's tiles times x_K to the pending sums of block rows K-1..K-c, so the
// ring is depth + 1 block rows and a subdomain's y may have any length (it waits
// in z_f).  C: tiles per block row, 1 or 2 with the pending sums in registers;
// 0: any c >= 3, pending sums in shared memory.
// ---------------------------------------------------------------------------
// NC consecutive values of a row (8-byte aligned for NC = 1, 16 for more).
template <int NC>
__device__ __forceinline__ void load_cols(const double* p, double (&v)[NC]) {
    if constexpr (NC == 1) {
        v[0] = *p;
    } else {
#pragma unroll
        for (int j = 0; j < NC; j += 2) {
            const double2 d = *reinterpret_cast<const double2*>(p + j);
            v[j] = d.x;
            v[j + 1] = d.y;
        }
    }
}
template <int NC>
__device__ __forceinline__ void load_cols(const float* p, float (&v)[NC]) {
    if constexpr (NC == 4) {
        const float4 d = *reinterpret_cast<const float4*>(p);
        v[0] = d.x, v[1] = d.y, v[2] = d.z, v[3] = d.w;
    } else if constexpr (NC == 2) {
        const float2 d = *reinterpret_cast<const float2*>(p);
        v[0] = d.x, v[1] = d.y;
    } else {
        v[0] = *p;
    }
}
template <int NC>
__device__ __forceinline__ void store_cols(float* p, const float (&v)[NC]) {
    if constexpr (NC == 4) *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else if constexpr (NC == 2) *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
    else *p = v[0];
}
// Row `lane` of a swizzled tile as 16 column pairs.
__device__ __forceinline__ void row_pairs(const float* T, const int (&rsw)[8], float2 (&a)[16]) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float4 m4 = *reinterpret_cast<const float4*>(T + rsw[j]);
        a[2 * j] = lo2(m4);
        a[2 * j + 1] = hi2(m4);
    }
}

template <typename TP, int NC, int W, int MM, int C>
__global__ void __launch_bounds__(32 * W, 8)
k_local_few(const __grid_constant__ CUtensorMap tmF, const SubInfo* __restrict__ subs,
            const int64_t* __restrict__ tile_row0, const float* __restrict__ piv, const double* __restrict__ rin,
            const double* __restrict__ qin, const CgScalars* __restrict__ csc, float* __restrict__ zf,
            const TP* __restrict__ psi, float* __restrict__ rc, int ld, int cmax, int depth, int64_t budget,
            SolveState* st, int32_t* err, int probe, const int32_t* __restrict__ order) {
    pdl_wait();
    if (st != nullptr && st->done) return;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char* base = smem_align1024(smem_raw);
    const int sid = order != nullptr ? order[blockIdx.x] : (int)blockIdx.x;
    const SubInfo S = subs[sid];
    if (!AMS_ROW_OK(S.row0, 5) || !AMS_ROW_OK(S.row0 + S.n - 1, 5)) return;
    const int c = C > 0 ? C : S.c, cs = C > 0 ? C : cmax;
    const int nb = S.nb, n = S.n, m = S.m;
    const int D = depth, nbuf = D + 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, cb = warp * NC;
    constexpr int BF = 32 * NC;                                // floats of a block [column][row]
    float* tiles = (float*)base;                               // nbuf * cs * 1024
    uint64_t* bars = (uint64_t*)(tiles + (size_t)nbuf * cs * 1024);
    // per warp: a block for t and w, a ring of cs blocks for y (block 0 then holds x), and pending blocks when C = 0
    float* tmp = (float*)(bars + ring_bar_slots(nbuf)) + (size_t)warp * BF * (1 + cs + (C > 0 ? 0 : cs));
    float* yr = tmp + BF;
    float* pw = yr + (size_t)cs * BF + lane;
    const int64_t trow = tile_row0[sid];
    const uint32_t row_bytes = 4096u * (uint32_t)c;
    uint32_t phase = 0, pend = 0;    // change only when a wait succeeds: the exit drain finds every copy in flight
    bool ok = true;

    int rsw[8], csw[8];
    float2 mk[16];                   // forward: 1 where column >= lane; backward: 1 where row > lane
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        rsw[j] = lane * 32 + ((j ^ (lane & 7)) << 2);               // chunk j of tile row `lane`
        csw[j] = (((lane >> 2) ^ j) << 2) + (lane & 3);             // element (r, lane) sits at r * 32 + csw[r & 7]
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) mk[i] = make_float2(2 * i >= lane ? 1.f : 0.f, 2 * i + 1 >= lane ? 1.f : 0.f);
    const float2 neg1 = make_float2(-1.f, -1.f);

    if (threadIdx.x == 0) {
        for (int i = 0; i <= nbuf; ++i) mbar_init(smem_u32(bars + i), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    __syncthreads();
    auto issue = [&](int K, int slot) {
        if (threadIdx.x == 0) {
            const uint32_t bar = smem_u32(bars + slot);
            mbar_expect_tx(bar, row_bytes);
            for (int d = 0; d < c; ++d)
                tma_load_2d(smem_u32(tiles + ((size_t)slot * cs + d) * 1024), &tmF, 0,
                            (int32_t)(trow + ((int64_t)K * c + d) * 32), bar);
        }
        pend |= 1u << slot;
    };
    auto wait_slot = [&](int slot) {
        if (!mbar_wait(smem_u32(bars + slot), (phase >> slot) & 1u, budget)) {
            ok = false;
            return;
        }
        phase ^= 1u << slot;
        pend &= ~(1u << slot);
    };

    // r' = r - alpha q for this warp's columns of (system, rhs) pairs still iterating
    double al[NC];
    bool up[NC], any = false;
#pragma unroll
    for (int j = 0; j < NC; ++j) {
        al[j] = 0.0;
        up[j] = false;
        if (qin != nullptr) {
            const CgScalars cj = csc[(int64_t)S.seg * ld + cb + j];
            up[j] = cj.active != 0;
            if (up[j]) al[j] = cj.alpha;
        }
        any = any || up[j];
    }
    float2 racc[NC][MM / 2];
#pragma unroll
    for (int j = 0; j < NC; ++j)
#pragma unroll
        for (int k = 0; k < MM / 2; ++k) racc[j][k] = make_float2(0.f, 0.f);

    // Inputs of a block row are loaded PF steps ahead, alternating registers (one where two warps take 128 registers).
    constexpr int PF = W == 1 ? 2 : 1;
    const int64_t e0 = (S.row0 + lane) * ld + cb;
    const bool vec = m == MM && (reinterpret_cast<uintptr_t>(psi + S.psi_off) & 15) == 0;
    double rn[PF][NC], qn[PF][NC];
    BasisRow<TP, MM> bn[PF];
    float pv[PF], yn[PF][NC];
    auto load_piv = [&](int K, float& p) {
        const int row = K * 32 + lane;
        p = 1.f;
        if (K >= 0 && row < n) p = __ldg(piv + S.row0 + row);
    };
    auto load_in = [&](int K, int u) {
        const int row = K * 32 + lane;
#pragma unroll
        for (int j = 0; j < NC; ++j) rn[u][j] = qn[u][j] = 0.0;
        bn[u].clear();
        load_piv(K < nb ? K : nb - 1, pv[u]);
        if (K < nb && row < n) {
            load_cols<NC>(rin + e0 + (int64_t)K * 32 * ld, rn[u]);
            if (any) load_cols<NC>(qin + e0 + (int64_t)K * 32 * ld, qn[u]);
            if (rc != nullptr) bn[u].load(psi + S.psi_off + (int64_t)row * m, m, vec);
        }
    };
    auto store_z = [&](int K, const float (&v)[NC]) {
        if (K * 32 + lane < n) store_cols<NC>(zf + e0 + (int64_t)K * 32 * ld, v);
    };

    for (int j = 0; j < D && j < nb; ++j) issue(j, j);
    if (probe) {   // timeout test hook: a bounded wait on a barrier nothing completes
        if (!mbar_wait(smem_u32(bars + nbuf), 0u, budget)) ok = false;
        ok = __syncthreads_and(ok);
    }
#pragma unroll
    for (int u = 0; u < PF; ++u) load_in(u, u);
    int sK = 0, sI = D;              // slots of block rows K and K + D
    int yK = 0;                      // K mod c

    // ---------------- forward ----------------
    // t = r'_K - sum_d L_{K,K-c+d} y_{K-c+d}, y_K = L_KK^{-1} t; y_K takes the ring block of y_{K-c}
    auto fwd_step = [&](int K, int u) {
        float t[NC];
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            t[j] = __double2float_rn(up[j] ? fma(-al[j], qn[u][j], rn[u][j]) : rn[u][j]);
            if (rc != nullptr) {
                const float2 t2 = make_float2(t[j], t[j]);
#pragma unroll
                for (int k = 0; k < MM / 2; ++k) racc[j][k] = __ffma2_rn(bn[u].get2(k), t2, racc[j][k]);
            }
        }
        const float p = pv[u];
        load_in(K + PF, u);
        wait_slot(sK);
        const float* T = tiles + (size_t)sK * cs * 1024;
        if (C != 1)
#pragma unroll 1
            for (int d = 1; d < c; ++d) {
                const int src = K - c + d;
                if (src < 0) continue;
                float2 a[16];
                row_pairs(T + d * 1024, rsw, a);
                const float* v = yr + (C == 2 ? yK ^ 1 : src % c) * BF;
#pragma unroll
                for (int j = 0; j < NC; ++j) t[j] -= pdot16(a, v + 32 * j);
            }
        float2 a[16];                // row `lane` of M_K: columns >= lane (L_{K,K-c}), then columns < lane (L_KK^{-1})
        if (K >= c) {
            row_pairs(T, rsw, a);
#pragma unroll
            for (int i = 0; i < 16; ++i) a[i] = __fmul2_rn(a[i], mk[i]);
#pragma unroll
            for (int j = 0; j < NC; ++j) t[j] -= pdot16(a, yr + yK * BF + 32 * j);
        }
#pragma unroll
        for (int j = 0; j < NC; ++j) tmp[32 * j + lane] = t[j];
        ok = __syncthreads_and(ok);  // t is there; every warp is past block row K - 1
        if (!ok) return;
        if (K + D < nb) issue(K + D, sI);
        row_pairs(T, rsw, a);
#pragma unroll
        for (int i = 0; i < 16; ++i) a[i] = __ffma2_rn(__fmul2_rn(a[i], mk[i]), neg1, a[i]);
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            t[j] = fmaf(p, t[j], pdot16(a, tmp + 32 * j));
            yr[yK * BF + 32 * j + lane] = t[j];
        }
        store_z(K, t);
        sK = sK + 1 == nbuf ? 0 : sK + 1;
        sI = sI + 1 == nbuf ? 0 : sI + 1;
        yK = yK + 1 == c ? 0 : yK + 1;
        __syncwarp();                // y_K is there; t is no longer read
    };
#pragma unroll 1
    for (int K = 0; K < nb && ok; K += PF) {
        fwd_step(K, 0);
        if (PF == 2 && K + 1 < nb && ok) fwd_step(K + 1, PF - 1);
    }
    if (rc != nullptr && ok) {
#pragma unroll
        for (int j = 0; j < NC; ++j)
#pragma unroll
            for (int k = 0; k < MM; ++k) {
                float v = (k & 1) ? racc[j][k / 2].y : racc[j][k / 2].x;
                for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
                if (lane == 0 && k < m) rc[(S.coff + k) * ld + cb + j] = v;
            }
    }
    pdl_trigger();

    // ---------------- backward ----------------
    // w = y_K - pending_K, x_K = L_KK^{-T} w, pending_{K-c+d} += L_{K,K-c+d}^T x_K; block rows nb - nbuf .. nb - 1 are
    // still in the ring, y of a step (written by this lane) is loaded PF steps ahead
    const int Rres = nb > nbuf ? nb - nbuf : 0;
    auto load_back = [&](int K, int u) {
#pragma unroll
        for (int j = 0; j < NC; ++j) yn[u][j] = 0.f;
        load_piv(K, pv[u]);
        if (K >= 0 && K * 32 + lane < n) load_cols<NC>(zf + e0 + (int64_t)K * 32 * ld, yn[u]);
    };
#pragma unroll
    for (int i = 0; i < 16; ++i) mk[i] = make_float2(2 * i > lane ? 1.f : 0.f, 2 * i + 1 > lane ? 1.f : 0.f);
    constexpr int NP = C > 0 ? C : 1;
    float pnd[NP][NC];               // C > 0: pending sums of block rows K, K - 1
#pragma unroll
    for (int j = 0; j < NC; ++j) pnd[0][j] = pnd[NP - 1][j] = 0.f;
    if (C == 0)
        for (int i = 0; i < c * NC; ++i) pw[32 * i] = 0.f;
    if (ok) {
#pragma unroll
        for (int u = 0; u < PF; ++u) load_back(nb - 1 - u, u);
    }
    sK = (nb - 1) % nbuf;
    auto bwd_step = [&](int K, int u) {
        float w[NC];
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            float* e = pw + ((size_t)(K % c) * NC + j) * 32;
            w[j] = yn[u][j] - (C > 0 ? pnd[0][j] : *e);
            if (C == 0) *e = 0.f;
            tmp[32 * j + lane] = w[j];
        }
        const float p = pv[u];
        load_back(K - PF, u);
        if (K < Rres) wait_slot(sK);
        ok = __syncthreads_and(ok);  // w is there; every warp is past block row K + 1
        if (!ok) return;
        if (K - D >= 0 && K - D < Rres) issue(K - D, sK + 1 == nbuf ? 0 : sK + 1);   // into its slot
        const float* T = tiles + (size_t)sK * cs * 1024;
        float2 a[16];                // column `lane` of M_K: rows > lane (L_KK^{-1}), then rows <= lane (L_{K,K-c})
        col_pairs(T, csw, a);
#pragma unroll
        for (int i = 0; i < 16; ++i) a[i] = __fmul2_rn(a[i], mk[i]);
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            w[j] = fmaf(p, w[j], pdot16(a, tmp + 32 * j));
            yr[32 * j + lane] = w[j];
        }
        store_z(K, w);
        __syncwarp();                // x_K is there; w is no longer read
        col_pairs(T, csw, a);
#pragma unroll
        for (int i = 0; i < 16; ++i) a[i] = __ffma2_rn(__fmul2_rn(a[i], mk[i]), neg1, a[i]);
        if constexpr (C > 0) {
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                pnd[0][j] = pnd[C - 1][j];
                pnd[C - 1][j] = pdot16(a, yr + 32 * j);
            }
            if (C == 2) {
                col_pairs(T + 1024, csw, a);
#pragma unroll
                for (int j = 0; j < NC; ++j) pnd[0][j] += pdot16(a, yr + 32 * j);
            }
        } else {
#pragma unroll 1
            for (int d = 0; d < c; ++d) {
                const int dst = K - c + d;
                if (d > 0) col_pairs(T + d * 1024, csw, a);
                if (dst < 0) continue;
                float* e = pw + (size_t)(dst % c) * BF;
#pragma unroll
                for (int j = 0; j < NC; ++j) e[32 * j] += pdot16(a, yr + 32 * j);
            }
        }
        sK = sK == 0 ? nbuf - 1 : sK - 1;
    };
#pragma unroll 1
    for (int K = nb - 1; K >= 0 && ok; K -= PF) {
        bwd_step(K, 0);
        if (PF == 2 && K >= 1 && ok) bwd_step(K - 1, PF - 1);
    }
    if (!ok) timeout_drain(bars, nbuf, pend, phase, err, st, threadIdx.x == 0);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
size_t local_tma1_smem(int cmax, int nbmax, int depth) {
    const int nbuf = cmax + depth + 1;
    return 1024 /* alignment slack */ + (size_t)nbuf * cmax * 4096 + (size_t)ring_bar_slots(nbuf) * 8 +
           ((size_t)nbmax * 32 + 32) * sizeof(float);
}

// Depth for the one-right-hand-side kernel: as deep as possible (at most 6)
// while about seven single-warp blocks still fit on an SM.
static int local_tma1_depth(int cmax, int nbmax) {
    int d = 6;
    while (d > 2 && local_tma1_smem(cmax, nbmax, d) > 31 * 1024) --d;
    return d;
}

template <typename TP, int MM, bool C1>
static cudaError_t tma1(const LocalTmaArgs& a, const void* psi, void* zf, void* rc) {
    const int depth = a.depth > 0 ? a.depth : local_tma1_depth(a.cmax, a.nbmax);
    const size_t smem = local_tma1_smem(a.cmax, a.nbmax, depth);
    auto kern = k_local_tma1<TP, MM, C1>;
    static size_t smem_set = 0;
    if (smem > smem_set) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        smem_set = smem;
    }
    return launch_kernel(a.pdl, kern, dim3(a.nsub), dim3(32), smem, a.stream, *a.tmF, a.subs, a.tile_row0,
                         a.piv,
                         a.in.r, a.in.q, a.in.sc, (float*)zf, (const TP*)psi, (float*)rc, a.cmax, a.nbmax, depth,
                         a.l2mode, a.l2keep, a.budget, a.st, a.err, a.probe);
}

// Staging of the few-column kernel: ring, barriers, and per column the blocks of t, y and (from three tiles) pending sums.
static size_t local_few_smem(int cmax, int ld, int depth) {
    const int nbuf = depth + 1;
    return 1024 /* alignment slack */ + (size_t)nbuf * cmax * 4096 + (size_t)ring_bar_slots(nbuf) * 8 +
           (size_t)ld * 128 * (1 + cmax + (cmax > 2 ? cmax : 0));
}

template <typename TP, int NC, int W, int MM, int C>
static cudaError_t few_launch(const LocalTmaArgs& a, const void* psi, void* zf, void* rc, int nsub, int cmax, int nbmax,
                              const int32_t* order) {
    auto kern = k_local_few<TP, NC, W, MM, C>;
    int depth = a.depth > 0 ? a.depth : 4;
    if (a.depth == 0)
        while (depth > 2 && local_few_smem(cmax, a.ld, depth) > 28 * 1024) --depth;
    depth = std::max(1, std::min(depth, nbmax));   // the rest of the ring would stay unused
    const size_t smem = local_few_smem(cmax, a.ld, depth);
    static size_t smem_set = 0;
    if (smem > smem_set) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        smem_set = smem;
    }
    return launch_kernel(a.pdl, kern, dim3(nsub), dim3(32 * W), smem, a.stream, *a.tmF, a.subs, a.tile_row0, a.piv,
                         a.in.r, a.in.q, a.in.sc, (float*)zf, (const TP*)psi, (float*)rc, a.ld, cmax, depth, a.budget, a.st, a.err, a.probe, order);
}
template <typename TP, int NC, int W>
static cudaError_t few_nc(const LocalTmaArgs& a, const void* psi, void* zf, void* rc) {
    return for_band_widths(a, [&](int nsub, int cmax, int nbmax, const int32_t* order) -> cudaError_t {
        auto mm = [&](auto M) -> cudaError_t {
            constexpr int MM = decltype(M)::value;
            if (cmax == 1) return few_launch<TP, NC, W, MM, 1>(a, psi, zf, rc, nsub, cmax, nbmax, order);
            if (cmax == 2) return few_launch<TP, NC, W, MM, 2>(a, psi, zf, rc, nsub, cmax, nbmax, order);
            return few_launch<TP, NC, W, MM, 0>(a, psi, zf, rc, nsub, cmax, nbmax, order);
        };
        return a.mmax > 8 ? mm(std::integral_constant<int, 16>{}) : mm(std::integral_constant<int, 8>{});
    });
}
// Columns a warp: all of them (a.nr = 4, or two columns), or two of four.
template <typename TP>
static cudaError_t few_tp(const LocalTmaArgs& a, const void* psi, void* zf, void* rc) {
    if (a.ld == 1) return few_nc<TP, 1, 1>(a, psi, zf, rc);
    if (a.ld == 2) return few_nc<TP, 2, 1>(a, psi, zf, rc);
    return a.nr == 4 ? few_nc<TP, 4, 1>(a, psi, zf, rc) : few_nc<TP, 2, 2>(a, psi, zf, rc);
}

// The one-right-hand-side kernel keeps y for a whole subdomain in shared
// memory; longer subdomains and two to four right-hand sides use the few-column
// kernel (both sides of that line are measured there), more the MMA kernel.
bool local_one_vector(const LocalTmaArgs& a) {
    return a.ld == 1 && local_tma1_smem(a.cmax, a.nbmax, 2) <= 200 * 1024;
}

size_t local_tma_launch_smem(const LocalTmaArgs& a, int depth) {
    if (local_one_vector(a)) return local_tma1_smem(a.cmax, a.nbmax, depth);
    return a.ld <= 4 ? local_few_smem(a.cmax, a.ld, depth) : local_mma_smem(a.cmax, a.ld, depth);
}

cudaError_t launch_local_tma(const LocalTmaArgs& a, int prec, const void* psi, const void* psif, void* zf, void* rc) {
    if (a.ld > 4) return launch_local_mma(a, prec, psif, zf, rc);
    if (!local_one_vector(a))
        return prec == AMS_PREC_FP32 ? few_tp<float>(a, psi, zf, rc) : few_tp<__nv_bfloat16>(a, psi, zf, rc);
    const bool big = a.mmax > 8, c1 = a.cmax == 1;
    if (prec == AMS_PREC_FP32) {
        if (big) return c1 ? tma1<float, 16, true>(a, psi, zf, rc) : tma1<float, 16, false>(a, psi, zf, rc);
        return c1 ? tma1<float, 8, true>(a, psi, zf, rc) : tma1<float, 8, false>(a, psi, zf, rc);
    }
    if (big)
        return c1 ? tma1<__nv_bfloat16, 16, true>(a, psi, zf, rc) : tma1<__nv_bfloat16, 16, false>(a, psi, zf, rc);
    return c1 ? tma1<__nv_bfloat16, 8, true>(a, psi, zf, rc) : tma1<__nv_bfloat16, 8, false>(a, psi, zf, rc);
}

// 2-D view [rows x 32] FP32 of a tile array; one box = one 32x32 tile,
// 128-byte swizzle in shared memory.
cudaError_t make_tile_map(void* base, int64_t rows, CUtensorMap* out) {
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        cudaDriverEntryPointQueryResult q;
        void* fn = nullptr;
        cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess) return e;
        if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorSymbolNotFound;
        encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
    }
    const cuuint64_t dims[2] = {32, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {32 * sizeof(float)};
    const cuuint32_t box[2] = {32, 32};
    const cuuint32_t estr[2] = {1, 1};
    CUresult r = encode(out, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

AMS_DEBUG_TU_HOOKS(local_tma)

}  // namespace ams
