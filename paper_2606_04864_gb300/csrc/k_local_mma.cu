// Local solves for five and more right-hand sides on the tensor cores (Section 3.2:
// z_f = sum_i R_i^T A_i^{-1} R_i r' with A_i = L_i L_i^T, and the restriction
// r_c = R_0 r' of the coarse correction, Section 3.1, fused in).
//
// With several right-hand sides every step of the block-row triangular solves
// is a dense product of 32x32 factor tiles with 32-row blocks of 8-32
// columns.  The products run as warp-level tensor-core MMAs (m16n8k8, TF32
// operands, FP32 accumulation).  Each FP32 operand is split into a TF32 head
// and a tail and the product is summed as tail*head + head*tail + head*head,
// each good to 2^-21 (mma_tf32.cuh); BF16 basis entries are exact in TF32 and
// are not split.  The sums are the tensor cores' FP32 ones, which truncate: the
// FP32 apply is 3.5e-7 (48^3 in 4^3 blocks x 32) to 3.7e-6 (512^2 in 32^2 x 8)
// relative from the FP64 one on N(0, 1), where plain FP32 is near 1e-7.
// Five to seven right-hand sides have a stride of 8 like eight.  Up to four, all
// in FP32 multiply-adds, are k_local_few's (k_local_tma.cu), which is faster
// there and closer to the FP64 apply.
//
// Why warp-level MMAs rather than tcgen05: one subdomain's solve is a
// chain of dependent 32-row steps, and tcgen05.mma needs M >= 64 rows per
// instruction from shared memory; stacking independent subdomains into M
// would need their tiles laid out block-diagonally with zero blocks, four
// times the shared memory of the tiles themselves (FP32, twice that with
// the head/tail split), which leaves no room for the copy ring.
//
// Layout.  Block row K of a subdomain holds c tiles of 4 KB back to back:
// [ M_K | L_{K,K-c+1} | .. | L_{K,K-1} ], M_K[r][q] = L_{K,K-c}[r][q]
// (q >= r) and (L_KK^{-1})[r][q] (q < r); reciprocal pivots per row.  The
// order inside a tile (mma_tile_off) is that of the MMA fragments: 2x2
// micro-tiles, 16 bytes each, so that a lane's A fragment is one 16-byte
// load, for the tile as well as for its transpose, and the eight lanes of a
// quarter warp hit all 32 banks either way.  For that the MMA's row g / g+8
// stands for tile row 2g / 2g+1 and its k index t / t+4 for tile column
// 2t / 2t+1.  Right-hand-side blocks sit in shared memory as B fragments
// (bswz): head and tail of two consecutive rows of a column in 16
// bytes, split once by the lane that made them.
//
// What bounds it: row-major tiles with scalar, separately addressed fragment
// loads and cvt.rna splits took 12,000 warp instructions a block row at 32
// right-hand sides (both sweeps; issue 57 %, tensor pipe 18 %), this layout
// 8,300 (8 columns a group; the tuned 16 take fewer).  What is left are fixed
// latencies (a third of the stalls), shared memory, the tensor pipe (23 %) and the
// bytes of the factor.
//
// Staging: one bulk copy per block row into a ring of depth + 1 slots with
// bounded mbarrier waits.  The backward sweep is right-looking: x_K updates
// the pending sums of block rows K-1..K-c with the transposes of block row
// K's own tiles, so a slot is free as soon as its row is done (a left-looking
// one keeps c more), and the last depth + 1 rows of the forward sweep are
// still there when the backward sweep starts.  Two warps share 8 NF
// columns, one for rows 0-15 of every block row, one for rows 16-31 (a step's
// chain of dependent instructions halves, and each A fragment is split once
// per column group); column groups share only the tiles.
//
// Measured (us a launch, row-major kernel with one warp per 8 columns before):
// 128^3 x 32 1224 -> 613-667, 96^3 x 16 314 -> 178, 8 uneven systems x 8
// 406 -> 172, 77^3 x 8 (cycle, with its scaling) 222 -> 105, 64^3 x 8 91 -> 57.  One warp per column group with both row
// halves: 742, 191, 192 and (64^3 x 8) 68.
#include <algorithm>
#include <cstdint>

#include <cuda.h>

#include "ams_internal.h"
#include "kernels.cuh"
#include "launch.h"
#include "mma_tf32.cuh"
#include "tma.cuh"

namespace ams {

// B-fragment block of one warp: 16-byte units {head, head, tail, tail} of
// rows 2 rho, 2 rho + 1 of a column.  Unit of (rho, column c) at
// rho * 8 NF + (c & ~7) + ((c & 7) ^ bswz(rho)): readers (rho = 4 ks + t,
// column g) and writers (rho = 8 mf + g, columns 2t, 2t + 1) both cover all
// banks in each quarter warp.
__device__ __forceinline__ int bswz(int rho) { return ((rho & 1) ? 5 : 0) ^ (rho & 2); }

// Which fragments (16 rows x 8 columns of the operand) a triangular mask
// empties.  MODE 0 all, 1 keep q >= r (L_{K,K-c}), 2 keep q < r (strict lower
// part, L_KK^{-1}); TR: the operand is the transposed tile.
template <int MODE, bool TR>
__device__ __forceinline__ constexpr bool frag_is_zero(int mf, int ks) {
    return TR ? (MODE == 1 ? (16 * mf + 15 < 8 * ks) : MODE == 2 ? (16 * mf >= 8 * ks + 7) : false)
              : (MODE == 1 ? (8 * ks + 7 < 16 * mf) : MODE == 2 ? (8 * ks >= 16 * mf + 15) : false);
}
// ... and which ones it cuts (the others are whole): those on the diagonal.
__device__ __forceinline__ constexpr bool frag_is_cut(int mf, int ks) { return (ks >> 1) == mf; }

// Per-lane constants of the fragment accesses.
struct LaneMap {
    int aE, aO;        // A fragment of the tile, ks even / odd (floats; + 512 mf + 32 (ks >> 1))
    int aT;            // A fragment of its transpose (floats; + 256 ks + 32 mf)
    int rd;            // B unit read (units; + 32 NF ks + 8 nf)
    int wr;            // B unit written for column 2t (units; + 64 NF mf + 8 nf); column 2t + 1: ^ 1
    bool eqE, gtE;     // micro-column vs micro-row on the cut fragments, ks even: Q == R, Q > R
    bool eqO, gtO;     // the same, ks odd
};
template <int NF>
__device__ __forceinline__ LaneMap lane_map(int g, int t) {
    LaneMap m;
    const int sg = ((g & 1) << 2) | (g & 2), st = ((t & 1) << 2) | (t & 2);
    m.aE = g * 64 + ((t ^ sg) << 2);
    m.aO = g * 64 + (((4 + t) ^ sg) << 2);
    m.aT = t * 64 + ((g ^ st) << 2);
    m.rd = t * 8 * NF + (g ^ bswz(t));
    m.wr = g * 8 * NF + ((2 * t) ^ bswz(g));
    m.eqE = t == g;
    m.gtE = t > g;
    m.eqO = t + 4 == g;
    m.gtO = t + 4 > g;
    return m;
}

// acc[nf] += A * B for row half MF of a tile operand A (mask MODE, transposed
// when TR) and a B block of 8 NF columns.  For the transpose the roles of the
// micro-tile's row and column swap: its lane reads micro-row 4 ks + t,
// micro-column 8 MF + g, whose comparison is the mirror of the untransposed one.
template <int MODE, bool TR, int NF, int MF>
__device__ __forceinline__ void half_mma(const float* T, const uint4* B, const LaneMap& L, float (&acc)[NF][4]) {
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
        if (frag_is_zero<MODE, TR>(MF, ks)) continue;
        uint4 b[NF];
#pragma unroll
        for (int nf = 0; nf < NF; ++nf) b[nf] = B[L.rd + 32 * NF * ks + 8 * nf];
        const float4 v = *reinterpret_cast<const float4*>(
            TR ? T + L.aT + 256 * ks + 32 * MF : T + ((ks & 1) ? L.aO : L.aE) + 512 * MF + 32 * (ks >> 1));
        // stored order T00, T10, T01, T11
        float a[4] = {v.x, TR ? v.z : v.y, TR ? v.y : v.z, v.w};
        if (MODE != 0 && frag_is_cut(MF, ks)) {
            const bool eq = (ks & 1) ? L.eqO : L.eqE;             // micro-tile on the diagonal
            const bool gt = (ks & 1) ? L.gtO : L.gtE;             // k index beyond the row index
            const bool up = TR ? !(gt || eq) : gt;                // micro-tile strictly above the diagonal (Q > R)
            // T10 lies below the diagonal of a diagonal micro-tile, the other three on or above it
            const bool keep = MODE == 1 ? (up || eq) : !(up || eq);
            const bool keep10 = MODE == 1 ? up : !up;
            a[0] = keep ? a[0] : 0.f;
            a[3] = keep ? a[3] : 0.f;
            a[TR ? 2 : 1] = keep10 ? a[TR ? 2 : 1] : 0.f;
            a[TR ? 1 : 2] = keep ? a[TR ? 1 : 2] : 0.f;
        }
        uint32_t ah[4], al[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) split_tf32(a[i], ah[i], al[i]);
#pragma unroll
        for (int nf = 0; nf < NF; ++nf) mma_tf32(acc[nf], al, b[nf].x, b[nf].y);
#pragma unroll
        for (int nf = 0; nf < NF; ++nf) mma_tf32(acc[nf], ah, b[nf].z, b[nf].w);
#pragma unroll
        for (int nf = 0; nf < NF; ++nf) mma_tf32(acc[nf], ah, b[nf].x, b[nf].y);
    }
}
template <int MODE, bool TR, int NF>
__device__ __forceinline__ void tile_mma(int mf, const float* T, const uint4* B, const LaneMap& L,
                                         float (&acc)[NF][4]) {
    if (mf == 0) half_mma<MODE, TR, NF, 0>(T, B, L, acc);
    else half_mma<MODE, TR, NF, 1>(T, B, L, acc);
}

template <int NF>
__device__ __forceinline__ void zero_acc(float (&acc)[NF][4]) {
#pragma unroll
    for (int nf = 0; nf < NF; ++nf)
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[nf][i] = 0.f;
}
// v += f acc (f = 1 or -1)
template <int NF>
__device__ __forceinline__ void add_block(float (&v)[NF][4], const float (&acc)[NF][4], float f) {
#pragma unroll
    for (int nf = 0; nf < NF; ++nf)
#pragma unroll
        for (int i = 0; i < 4; ++i) v[nf][i] += f * acc[nf][i];
}
// Accumulator element i of column fragment nf: row 16 mf + 2 g + (i >> 1),
// column 8 nf + 2 t + (i & 1); split and stored as B units (wr includes mf).
template <int NF>
__device__ __forceinline__ void put_block(uint4* B, int wr, const float (&v)[NF][4]) {
#pragma unroll
    for (int nf = 0; nf < NF; ++nf)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            uint4 u;
            split_tf32(v[nf][j], u.x, u.z);
            split_tf32(v[nf][2 + j], u.y, u.w);
            B[(wr ^ j) + 8 * nf] = u;
        }
}
// Barrier of the two warps that share a column group (at most four groups).
// The barrier numbers are immediates: with one in a register a block is taken
// to use all sixteen, and only four such blocks fit on an SM.
__device__ __forceinline__ void pair_sync(int group) {
    if (group == 0) asm volatile("bar.sync 1, 64;\n" ::: "memory");
    else if (group == 1) asm volatile("bar.sync 2, 64;\n" ::: "memory");
    else if (group == 2) asm volatile("bar.sync 3, 64;\n" ::: "memory");
    else asm volatile("bar.sync 4, 64;\n" ::: "memory");
}

// A fragments of Psi_K^T for one block row (k_pack_psi): rows 8 ks + 2t,
// 8 ks + 2t + 1 of mode g (and g + 8 when MM = 16), the four ks together.
template <typename TP, int MM>
struct PsiFrag {
    static constexpr int NV = (int)sizeof(TP) * 8 * (MM / 8) / 16;   // 16-byte words a lane
    uint4 w[NV];
    __device__ __forceinline__ void load(const uint4* p, int lane) {
#pragma unroll
        for (int i = 0; i < NV; ++i) w[i] = __ldg(p + i * 32 + lane);
    }
    // mode half hm, k-step 2 mf + k2, row parity kk
    __device__ __forceinline__ float get(int hm, int k2, int kk, int mf) const {
        if constexpr (sizeof(TP) == 2) {
            const uint32_t* p = reinterpret_cast<const uint32_t*>(w) + 4 * hm;
            const uint32_t u = mf ? p[(k2 + 2) & 3] : p[k2];
            return __uint_as_float(kk ? (u & 0xffff0000u) : (u << 16));
        } else {
            const float* p = reinterpret_cast<const float*>(w) + 8 * hm + kk;
            return mf ? p[2 * ((k2 + 2) & 3)] : p[2 * k2];
        }
    }
};

// C: tiles per block row, 1 or 2 with the pending sums of the backward sweep
// in registers; 0: any c >= 3, pending sums in shared memory.  Two column
// fragments stay within 128 registers, two blocks of eight warps an SM (154
// without the bound: 512^2 in 16^2 blocks x 32 97 us, with it 82); one (0: no bound) takes
// what it needs, 80 to 118.
template <typename TP, int NF, int MM, int C>
__global__ void __launch_bounds__(256, NF == 2 ? 2 : 0)
k_local_mma(const float* __restrict__ tiles_g, const SubInfo* __restrict__ subs,
            const int64_t* __restrict__ tile_off, const int64_t* __restrict__ brow0, const float* __restrict__ piv,
            const double* __restrict__ rin, const double* __restrict__ qin, const CgScalars* __restrict__ csc,
            float* __restrict__ zf, const uint4* __restrict__ psif, float* __restrict__ rc, int ld, int cmax,
            int depth, int64_t budget, SolveState* st, int32_t* err, int probe, const int32_t* __restrict__ order) {
    static_assert(MM == 8 || MM == 16, "basis blocks of up to 8 or 16 modes");
    pdl_wait();
    if (st != nullptr && st->done) return;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int sid = order != nullptr ? order[blockIdx.x] : (int)blockIdx.x;
    const SubInfo S = subs[sid];
    if (!AMS_ROW_OK(S.row0, 4) || !AMS_ROW_OK(S.row0 + S.n - 1, 4)) return;
    const int c = C > 0 ? C : S.c;
    const int nb = S.nb, n = S.n, m = S.m;
    const int D = depth, nbuf = D + 1;
    const int slot_floats = (C > 0 ? C : cmax) * 1024;
    constexpr int BU = 128 * NF;                                   // 16-byte units of a B block
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int mf = warp & 1, group = warp >> 1;                    // row half, column group
    float* tiles = (float*)smem_raw;                               // nbuf * slot_floats
    uint64_t* bars = (uint64_t*)(tiles + (size_t)nbuf * slot_floats);
    // per column group: a block for r', t (forward) and w (backward), and a ring of c blocks for y (then x)
    uint4* tmp = (uint4*)(bars + ring_bar_slots(nbuf)) + (size_t)group * ((C > 0 ? C : cmax) + 1) * BU;
    uint4* yblk = tmp + BU;
    const int g = lane >> 2, t = lane & 3;
    const int cb = group * 8 * NF;
    const LaneMap L = lane_map<NF>(g, t);
    const int wr = L.wr + 64 * NF * mf;
    const float* gt = tiles_g + tile_off[sid];
    const uint4* pf = psif + brow0[sid] * (32 * PsiFrag<TP, MM>::NV);
    const uint32_t row_bytes = 4096u * (uint32_t)c;
    uint32_t phase = 0, pend = 0;    // change only when a wait succeeds: the exit drain finds every copy in flight
    bool ok = true;

    if (threadIdx.x == 0) {
        for (int i = 0; i <= nbuf; ++i) mbar_init(smem_u32(bars + i), 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    __syncthreads();
    auto issue = [&](int K, int slot) {
        if (threadIdx.x == 0) {
            const uint32_t bar = smem_u32(bars + slot);
            mbar_expect_tx(bar, row_bytes);
            bulk_load(smem_u32(tiles + (size_t)slot * slot_floats), gt + (int64_t)K * c * 1024, row_bytes, bar);
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
    // r' = r - alpha q for this lane's columns of (system, rhs) pairs still iterating
    double al[NF][2];
    bool up[NF][2];
#pragma unroll
    for (int nf = 0; nf < NF; ++nf) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            al[nf][j] = 0.0;
            up[nf][j] = false;
            if (qin != nullptr) {
                const CgScalars cs = csc[(int64_t)S.seg * ld + cb + 8 * nf + 2 * t + j];
                up[nf][j] = cs.active != 0;
                if (up[nf][j]) al[nf][j] = cs.alpha;
            }
        }
    }
    float racc[NF][4];   // restriction over this warp's rows: rows = modes g, g + 8; columns as the accumulators
#pragma unroll
    for (int nf = 0; nf < NF; ++nf)
#pragma unroll
        for (int i = 0; i < 4; ++i) racc[nf][i] = 0.f;

    // Inputs of the next block row (r and q in FP64, basis fragments, pivots)
    // are loaded while the current one is computed.
    double2 rraw[2][NF], qraw[2][NF];
    float2 pvr;
    PsiFrag<TP, MM> pfr;
    const int64_t e0 = (S.row0 + 16 * mf + 2 * g) * ld + cb + 2 * t;   // this lane's row and column of block row 0
    const int row0 = 16 * mf + 2 * g;
    auto load_piv = [&](int K) {
        const int row = K * 32 + row0;
        pvr = make_float2(1.f, 1.f);
        if (K >= 0 && row < n) pvr.x = __ldg(piv + S.row0 + row);
        if (K >= 0 && row + 1 < n) pvr.y = __ldg(piv + S.row0 + row + 1);
    };
    auto load_inputs = [&](int K) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = K * 32 + h;   // + row0
            const bool valid = K < nb && row + row0 < n;
#pragma unroll
            for (int nf = 0; nf < NF; ++nf) {
                rraw[h][nf] = make_double2(0.0, 0.0);
                qraw[h][nf] = make_double2(0.0, 0.0);
                if (valid) {
                    const int64_t e = e0 + (int64_t)row * ld + 8 * nf;
                    rraw[h][nf] = *reinterpret_cast<const double2*>(rin + e);
                    if (up[nf][0] || up[nf][1]) qraw[h][nf] = *reinterpret_cast<const double2*>(qin + e);
                }
            }
        }
    };
    auto store_z = [&](int K, const float (&v)[NF][4]) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int row = K * 32 + h;
            if (row + row0 < n)
#pragma unroll
                for (int nf = 0; nf < NF; ++nf)
                    *reinterpret_cast<float2*>(zf + e0 + (int64_t)row * ld + 8 * nf) =
                        make_float2(v[nf][2 * h], v[nf][2 * h + 1]);
        }
    };
    // v = pivot * v + acc
    auto scale_add = [&](float (&v)[NF][4], const float (&acc)[NF][4]) {
#pragma unroll
        for (int nf = 0; nf < NF; ++nf)
#pragma unroll
            for (int i = 0; i < 4; ++i) v[nf][i] = fmaf(i < 2 ? pvr.x : pvr.y, v[nf][i], acc[nf][i]);
    };
    auto subtract = [&](float (&v)[NF][4], const float (&acc)[NF][4]) { add_block<NF>(v, acc, -1.f); };

    // ---------------- forward ----------------
    // t = r'_K - sum_d L_{K,K-c+d} y_{K-c+d}, y_K = L_KK^{-1} t; y_K goes to ring block K mod c,
    // where y_{K-c} was read for the last time before the step's first barrier
    for (int j = 0; j < D && j < nb; ++j) issue(j, j);
    if (probe) {   // timeout test hook: a bounded wait on a barrier nothing completes
        if (!mbar_wait(smem_u32(bars + nbuf), 0u, budget)) ok = false;
        ok = __syncthreads_and(ok);
    }
    load_inputs(0);
    if (rc != nullptr) pfr.load(pf, lane);
    load_piv(0);
    int sK = 0, sI = D;                  // slots of block rows K and K + D
    int yK = 0;                          // K mod c
#pragma unroll 1
    for (int K = 0; K < nb && ok; ++K) {
        float rp[NF][4];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int nf = 0; nf < NF; ++nf) {
                const double2 rv = rraw[h][nf], qv = qraw[h][nf];
                rp[nf][2 * h] = f64_to_f32(up[nf][0] ? fma(-al[nf][0], qv.x, rv.x) : rv.x);
                rp[nf][2 * h + 1] = f64_to_f32(up[nf][1] ? fma(-al[nf][1], qv.y, rv.y) : rv.y);
            }
        load_inputs(K + 1);
        if (rc != nullptr) {   // r_c += Psi_K^T r'_K over this warp's 16 rows (k-steps 2 mf, 2 mf + 1)
            put_block<NF>(tmp, wr, rp);
            __syncwarp();
#pragma unroll
            for (int k2 = 0; k2 < 2; ++k2) {
                const float a[4] = {pfr.get(0, k2, 0, mf), MM > 8 ? pfr.get(MM / 8 - 1, k2, 0, mf) : 0.f,
                                    pfr.get(0, k2, 1, mf), MM > 8 ? pfr.get(MM / 8 - 1, k2, 1, mf) : 0.f};
                uint32_t ah[4], alo[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (sizeof(TP) == 2) ah[i] = __float_as_uint(a[i]);   // BF16 entries are exact in TF32
                    else split_tf32(a[i], ah[i], alo[i]);
                }
#pragma unroll
                for (int nf = 0; nf < NF; ++nf) {
                    const uint4 b = tmp[L.rd + 32 * NF * (2 * mf + k2) + 8 * nf];
                    if (sizeof(TP) != 2) mma_tf32(racc[nf], alo, b.x, b.y);
                    mma_tf32(racc[nf], ah, b.z, b.w);
                    mma_tf32(racc[nf], ah, b.x, b.y);
                }
            }
            if (K + 1 < nb) pfr.load(pf + (size_t)(K + 1) * (32 * PsiFrag<TP, MM>::NV), lane);
            __syncwarp();            // r'_K in tmp is no longer read
        }
        wait_slot(sK);
        const float* T = tiles + (size_t)sK * slot_floats;
        float acc[NF][4];
        zero_acc<NF>(acc);
        if constexpr (C == 1) {
            if (K >= 1) tile_mma<1, false, NF>(mf, T, yblk, L, acc);
        } else if constexpr (C == 2) {
            if (K >= 2) {   // separate accumulators: the two tiles' MMA chains interleave
                float acc1[NF][4];
                zero_acc<NF>(acc1);
                tile_mma<1, false, NF>(mf, T, yblk + yK * BU, L, acc);
                tile_mma<0, false, NF>(mf, T + 1024, yblk + (yK ^ 1) * BU, L, acc1);
                add_block<NF>(acc, acc1, 1.f);
            } else if (K == 1) {
                tile_mma<0, false, NF>(mf, T + 1024, yblk, L, acc);
            }
        } else {
            for (int d = 0; d < c; ++d) {
                const int src = K - c + d;
                if (src < 0) continue;
                const uint4* Y = yblk + (size_t)(src % c) * BU;
                if (d == 0) tile_mma<1, false, NF>(mf, T, Y, L, acc);
                else tile_mma<0, false, NF>(mf, T + d * 1024, Y, L, acc);
            }
        }
        subtract(rp, acc);
        put_block<NF>(tmp, wr, rp);
        ok = __syncthreads_and(ok);      // t complete; every warp is past block row K - 1
        if (K + D < nb && ok) issue(K + D, sI);
        zero_acc<NF>(acc);
        tile_mma<2, false, NF>(mf, T, tmp, L, acc);
        scale_add(rp, acc);
        put_block<NF>(yblk + (size_t)yK * BU, wr, rp);
        store_z(K, rp);
        load_piv(K + 1 < nb ? K + 1 : nb - 1);
        sK = sK + 1 == nbuf ? 0 : sK + 1;
        sI = sI + 1 == nbuf ? 0 : sI + 1;
        yK = yK + 1 == c ? 0 : yK + 1;
        pair_sync(group);                // y_K complete; t is no longer read
    }
    if (rc != nullptr && ok) {   // the two halves' sums, in order
        float* h1 = reinterpret_cast<float*>(tmp) + lane;
        if (mf == 1)
#pragma unroll
            for (int nf = 0; nf < NF; ++nf)
#pragma unroll
                for (int i = 0; i < 4; ++i) h1[(nf * 4 + i) * 32] = racc[nf][i];
        pair_sync(group);
        if (mf == 0)
#pragma unroll
            for (int nf = 0; nf < NF; ++nf)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int mode = g + 8 * (i >> 1);
                    if (mode < m)
                        rc[(S.coff + mode) * ld + cb + 8 * nf + 2 * t + (i & 1)] = racc[nf][i] + h1[(nf * 4 + i) * 32];
                }
        pair_sync(group);
    }
    pdl_trigger();

    // ---------------- backward ----------------
    // w = y_K - pending_K, x_K = L_KK^{-T} w, pending_{K-c+d} += L_{K,K-c+d}^T x_K.
    // Rows nb - nbuf .. nb - 1 are still in the ring; y of the next row
    // (written by this lane in the forward sweep) is loaded a step ahead.
    const int Rres = nb > nbuf ? nb - nbuf : 0;
    float2 yraw[2][NF];
    auto load_y = [&](int K) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int nf = 0; nf < NF; ++nf) {
                const int row = K * 32 + h;
                yraw[h][nf] = make_float2(0.f, 0.f);
                if (K >= 0 && row + row0 < n)
                    yraw[h][nf] = *reinterpret_cast<const float2*>(zf + e0 + (int64_t)row * ld + 8 * nf);
            }
    };
    constexpr int NP = C > 0 ? C : 1;
    float pnd[NP][NF][4];                // C > 0: pending sums of block rows K, K - 1
#pragma unroll
    for (int d = 0; d < NP; ++d) zero_acc<NF>(pnd[d]);
    // C == 0: pending sums in ring blocks 1 .., a lane's own values at [warp half][block row mod c][element][lane]
    constexpr int PE = 4 * NF * 32;      // floats of one pending block of a warp
    float* pw = reinterpret_cast<float*>(yblk + BU) + (size_t)mf * c * PE + lane;
    if (C == 0)
        for (int i = 0; i < c * 4 * NF; ++i) pw[i * 32] = 0.f;
    if (ok) {
        load_y(nb - 1);
        load_piv(nb - 1);
    }
    sK = (nb - 1) % nbuf;
#pragma unroll 1
    for (int K = nb - 1; K >= 0 && ok; --K) {
        float w[NF][4];
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int nf = 0; nf < NF; ++nf) {
                w[nf][2 * h] = yraw[h][nf].x;
                w[nf][2 * h + 1] = yraw[h][nf].y;
            }
        load_y(K - 1);
        if (C > 0) {
            subtract(w, pnd[0]);
        } else {
            float* p = pw + (size_t)(K % c) * PE;
#pragma unroll
            for (int nf = 0; nf < NF; ++nf)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float* e = p + (nf * 4 + i) * 32;
                    w[nf][i] -= *e;
                    *e = 0.f;
                }
        }
        put_block<NF>(tmp, wr, w);
        if (K < Rres) wait_slot(sK);
        ok = __syncthreads_and(ok);      // w complete; every warp is past block row K + 1
        if (K - D >= 0 && K - D < Rres && ok) issue(K - D, sK + 1 == nbuf ? 0 : sK + 1);   // into its slot
        const float* T = tiles + (size_t)sK * slot_floats;
        float acc[NF][4];
        zero_acc<NF>(acc);
        tile_mma<2, true, NF>(mf, T, tmp, L, acc);
        scale_add(w, acc);
        put_block<NF>(yblk, wr, w);
        store_z(K, w);
        load_piv(K - 1);
        pair_sync(group);                // x_K complete; w is no longer read
        if constexpr (C == 1) {
            zero_acc<NF>(pnd[0]);
            if (K >= 1) tile_mma<1, true, NF>(mf, T, yblk, L, pnd[0]);
        } else if constexpr (C == 2) {
#pragma unroll
            for (int nf = 0; nf < NF; ++nf)
#pragma unroll
                for (int i = 0; i < 4; ++i) pnd[0][nf][i] = pnd[NP - 1][nf][i];
            zero_acc<NF>(pnd[NP - 1]);
            if (K >= 1) tile_mma<0, true, NF>(mf, T + 1024, yblk, L, pnd[0]);
            if (K >= 2) tile_mma<1, true, NF>(mf, T, yblk, L, pnd[NP - 1]);
        } else {
            for (int d = c - 1; d >= 0; --d) {
                const int dst = K - c + d;
                if (dst < 0) break;
                zero_acc<NF>(acc);
                if (d == 0) tile_mma<1, true, NF>(mf, T, yblk, L, acc);
                else tile_mma<0, true, NF>(mf, T + d * 1024, yblk, L, acc);
                float* p = pw + (size_t)(dst % c) * PE;
#pragma unroll
                for (int nf = 0; nf < NF; ++nf)
#pragma unroll
                    for (int i = 0; i < 4; ++i) p[(nf * 4 + i) * 32] += acc[nf][i];
            }
        }
        sK = sK == 0 ? nbuf - 1 : sK - 1;
    }
    if (!ok) timeout_drain(bars, nbuf, pend, phase, err, st, threadIdx.x == 0);
}

// Basis in A-fragment order: per block row [16-byte word][lane], the words of
// a lane holding for mode g (then g + 8) the rows 8 ks + 2t, 8 ks + 2t + 1 of
// ks = 0..3; zero past the subdomain's rows and modes.
template <typename TP, int MM>
__global__ void k_pack_psi(const SubInfo* __restrict__ subs, const int64_t* __restrict__ brow0,
                           const TP* __restrict__ psi, uint4* __restrict__ out) {
    constexpr int NV = PsiFrag<TP, MM>::NV;
    const SubInfo S = subs[blockIdx.x];
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    for (int K = threadIdx.x >> 5; K < S.nb; K += blockDim.x >> 5) {
        uint4 w[NV];
        TP* e = reinterpret_cast<TP*>(w);
#pragma unroll
        for (int hm = 0; hm < MM / 8; ++hm)
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
#pragma unroll
                for (int kk = 0; kk < 2; ++kk) {
                    const int row = K * 32 + 8 * ks + 2 * t + kk, mode = g + 8 * hm;
                    e[8 * hm + 2 * ks + kk] =
                        row < S.n && mode < S.m ? psi[S.psi_off + (int64_t)row * S.m + mode] : TP(0.f);
                }
#pragma unroll
        for (int i = 0; i < NV; ++i) out[(brow0[blockIdx.x] + K) * (32 * NV) + i * 32 + lane] = w[i];
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static int mma_mm(int mmax) { return mmax > 8 ? 16 : 8; }

size_t local_mma_psi_words(int prec, int mmax) {
    return (size_t)32 * ((prec == AMS_PREC_FP32 ? 4 : 2) * 8 * (mma_mm(mmax) / 8) / 16);
}

void launch_pack_psi(cudaStream_t s, int nsub, const SubInfo* subs, const int64_t* brow0, int prec, int mmax,
                     const void* psi, void* out) {
    uint4* o = (uint4*)out;
    if (prec == AMS_PREC_FP32) {
        if (mmax > 8) k_pack_psi<float, 16><<<nsub, 128, 0, s>>>(subs, brow0, (const float*)psi, o);
        else k_pack_psi<float, 8><<<nsub, 128, 0, s>>>(subs, brow0, (const float*)psi, o);
    } else {
        const __nv_bfloat16* p = (const __nv_bfloat16*)psi;
        if (mmax > 8) k_pack_psi<__nv_bfloat16, 16><<<nsub, 128, 0, s>>>(subs, brow0, p, o);
        else k_pack_psi<__nv_bfloat16, 8><<<nsub, 128, 0, s>>>(subs, brow0, p, o);
    }
}

size_t local_mma_smem(int cmax, int ld, int depth) {
    const int nbuf = depth + 1;
    return (size_t)nbuf * cmax * 4096 + (size_t)ring_bar_slots(nbuf) * 8 + (size_t)(cmax + 1) * ld * 256;
}

// Default ring depth: the deepest (at most 4) whose staging stays within
// 48 KB, so that four or more blocks fit on an SM.
static int local_mma_depth(int cmax, int ld) {
    int d = 4;
    while (d > 1 && local_mma_smem(cmax, ld, d) > 48 * 1024) --d;
    return d;
}

template <typename TP, int NF, int MM, int C>
static cudaError_t mma_launch(const LocalTmaArgs& a, const void* psif, void* zf, void* rc, int nsub, int cmax,
                              int nbmax, const int32_t* order) {
    const int warps = 2 * a.ld / (8 * NF);
    auto kern = k_local_mma<TP, NF, MM, C>;
    static size_t smem_set = 0;
    // no deeper than the group's block rows: the rest of the ring would stay unused
    const int depth = std::max(1, std::min(a.depth > 0 ? a.depth : local_mma_depth(cmax, a.ld), nbmax));
    const size_t smem = local_mma_smem(cmax, a.ld, depth);
    if (smem > smem_set) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        smem_set = smem;
    }
    return launch_kernel(a.pdl, kern, dim3(nsub), dim3(warps * 32), smem, a.stream, a.mma_tiles, a.subs, a.mma_off,
                         a.brow0, a.piv, a.in.r, a.in.q, a.in.sc, (float*)zf, (const uint4*)psif, (float*)rc, a.ld,
                         cmax, depth, a.budget, a.st, a.err, a.probe, order);
}

template <typename TP, int NF, int MM>
static cudaError_t mma_nf(const LocalTmaArgs& a, const void* psif, void* zf, void* rc) {
    return for_band_widths(a, [&](int nsub, int cmax, int nbmax, const int32_t* order) -> cudaError_t {
        if (cmax == 1) return mma_launch<TP, NF, MM, 1>(a, psif, zf, rc, nsub, cmax, nbmax, order);
        if (cmax == 2) return mma_launch<TP, NF, MM, 2>(a, psif, zf, rc, nsub, cmax, nbmax, order);
        return mma_launch<TP, NF, MM, 0>(a, psif, zf, rc, nsub, cmax, nbmax, order);
    });
}

// Right-hand sides per column group: 8 (default), or 16 (a.nr).
template <typename TP>
static cudaError_t mma_tp(const LocalTmaArgs& a, const void* psif, void* zf, void* rc) {
    const bool big = a.mmax > 8;
    if (a.nr == 16 && a.ld >= 16) return big ? mma_nf<TP, 2, 16>(a, psif, zf, rc) : mma_nf<TP, 2, 8>(a, psif, zf, rc);
    return big ? mma_nf<TP, 1, 16>(a, psif, zf, rc) : mma_nf<TP, 1, 8>(a, psif, zf, rc);
}

cudaError_t launch_local_mma(const LocalTmaArgs& a, int prec, const void* psif, void* zf, void* rc) {
    if (prec == AMS_PREC_FP32) return mma_tp<float>(a, psif, zf, rc);
    return mma_tp<__nv_bfloat16>(a, psif, zf, rc);
}

AMS_DEBUG_TU_HOOKS(local_mma)

}  // namespace ams
