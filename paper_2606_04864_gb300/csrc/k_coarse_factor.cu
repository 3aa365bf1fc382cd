// Cholesky factor of the coarse matrix A_0 (Section 3.1) and the inverse of
// that factor, L_c^{-1}, whose nested-dissection blocks the coarse solve
// multiplies by.  FP64 throughout, on 64 x 64 tiles of the dense N_c x N_c
// column-major array, skipping every tile that the nested-dissection order
// of the subdomain graph keeps zero.
//
// Structure.  The coarse rows are ordered by a nested-dissection tree of the
// subdomain graph, each tree node a contiguous row range, children before
// parents.  A_0(r, c) != 0 only for neighbouring subdomains, and neighbours
// are never split into different child subtrees, so with node(r) the node
// owning row r:
//     L(r, c) and L^{-1}(r, c) (r >= c) can be non-zero only where node(r)
//     is node(c) or an ancestor of it.
// A product L(r, l) X(l, c) of two such entries is non-zero only where
// node(r) is an ancestor-or-self of node(c) as well, so every entry outside
// the pattern stays an exact zero through the factorisation and the
// inversion.  A tile is kept when any of its entries lies in the pattern;
// an update of a tile outside it is a sum of exact zeros and is skipped.
//
// Factorisation (right-looking, by column tile k):
//     L_kk = chol(A_kk), kept with its inverse L_kk^{-1};
//     L_ik = A_ik L_kk^{-T}                   for kept tiles i > k;
//     A_ij -= L_ik L_jk^T                     for kept tiles i >= j > k.
// Inversion (X = L^{-1}, right-looking over row tile k of X):
//     X_kk = L_kk^{-1};
//     X_ic -= L_ik X_kc                       for kept i > k, c <= k,
// and X_ic = L_ii^{-1} X_ic once the last update of X_ic has landed (the
// step that applies it is known from the pattern, so the same thread block
// finishes the tile).
#include <algorithm>
#include <cstdint>
#include <vector>

#include "ams_internal.h"
#include "launch.h"

namespace ams {

namespace {

constexpr int TB = 64;          // tile edge
constexpr int TN = 16;          // a block of the tile products makes 64 x 16 (or 16 x 64) outputs of a tile
constexpr int TSPLIT = TB / TN; // blocks per tile
constexpr int TKC = 32;         // contraction chunk staged in shared memory
constexpr int TP = TB + 1;      // padded shared-memory row
constexpr int TTHREADS = 256;   // 16 x 16 threads, 4 outputs each

__device__ __forceinline__ int tile_rows(int64_t nc, int t) {
    const int64_t r = nc - (int64_t)t * TB;
    return r < TB ? (int)r : TB;
}

// A 64 x 64 x 64 tile product is 8192 FP64 warp instructions, 70 us of one
// SM's FP64 pipe, and most steps of the factorisation have fewer tiles than
// the GPU has SMs: four blocks share a tile (factor and inverse at N_c = 3072
// 22 -> 13 ms, 8192 62 -> 37, 24,576 401 -> 343) (MR x NC outputs each, 64 x 16 or
// 16 x 64; thread (tx, ty) has rows tx + 16 a, columns ty + 16 b).
// acc += sum_kk Aop(m, kk) Bop(kk, n), kk < kdim, with Aop(m, kk) =
// A[m + kk*lda] (zero for m >= am) and Bop(kk, n) = BT ? B[n + kk*ldb] :
// B[kk + n*ldb] (zero for n >= bn).
template <bool BT, int MR, int NC>
__device__ __forceinline__ void tile_gemm(double (&acc)[MR / 16][NC / 16], const double* __restrict__ A, int64_t lda,
                                          int am, const double* __restrict__ B, int64_t ldb, int bn, int kdim,
                                          double (*As)[TP], double (*Bs)[TP]) {
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    for (int k0 = 0; k0 < kdim; k0 += TKC) {
#pragma unroll
        for (int e = tid; e < TKC * MR; e += TTHREADS) {
            const int m = e % MR, kk = e / MR;
            As[kk][m] = (m < am && k0 + kk < kdim) ? A[m + (int64_t)(k0 + kk) * lda] : 0.0;
        }
#pragma unroll
        for (int e = tid; e < TKC * NC; e += TTHREADS) {
            const int n = BT ? e % NC : e / TKC, kk = BT ? e / NC : e % TKC;
            Bs[kk][n] = (n < bn && k0 + kk < kdim) ? (BT ? B[n + (int64_t)(k0 + kk) * ldb] : B[(k0 + kk) + (int64_t)n * ldb])
                                                   : 0.0;
        }
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < TKC; ++kk) {
            double a[MR / 16], b[NC / 16];
#pragma unroll
            for (int i = 0; i < MR / 16; ++i) a[i] = As[kk][tx + 16 * i];
#pragma unroll
            for (int j = 0; j < NC / 16; ++j) b[j] = Bs[kk][ty + 16 * j];
#pragma unroll
            for (int i = 0; i < MR / 16; ++i)
#pragma unroll
                for (int j = 0; j < NC / 16; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
        __syncthreads();
    }
}

template <int MI, int NJ>
__device__ __forceinline__ void zero_acc(double (&acc)[MI][NJ]) {
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j) acc[i][j] = 0.0;
}

// C[m][n] = acc (SUB = false) or C[m][n] -= acc (SUB = true), m < cm, n < cn.
template <bool SUB, int MI, int NJ>
__device__ __forceinline__ void tile_store(const double (&acc)[MI][NJ], double* __restrict__ C, int64_t ldc, int cm,
                                           int cn) {
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int n = ty + 16 * j;
        if (n >= cn) continue;
#pragma unroll
        for (int i = 0; i < MI; ++i) {
            const int m = tx + 16 * i;
            if (m >= cm) continue;
            double* p = C + m + (int64_t)n * ldc;
            *p = SUB ? *p - acc[i][j] : acc[i][j];
        }
    }
}

// Diagonal tile t: L_tt = chol(A_tt) in place (lower triangle), its inverse
// into invd[t] (64 x 64 column-major; identity on the padding of a ragged
// last tile) and into the diagonal tile of X.  One block, the
// serial part of every step (with a square root and a reciprocal in each of
// the 64 pivots' chain 171 us).  A pivot that is not positive
// records its coarse row in *bad (min over tiles) and is replaced by 1 so
// that the sweep stays finite; the host reports the failure.
__global__ void __launch_bounds__(TTHREADS) k_tile_potrf(double* __restrict__ A, double* __restrict__ X, int64_t nc,
                                                         int t, double* __restrict__ invd,
                                                         unsigned long long* __restrict__ bad) {
    extern __shared__ double sm[];
    double(*S)[TP] = reinterpret_cast<double(*)[TP]>(sm);             // S[r][c]
    double(*Li)[TP] = reinterpret_cast<double(*)[TP]>(sm + TB * TP);  // Li[r][c]
    const int nr = tile_rows(nc, t);
    const int tid = threadIdx.x;
    const int64_t base = (int64_t)t * TB * (nc + 1);
    for (int e = tid; e < TB * TB; e += TTHREADS) {
        const int r = e & 63, c = e >> 6;   // r fastest: coalesced column reads
        double v;
        if (r < nr && c < nr) v = (r >= c) ? A[base + r + (int64_t)c * nc] : 0.0;
        else v = (r == c) ? 1.0 : 0.0;
        S[r][c] = v;
    }
    __shared__ double s_inv[TB];    // reciprocal pivots 1 / d_j, then 1 / sqrt(d_j)
    __shared__ double s_sq[TB];
    // The factor as unscaled columns (S[r][c] -= S[r][j] S[c][j] / d_j), the
    // square roots taken together at the end: a step waits for one reciprocal
    // only, and the thread that makes the next pivot takes it while the
    // others update the rest (the FP64 square root and division are long
    // sequences, at a quarter of the pipe's rate for a single warp).
    auto pivot = [&](int j, double d) {
        if (!(d > 0.0)) {
            atomicMin(bad, (unsigned long long)((int64_t)t * TB + j));
            d = 1.0;
        }
        s_sq[j] = d;
        s_inv[j] = 1.0 / d;
    };
    __syncthreads();
    if (tid == 0) pivot(0, S[0][0]);
    __syncthreads();
    // 4 x 4 register tiles of the lower triangle, one per thread, last rows first
    int br = 15, bc = tid;
    while (br >= 0 && bc > br) bc -= br + 1, --br;
    const bool own = br >= 0;
    double v[4][4];
    if (own)
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) v[a][b] = S[4 * br + a][4 * bc + b];
    for (int j = 0; j < TB - 1; ++j) {
        if (own && 4 * br + 3 > j && 4 * bc + 3 > j) {
            const double inv = s_inv[j];
            double lr[4], lc[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                lr[a] = S[4 * br + a][j] * inv;
                lc[a] = S[4 * bc + a][j];
            }
            if (br == bc && (j + 1) >> 2 == br) {     // the next pivot and its reciprocal first
                const int k = (j + 1) & 3;
                double d = 0.0;
#pragma unroll
                for (int a = 0; a < 4; ++a)
                    if (a == k) d = fma(-lr[a], lc[a], v[a][a]);
                pivot(j + 1, d);
            }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if (4 * bc + b > j && 4 * br + a >= 4 * bc + b) v[a][b] = fma(-lr[a], lc[b], v[a][b]);
            if (bc == (j + 1) >> 2) {                 // column j + 1 is final: show it
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if (b == ((j + 1) & 3))
#pragma unroll
                        for (int a = 0; a < 4; ++a)
                            if (4 * br + a > j) S[4 * br + a][j + 1] = v[a][b];
            }
        }
        __syncthreads();
    }
    if (tid < TB) {
        const double sq = sqrt(s_sq[tid]);
        s_sq[tid] = sq;
        s_inv[tid] = 1.0 / sq;
    }
    __syncthreads();
    for (int e = tid; e < TB * TB; e += TTHREADS) {
        const int r = e >> 6, c = e & 63;
        if (r > c) S[r][c] *= s_inv[c];
        else if (r == c) S[r][c] = s_sq[c];
        Li[r][c] = 0.0;
    }
    __syncthreads();
    // Inverse of the lower-triangular S: the four 16 x 16 diagonal blocks by
    // forward substitution (a thread per column), then twice
    // Li21 = -Li22 (S21 Li11), on blocks of 16 and of 32 (the product in the
    // unused upper triangle of Li).
    if (tid < TB) {
        const int b0 = tid & ~15, c = tid & 15;
        double x[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            double w = 0.0;
#pragma unroll
            for (int l = 0; l < 16; ++l)
                if (l < r) w = fma(S[b0 + r][b0 + l], x[l], w);
            x[r] = r < c ? 0.0 : r == c ? s_inv[b0 + r] : -w * s_inv[b0 + r];
        }
#pragma unroll
        for (int r = 0; r < 16; ++r) Li[b0 + r][b0 + c] = x[r];
    }
    __syncthreads();
#pragma unroll 1
    for (int h = 16; h < TB; h *= 2) {
        const int per = h * h, npair = TB / (2 * h);      // outputs per pair of blocks
        for (int e = tid; e < per * npair; e += TTHREADS) {
            const int b0 = e / per * 2 * h, m = e % per / h, n = e % h;
            double w = 0.0;
            for (int l = n; l < h; ++l) w = fma(S[b0 + h + m][b0 + l], Li[b0 + l][b0 + n], w);
            Li[b0 + m][b0 + h + n] = w;
        }
        __syncthreads();
        for (int e = tid; e < per * npair; e += TTHREADS) {
            const int b0 = e / per * 2 * h, m = e % per / h, n = e % h;
            double w = 0.0;
            for (int l = 0; l <= m; ++l) w = fma(Li[b0 + h + m][b0 + h + l], Li[b0 + l][b0 + h + n], w);
            Li[b0 + h + m][b0 + n] = -w;
        }
        __syncthreads();
    }
    for (int e = tid; e < TB * TB; e += TTHREADS) {
        const int r = e >> 6, c = e & 63;
        if (r < c) Li[r][c] = 0.0;
    }
    __syncthreads();
    double* iv = invd + (int64_t)t * TB * TB;
    for (int e = tid; e < TB * TB; e += TTHREADS) {
        const int r = e & 63, c = e >> 6;
        iv[r + c * TB] = Li[r][c];
        if (r < nr && c < nr) {
            if (r >= c) A[base + r + (int64_t)c * nc] = S[r][c];
            X[base + r + (int64_t)c * nc] = Li[r][c];
        }
    }
}

// Column step k of the factorisation: L_ik = A_ik L_kk^{-T}, four blocks per
// kept row tile i > k (rows[blockIdx.x / 4]), 16 rows each (in place: a row's
// outputs need that row only).
__global__ void __launch_bounds__(TTHREADS) k_tile_trsm(double* __restrict__ A, int64_t nc, int k,
                                                        const int32_t* __restrict__ rows,
                                                        const double* __restrict__ invd) {
    __shared__ double As[TKC][TP], Bs[TKC][TP];
    const int i = rows[blockIdx.x / TSPLIT], m0 = blockIdx.x % TSPLIT * TN;
    const int mi = tile_rows(nc, i) - m0, mk = tile_rows(nc, k);
    if (mi <= 0) return;
    double* Cik = A + (int64_t)i * TB + m0 + (int64_t)k * TB * nc;
    double acc[1][4];
    zero_acc(acc);
    tile_gemm<true, TN, TB>(acc, Cik, nc, mi, invd + (int64_t)k * TB * TB, TB, mk, mk, As, Bs);
    tile_store<false>(acc, Cik, nc, mi, mk);
}

// Column step k of the factorisation: A_ij -= L_ik L_jk^T for the kept
// pairs (pairs[blockIdx.x / 4] = (i, j), i >= j > k), 16 columns per block.
__global__ void __launch_bounds__(TTHREADS) k_tile_update(double* __restrict__ A, int64_t nc, int k,
                                                          const int2* __restrict__ pairs) {
    __shared__ double As[TKC][TP], Bs[TKC][TP];
    const int2 p = pairs[blockIdx.x / TSPLIT];
    const int n0 = blockIdx.x % TSPLIT * TN;
    const int mi = tile_rows(nc, p.x), mj = tile_rows(nc, p.y) - n0, mk = tile_rows(nc, k);
    if (mj <= 0) return;
    const double* Lik = A + (int64_t)p.x * TB + (int64_t)k * TB * nc;
    const double* Ljk = A + (int64_t)p.y * TB + n0 + (int64_t)k * TB * nc;
    double acc[4][1];
    zero_acc(acc);
    tile_gemm<true, TB, TN>(acc, Lik, nc, mi, Ljk, nc, mj, mk, As, Bs);
    tile_store<true>(acc, A + (int64_t)p.x * TB + ((int64_t)p.y * TB + n0) * nc, nc, mi, mj);
}

// Row step k of the inversion: X_ic -= L_ik X_kc for the kept pairs
// (tasks[blockIdx.x / 4] = (i, c | last << 31), i > k >= c), 16 columns per
// block; on the pair's last update, X_ic = L_ii^{-1} X_ic.
__global__ void __launch_bounds__(TTHREADS) k_tile_inv_step(const double* __restrict__ A, double* __restrict__ X,
                                                            int64_t nc, int k, const int2* __restrict__ tasks,
                                                            const double* __restrict__ invd) {
    __shared__ double As[TKC][TP], Bs[TKC][TP];
    const int2 p = tasks[blockIdx.x / TSPLIT];
    const int n0 = blockIdx.x % TSPLIT * TN;
    const int i = p.x, c = p.y & 0x7fffffff;
    const bool last = (p.y >> 31) & 1;
    const int mi = tile_rows(nc, i), mc = tile_rows(nc, c) - n0, mk = tile_rows(nc, k);
    if (mc <= 0) return;
    double* Xic = X + (int64_t)i * TB + ((int64_t)c * TB + n0) * nc;
    double acc[4][1];
    zero_acc(acc);
    tile_gemm<false, TB, TN>(acc, A + (int64_t)i * TB + (int64_t)k * TB * nc, nc, mi,
                             X + (int64_t)k * TB + ((int64_t)c * TB + n0) * nc, nc, mc, mk, As, Bs);
    tile_store<true>(acc, Xic, nc, mi, mc);
    if (!last) return;
    __syncthreads();   // the block's own global writes are visible to it after the barrier
    zero_acc(acc);
    tile_gemm<false, TB, TN>(acc, invd + (int64_t)i * TB * TB, TB, mi, Xic, nc, mc, mi, As, Bs);
    tile_store<false>(acc, Xic, nc, mi, mc);
}

}  // namespace

// ---------------------------------------------------------------------------
// host: the kept tiles and the task lists of every step
// ---------------------------------------------------------------------------
void build_coarse_tile_plan(const std::vector<NDNode>& nodes, int64_t nc, CoarseTilePlan& P) {
    P = CoarseTilePlan{};
    P.nc = nc;
    const int T = (int)((nc + TB - 1) / TB);
    P.T = T;
    if (T == 0) return;
    auto first_tile = [](int64_t row) { return (int)(row / TB); };
    // kept tiles of each column tile K (rows >= K), from the nodes that own
    // K's columns and their ancestors
    std::vector<std::vector<int32_t>> colpat(T), rowpat(T);
    std::vector<int32_t> stamp(T, -1);
    std::vector<uint64_t> kept((size_t)T * ((T + 63) / 64), 0);
    const size_t wpr = (size_t)(T + 63) / 64;
    auto is_kept = [&](int i, int j) { return (kept[(size_t)j * wpr + (i >> 6)] >> (i & 63)) & 1u; };
    size_t q0 = 0;   // first node whose range may reach column tile K
    for (int K = 0; K < T; ++K) {
        const int64_t c0 = (int64_t)K * TB, c1 = std::min<int64_t>(nc, c0 + TB);
        auto& col = colpat[K];
        auto mark = [&](int64_t r0, int64_t r1) {   // rows [r0, r1), r1 > r0
            for (int I = std::max(K, first_tile(r0)); I <= first_tile(r1 - 1); ++I)
                if (stamp[I] != K) {
                    stamp[I] = K;
                    col.push_back(I);
                }
        };
        mark(c0, c0 + 1);   // the diagonal tile
        while (q0 < nodes.size() && nodes[q0].a + nodes[q0].k <= c0) ++q0;
        for (size_t q = q0; q < nodes.size() && nodes[q].a < c1; ++q) {
            if (nodes[q].k == 0) continue;
            mark(std::max<int64_t>(nodes[q].a, c0), nodes[q].a + nodes[q].k);
            for (int32_t p = nodes[q].parent; p >= 0; p = nodes[p].parent)
                if (nodes[p].k > 0) mark(nodes[p].a, nodes[p].a + nodes[p].k);
        }
        std::sort(col.begin(), col.end());
        for (int32_t I : col) {
            kept[(size_t)K * wpr + (I >> 6)] |= uint64_t(1) << (I & 63);
            rowpat[I].push_back(K);   // K ascending: each row list is sorted
        }
        P.kept_tiles += (int64_t)col.size();
    }
    // factorisation steps
    P.trsm_ptr.assign(T + 1, 0);
    P.upd_ptr.assign(T + 1, 0);
    for (int k = 0; k < T; ++k) {
        const auto& col = colpat[k];   // col[0] == k
        for (size_t a = 1; a < col.size(); ++a) P.trsm.push_back(col[a]);
        for (size_t a = 1; a < col.size(); ++a)
            for (size_t b = 1; b <= a; ++b)
                if (is_kept(col[a], col[b])) {
                    P.upd.push_back(col[a]);
                    P.upd.push_back(col[b]);
                }
        P.trsm_ptr[k + 1] = (int64_t)P.trsm.size();
        P.upd_ptr[k + 1] = (int64_t)P.upd.size() / 2;
    }
    // inversion steps; then flag each pair's last update (latest step)
    P.inv_ptr.assign(T + 1, 0);
    for (int k = 0; k < T; ++k) {
        const auto& col = colpat[k];
        for (size_t a = 1; a < col.size(); ++a)
            for (int32_t c : rowpat[k])
                if (is_kept(col[a], c)) {
                    P.inv.push_back(col[a]);
                    P.inv.push_back(c);
                }
        P.inv_ptr[k + 1] = (int64_t)P.inv.size() / 2;
    }
    std::vector<uint64_t> seen(kept.size(), 0);
    for (int64_t t = (int64_t)P.inv.size() / 2 - 1; t >= 0; --t) {
        const int i = P.inv[2 * t], c = P.inv[2 * t + 1];
        uint64_t& w = seen[(size_t)c * wpr + (i >> 6)];
        const uint64_t bit = uint64_t(1) << (i & 63);
        if (!(w & bit)) {
            w |= bit;
            P.inv[2 * t + 1] = (int32_t)((uint32_t)c | 0x80000000u);
        }
    }
    const double tile_fma = (double)TB * TB * TB;
    P.fma = tile_fma * ((double)P.upd.size() / 2 + (double)P.trsm.size() + (double)P.inv.size() / 2);
}

size_t coarse_tile_invd_elems(int T) { return (size_t)T * TB * TB; }

void launch_coarse_tile_factor(cudaStream_t s, const CoarseTilePlan& P, const int32_t* d_trsm, const int2* d_upd,
                               const int2* d_inv, double* d_A, double* d_X, double* d_invd,
                               unsigned long long* d_bad) {
    const int T = P.T;
    if (T == 0) return;
    const size_t psmem = 2 * TB * TP * sizeof(double);
    cudaFuncSetAttribute(k_tile_potrf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psmem);
    k_tile_potrf<<<1, TTHREADS, psmem, s>>>(d_A, d_X, P.nc, 0, d_invd, d_bad);
    for (int k = 0; k < T; ++k) {
        const int64_t nt = P.trsm_ptr[k + 1] - P.trsm_ptr[k];
        if (nt > 0) k_tile_trsm<<<(unsigned)(TSPLIT * nt), TTHREADS, 0, s>>>(d_A, P.nc, k, d_trsm + P.trsm_ptr[k], d_invd);
        const int64_t nu = P.upd_ptr[k + 1] - P.upd_ptr[k];
        if (nu > 0) k_tile_update<<<(unsigned)(TSPLIT * nu), TTHREADS, 0, s>>>(d_A, P.nc, k, d_upd + P.upd_ptr[k]);
        if (k + 1 < T) k_tile_potrf<<<1, TTHREADS, psmem, s>>>(d_A, d_X, P.nc, k + 1, d_invd, d_bad);
    }
    for (int k = 0; k + 1 < T; ++k) {
        const int64_t ni = P.inv_ptr[k + 1] - P.inv_ptr[k];
        if (ni > 0)
            k_tile_inv_step<<<(unsigned)(TSPLIT * ni), TTHREADS, 0, s>>>(d_A, d_X, P.nc, k, d_inv + P.inv_ptr[k], d_invd);
    }
}

}  // namespace ams
