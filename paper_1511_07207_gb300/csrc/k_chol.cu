// k_chol.cu -- the paper's Cholesky factorization A = L L^T (FP64) and the
// solve L y = b, L^T x = y.
//
// The paper writes the blocked Cholesky (the direct-methods section, Fig. 3
// and the three block relations after it) as the factorization of a leading
// block, a triangular solve for the block below it and the update of the
// trailing block.  Element by element that is the column-by-column
// factorization: at step k, l_kk = sqrt(w_kk), l_ik = w_ik / l_kk for i > k,
// and w_ij = w_ij - l_ik l_jk for k < j <= i.  b rides along as an extra row
// n of the working matrix W (only its lower triangle is used), so row n
// becomes y = L^-1 b during the factorization: y_k = w_nk / l_kk is the
// forward substitution's division and w_nj -= y_k l_jk its updates, in the
// same order.
//
// Per panel of CH_NB = 32 columns:
// chol_panel_kernel: the panel's columns.  Every CTA factors the panel's
//   diagonal block and some rows below it (row n included) in shared memory:
//   l_kk = sqrt(w_kk), l_ik = w_ik / l_kk (IEEE division), and w_ij = w_ij -
//   l_ik l_jk as a separate multiply and subtract.
// chol_trail_kernel: the trailing lower triangle (rows k1 .. n, columns
//   k1 .. min(i, n - 1)) in 32 x 32 tiles: each element takes the panel's 32
//   updates in order from the panel's l's staged in shared memory, the product on
//   the integer pipes and the difference on the FP64 pipe (ls_rank.cuh).
// chol_backsolve_kernel (cooperative): L^T x = y by blocks of 64 rows from
//   the bottom: CTA 0 solves the diagonal block (one warp), then every CTA
//   subtracts the block's contribution l_ji x_j from the rows above it (32
//   rows a CTA, reading the block's rows of L, which are contiguous).
// So L and y are bit for bit those of the plain column factorization and
// forward substitution; x differs from a scalar back substitution by the
// order of its sums.
//
// Work: n^3 / 6 updates, a rounded product and a rounded difference each (half of the LU's).
#include <cuda_runtime.h>

#include "ls_device.cuh"
#include "ls_internal.h"
#include "ls_rank.cuh"

namespace lsi {

namespace {
constexpr int CT = 512;            // threads per CTA of the cooperative kernels (16 warps)
constexpr int CW = CT / 32;
constexpr int CH_NB = 32;          // panel width
constexpr int CP_T = 256;           // threads of a panel CTA
constexpr int CB = BACK_B;         // rows per back-substitution block
static_assert(CH_NB == RANK_NB, "panel width");
}  // namespace

// One panel, k0 .. k1 - 1.  Row i needs the panel's diagonal block and itself only, so
// every CTA factors the 32 x 32 block for itself (the same operations, the
// same bits) beside `rows` rows of its own below it, in shared memory: no CTA waits for
// another.  Per step: a thread a row, l_kk and l_rk; then the updates, a thread
// an element.  What bounds it is that chain of FP64 square root, division and
// update, 1.5 us a step (49 us a panel); a barrier of the grid a step took
// 228 us a panel (n = 3500: whole factorization 40.8 -> 21.2 ms).
__global__ void __launch_bounds__(CP_T) chol_panel_kernel(CholArgs a, int k0, int k1, int rows) {
    extern __shared__ double w[];                // [CH_NB + rows][CH_NB + 1]
    constexpr int P = CH_NB + 1;
    State *st = a.st;
    count_launch(st);
    if (*(volatile int *)&st->status == LS_BREAKDOWN) return;
    const int n = a.n, nb = k1 - k0;
    const long long ld = a.ld;
    const int i0 = k1 + blockIdx.x * rows;       // the CTA's rows i0 .. i0 + mine - 1
    const int mine = max(0, min(rows, n + 1 - i0)), all = CH_NB + mine;
    for (int e = threadIdx.x; e < all * CH_NB; e += CP_T) {
        const int r = e / CH_NB, t = e % CH_NB, i = r < CH_NB ? k0 + r : i0 + r - CH_NB;
        const bool in = t < nb && (r >= CH_NB || (r < nb && t <= r));
        w[r * P + t] = in ? a.W[(long long)i * ld + k0 + t] : 0.0;
    }
    __syncthreads();
    for (int k = 0; k < nb; k++) {
        const double piv = w[k * P + k];
        const long long pb = __double_as_longlong(piv);
        if (pb <= 0 || pb > 0x7FF0000000000000ll) {   // not above 0 (or NaN), the same in every CTA
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                st->status = LS_BREAKDOWN;
                st->iter = k0 + k;
            }
            return;
        }
        // l_rk in place of w_rk; the pivot itself after the barrier, when all have read it
        if ((int)(threadIdx.x | 31) > k && threadIdx.x < all) {
            const double lkk = sqrt(piv);
            for (int r = threadIdx.x; r < all; r += CP_T)
                if (r > k) w[r * P + k] = w[r * P + k] / lkk;
        }
        __syncthreads();
        if (threadIdx.x == CP_T - 1) w[k * P + k] = sqrt(piv);
        // elements (r, j), r > k and j = k + 1 .. min(r, nb - 1)
        const int nc = nb - 1 - k;
        for (int e = threadIdx.x; e < nc * (all - 1 - k); e += CP_T) {
            const int r = k + 1 + e / nc, j = k + 1 + e % nc;
            if (r >= j) w[r * P + j] = __dsub_rn(w[r * P + j], __dmul_rn(w[r * P + k], w[j * P + k]));
        }
        __syncthreads();
    }
    // the l's into the panel buffer and W.  The other CTAs may still read the
    // diagonal block from W: only a CTA that is alone writes it here (else the trailing update).
    for (int e = threadIdx.x; e < all * CH_NB; e += CP_T) {
        const int r = e / CH_NB, t = e % CH_NB, i = r < CH_NB ? k0 + r : i0 + r - CH_NB;
        if (t >= nb || (r < CH_NB && (r >= nb || blockIdx.x != 0 || t > r))) continue;
        a.Lp[(long long)i * CH_NB + t] = w[r * P + t];
        if (r >= CH_NB || gridDim.x == 1) a.W[(long long)i * ld + k0 + t] = w[r * P + t];
    }
}

// Rows k1 .. n, columns k1 .. min(i, n - 1): w_ij -= l_it l_jt for the
// panel's steps t in order.
__global__ void __launch_bounds__(RANK_T, 4) chol_trail_kernel(CholArgs a, int k0, int nb) {
    constexpr int RT = RANK_R, TT = RANK_TT, PITCH = RANK_PITCH;
    __shared__ Op53 Ls[CH_NB * PITCH], Ms[CH_NB * PITCH];
    State *st = a.st;
    count_launch(st);
    if (*(volatile int *)&st->status == LS_BREAKDOWN) return;
    const int n = a.n;
    const long long ld = a.ld;
    double *W = a.W;
    const double *Lp = a.Lp;
    const int k1 = k0 + nb;
    const int r0 = k1 + blockIdx.y * TT, c0 = k1 + blockIdx.x * TT;
    if (c0 > r0 + TT - 1) return;                // the tile lies above the diagonal
    if (blockIdx.x == 0 && blockIdx.y == 0)      // the panel's diagonal block of L (see chol_panel_kernel)
        for (int e = threadIdx.x; e < nb * CH_NB; e += RANK_T) {
            const int r = e / CH_NB, t = e % CH_NB;
            if (t <= r) W[(long long)(k0 + r) * ld + k0 + t] = Lp[(long long)(k0 + r) * CH_NB + t];
        }
    // rows and columns past the block are staged as ones and not stored
    RankRange range;
    for (int e = threadIdx.x; e < TT * CH_NB; e += RANK_T) {
        const int r = e / CH_NB, t = e % CH_NB;
        const Op53 l = op53_a((r0 + r <= n && t < nb) ? __ldcg(&Lp[(long long)(r0 + r) * CH_NB + t]) : 1.0);
        const Op53 m = op53_b((c0 + r < n && t < nb) ? __ldcg(&Lp[(long long)(c0 + r) * CH_NB + t]) : 1.0);
        range.a(l);
        range.b(m);
        Ls[t * PITCH + r] = l;
        Ms[t * PITCH + r] = m;
    }
    const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
    double acc[RT][RT];
#pragma unroll
    for (int p = 0; p < RT; p++)
#pragma unroll
        for (int q = 0; q < RT; q++) {
            const int r = r0 + ty + 16 * p, c = c0 + tx + 16 * q;
            acc[p][q] = (r <= n && c < n && c <= r) ? W[(long long)r * ld + c] : 0.0;
        }
    rank_tile(acc, Ls, Ms, nb, range.all_in_range(), ty, tx);
#pragma unroll
    for (int p = 0; p < RT; p++)
#pragma unroll
        for (int q = 0; q < RT; q++) {
            const int r = r0 + ty + 16 * p, c = c0 + tx + 16 * q;
            if (r <= n && c < n && c <= r) W[(long long)r * ld + c] = acc[p][q];
        }
}

__global__ void __launch_bounds__(CT, 1) chol_backsolve_kernel(CholArgs a) {
    __shared__ double s[CB], xs[CB], T[CB][CB + 1];
    __shared__ double part[CW][33];
    State *st = a.st;
    count_launch(st);
    const int n = a.n;
    const long long ld = a.ld;
    double *W = a.W;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (*(volatile int *)&st->status == LS_BREAKDOWN) return;
    double *y = a.y;                             // a copy of row n: y, then the updated right sides
    for (int r1 = n; r1 > 0; r1 -= CB) {
        const int r0 = r1 > CB ? r1 - CB : 0, nb = r1 - r0;
        if (blockIdx.x == 0) {                   // the diagonal block, transposed: t_rc = l_cr
            for (int e = threadIdx.x; e < CB * CB; e += CT) {
                const int c = e / CB, r = e % CB;
                T[r][c] = r <= c && c < nb ? W[(long long)(r0 + c) * ld + r0 + r] : 0.0;
            }
            for (int r = threadIdx.x; r < nb; r += CT) s[r] = __ldcg(&y[r0 + r]);
            __syncthreads();
            if (warp == 0) back_solve_block(nb, T, s, xs);
            __syncthreads();
            for (int r = threadIdx.x; r < nb; r += CT) a.x[r0 + r] = xs[r];
        }
        if (!grid_sync(a.bar, st)) return;
        // rows above the block: y_i -= sum_{j in block} l_ji x_j.  A CTA takes 32 rows i (the
        // block's rows of L are contiguous in i), a warp four of the block's rows;
        // the warps' sums are added pairwise.
        for (int i0 = blockIdx.x * 32; i0 < r0; i0 += gridDim.x * 32) {
            const int i = i0 + lane;
            double acc = 0.0;
            if (i < r0) {
#pragma unroll
                for (int u = 0; u < CB / CW; u++) {
                    const int jj = warp * (CB / CW) + u;
                    if (jj < nb) acc += W[(long long)(r0 + jj) * ld + i] * __ldcg(&a.x[r0 + jj]);
                }
            }
            part[warp][lane] = acc;
            __syncthreads();
            for (int o = CW / 2; o > 0; o >>= 1) {
                if (warp < o) part[warp][lane] += part[warp + o][lane];
                __syncthreads();
            }
            if (warp == 0 && i < r0) y[i] = __ldcg(&y[i]) - part[0][lane];
            __syncthreads();
        }
        if (!grid_sync(a.bar, st)) return;
    }
}

// Entries above the diagonal of the n x n factor (the rest of A's copy) to zero.
__global__ void chol_zero_upper_kernel(CholArgs a) {
    const int n = a.n;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < (long long)n * n;
         e += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(e / n), j = (int)(e % n);
        if (j > i) a.W[(long long)i * a.ld + j] = 0.0;
    }
}

CholKernels chol_kernels() {
    CholKernels K{};
    K.panel = reinterpret_cast<void *>(&chol_panel_kernel);
    K.trail = reinterpret_cast<void *>(&chol_trail_kernel);
    K.backsolve = reinterpret_cast<void *>(&chol_backsolve_kernel);
    K.zero_upper = reinterpret_cast<void *>(&chol_zero_upper_kernel);
    K.nb = CH_NB;
    K.tile = RANK_TT;
    K.block = CT;
    K.panel_block = CP_T;
    return K;
}

}  // namespace lsi
