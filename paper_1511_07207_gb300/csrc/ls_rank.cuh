// ls_rank.cuh -- the rank updates of the direct methods' trailing blocks: a tile
// of a_ij takes a_ij - l_it u_tj for the panel's steps t in order, product and
// difference each rounded (k_lu.cu, k_chol.cu).
//
// What bounds it is the FP64 pipe: one warp instruction every 64 cycles per
// scheduler.  With the product there too an update takes two of them; the
// integer pipes form the product instead (mul53.h, about 17 integer instructions,
// which issue in well under 64 cycles), which leaves one.  A tile whose
// operands leave the exponent range of mul53 (zeros, subnormals, infinities, NaN
// among them) takes the FP64 pipe for both, and so does a step of a thread's
// elements in which a product's rounding is decided below the bits mul53 forms.
//
// Tiles of 32 x 32 with 2 x 2 elements a thread: 53 registers keep 32 warps on
// an SM, which hide the integer chains behind the FP64 pipe and waste less in the
// last wave.  Staged operands are 16 bytes (one shared load each); a thread's
// elements lie 16 rows and columns apart, so that the row operands are broadcasts.
//
// Measured, whole solve: LU n = 8192 836 -> 477 ms, Cholesky n = 3500 61.0 ->
// 40.8 ms; with tiles of 64 x 64 (4 x 4 a thread, 127 registers, 16 warps) 491
// and 44.1 ms (Cholesky n = 8000: 257 against 248 ms).  The updates of n = 8192
// alone run at about 0.87 of one FP64 instruction an update (n^3 / 3 of them
// over 152 SMs x 2 a clock).
#pragma once

#include "ls_device.cuh"
#include "mul53.h"

namespace lsi {

constexpr int RANK_NB = 32;               // steps of a panel, at most
constexpr int RANK_T = 256;               // threads of a tile: 16 x 16
constexpr int RANK_R = 2;                 // rows and columns a thread
constexpr int RANK_TT = 16 * RANK_R;      // tile rows and columns
constexpr int RANK_PITCH = RANK_TT + 1;   // in operands: a column store meets each bank group once

// The extremes of the exponent fields a thread staged, joined over the tile.
struct RankRange {
    int amin = 2047, amax = 0, bmin = 2047, bmax = 0;
    __device__ __forceinline__ void a(const Op53 &o) {
        const int f = op53_field(o);
        amin = min(amin, f);
        amax = max(amax, f);
    }
    __device__ __forceinline__ void b(const Op53 &o) {
        const int f = op53_field(o);
        bmin = min(bmin, f);
        bmax = max(bmax, f);
    }
    // A barrier for the tile's threads (all RANK_T of them); true when every product is in mul53's range.
    __device__ __forceinline__ bool all_in_range() const {
        __shared__ int w[RANK_T / 32][4];
        const int lo_a = __reduce_min_sync(0xffffffffu, amin), hi_a = __reduce_max_sync(0xffffffffu, amax);
        const int lo_b = __reduce_min_sync(0xffffffffu, bmin), hi_b = __reduce_max_sync(0xffffffffu, bmax);
        if ((threadIdx.x & 31) == 0) {
            int *m = w[threadIdx.x >> 5];
            m[0] = lo_a;
            m[1] = hi_a;
            m[2] = lo_b;
            m[3] = hi_b;
        }
        __syncthreads();
        int r[4] = {w[0][0], w[0][1], w[0][2], w[0][3]};
#pragma unroll
        for (int i = 1; i < RANK_T / 32; i++) {
            r[0] = min(r[0], w[i][0]);
            r[1] = max(r[1], w[i][1]);
            r[2] = min(r[2], w[i][2]);
            r[3] = max(r[3], w[i][3]);
        }
        return mul53_in_range(r[0], r[1], r[2], r[3]);
    }
};

// acc[p][q] -= l(ty + 16 p, t) u(t, tx + 16 q) for t = 0 .. nb - 1 in order.
// Ls[t * RANK_PITCH + row] and Us[t * RANK_PITCH + column] are the staged operands.
__device__ __forceinline__ void rank_tile(double (&acc)[RANK_R][RANK_R], const Op53 *Ls, const Op53 *Us, int nb,
                                          bool fast, int ty, int tx) {
    constexpr int RT = RANK_R, PITCH = RANK_PITCH;
    if (fast) {
#pragma unroll 1
        for (int t = 0; t < nb; t++) {
            Op53 l[RT], u[RT];
#pragma unroll
            for (int p = 0; p < RT; p++) l[p] = Ls[t * PITCH + ty + 16 * p];
#pragma unroll
            for (int q = 0; q < RT; q++) u[q] = Us[t * PITCH + tx + 16 * q];
            double pr[RT][RT];
            bool tie = false;
#pragma unroll
            for (int p = 0; p < RT; p++)
#pragma unroll
                for (int q = 0; q < RT; q++) pr[p][q] = mul53(l[p], u[q], tie);
            if (tie) {
#pragma unroll
                for (int p = 0; p < RT; p++)
#pragma unroll
                    for (int q = 0; q < RT; q++)
                        pr[p][q] = __dmul_rn(op53_value(l[p], 5), op53_value(u[q], 6));
            }
#pragma unroll
            for (int p = 0; p < RT; p++)
#pragma unroll
                for (int q = 0; q < RT; q++) acc[p][q] = __dsub_rn(acc[p][q], pr[p][q]);
        }
    } else {
#pragma unroll 1
        for (int t = 0; t < nb; t++) {
            double l[RT], u[RT];
#pragma unroll
            for (int p = 0; p < RT; p++) l[p] = op53_value(Ls[t * PITCH + ty + 16 * p], 5);
#pragma unroll
            for (int q = 0; q < RT; q++) u[q] = op53_value(Us[t * PITCH + tx + 16 * q], 6);
#pragma unroll
            for (int p = 0; p < RT; p++)
#pragma unroll
                for (int q = 0; q < RT; q++) acc[p][q] = __dsub_rn(acc[p][q], __dmul_rn(l[p], u[q]));
        }
    }
}

// ---- back substitution: one diagonal block -----------------------------------------------
constexpr int BACK_B = 64;           // rows of a block

// One warp: T x = s for the upper triangular nb x nb block T (shared memory), column
// oriented: x_i = s_i / t_ii, then s_r -= t_ri x_i for r < i.  The chain is 64 of those, so
// the block is in shared memory, the reciprocals of its diagonal are formed
// at once and a quotient from one is corrected by its remainder (three dependent FP64
// instructions instead of a division's ten).
__device__ __forceinline__ void back_solve_block(int nb, const double (*T)[BACK_B + 1], const double *s, double *x) {
    const int lane = threadIdx.x & 31;
    double sv[2], d[2], inv[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int r = lane + 32 * h;
        sv[h] = r < nb ? s[r] : 0.0;
        d[h] = r < nb ? T[r][r] : 1.0;
        inv[h] = 1.0 / d[h];
    }
    for (int i = nb - 1; i >= 0; i--) {
        const int h = i >> 5, src = i & 31;
        const double si = __shfl_sync(0xffffffffu, h ? sv[1] : sv[0], src);
        const double di = __shfl_sync(0xffffffffu, h ? d[1] : d[0], src);
        const double ri = __shfl_sync(0xffffffffu, h ? inv[1] : inv[0], src);
        const double t0 = T[lane][i], t1 = T[lane + 32][i];
        double xi = si * ri;
        xi = fma(ri, fma(-di, xi, si), xi);
        // a diagonal entry or a quotient near the ends of the range: the division itself
        const int er = (__double2hiint(ri) >> 20) & 0x7FF, ex = (__double2hiint(xi) >> 20) & 0x7FF;
        if (er < 64 || er > 1982 || ex < 64 || ex > 1982) xi = si / di;
        if (lane < i) sv[0] -= t0 * xi;
        if (lane + 32 < i) sv[1] -= t1 * xi;
        if (lane == 0) x[i] = xi;
    }
}

}  // namespace lsi
