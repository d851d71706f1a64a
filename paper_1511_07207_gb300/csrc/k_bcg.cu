// k_bcg.cu -- block conjugate gradient for s right-hand sides: O'Leary's form
// and a deflating form with orthonormal, rank-revealed search directions (the
// second half of this file).
//
// Block CG (the paper's CG paragraph, for several right-hand sides at once
// in O'Leary's block form) replaces CG's scalars by s x s matrices:
//   Q = A P;  gamma = P^T Q;  alpha = gamma^-1 rho;  X += P alpha;
//   R -= Q alpha;  rho' = R^T R;  beta = rho^-1 rho';  P = R + P beta.
// The products Q = A P are s launches of the solvers' GEMV (one per column,
// each streaming A once as the FP32 pair); everything else of a step is
// one cooperative kernel:
//   bcg_step   gamma (per-CTA partial Gram matrices over row ranges, reduced
//              in CTA order), one warp factors gamma (Cholesky) and solves
//              for alpha; every CTA updates its rows of X and R and forms
//              its partial R^T R; one warp tests every column, factors rho'
//              and solves for beta; every CTA forms P = R + P beta row by
//              row.  Three bounded grid barriers.
//   bcg_init   X = 0 (or keep X0, R from the residual GEMVs), P = R,
//              rho = R^T R and its factor, ||B_j||, the loop conditions.
//   bcg_check  after the loop: accept when every column's true residual
//              passes, or restart from it (P = R, rho = R^T R).
// The s x s algebra is FP64 on one warp (s <= 16): Cholesky column by column
// with the lanes over rows, triangular solves with the lanes over right-hand
// sides.  A factor that meets a non-positive pivot (a rank-deficient block)
// is a breakdown.  Blocks are column-major n x s with column stride ld.
#include <cuda_runtime.h>

#include "ls_device.cuh"
#include "ls_internal.h"

namespace lsi {

constexpr int BK = 256;   // threads per CTA

// ---- one warp: s x s Cholesky and solves (column-major, shared memory) ------------
// G = L L^T in place (L in the lower triangle); false on a non-positive pivot.
__device__ bool warp_chol(int s, double *G) {
    const int lane = threadIdx.x & 31;
    for (int j = 0; j < s; j++) {
        double d = G[j + j * s];
        for (int k = 0; k < j; k++) d -= G[j + k * s] * G[j + k * s];
        if (!(d > 0.0)) return false;          // same value in every lane
        d = sqrt(d);
        __syncwarp();
        if (lane > j && lane < s) {
            double v = G[lane + j * s];
            for (int k = 0; k < j; k++) v -= G[lane + k * s] * G[j + k * s];
            G[lane + j * s] = v / d;
        }
        if (lane == 0) G[j + j * s] = d;
        __syncwarp();
    }
    return true;
}

// Y = (L L^T)^-1 Y, one right-hand side per lane.
__device__ void warp_chol_solve(int s, const double *L, double *Y) {
    const int c = threadIdx.x & 31;
    if (c < s) {
        double *y = Y + c * s;
        for (int i = 0; i < s; i++) {
            double v = y[i];
            for (int k = 0; k < i; k++) v -= L[i + k * s] * y[k];
            y[i] = v / L[i + i * s];
        }
        for (int i = s - 1; i >= 0; i--) {
            double v = y[i];
            for (int k = i + 1; k < s; k++) v -= L[k + i * s] * y[k];
            y[i] = v / L[i + i * s];
        }
    }
    __syncwarp();
}

// ---- Gram matrices -------------------------------------------------------------------
// This CTA's partial U^T V over rows [lo, hi) into part[cta][s*s]: T =
// BK / s^2 threads per entry, thread q summing rows lo + q, lo + q + T, ...,
// the T sums added in q order (all threads of the CTA call it).
__device__ __forceinline__ void gram_partial(const BcgVecs &v, const double *U, const double *V, long long lo,
                                             long long hi) {
    __shared__ double red[BK];
    const int s = v.s, E = s * s, T = BK / E;
    const int e = threadIdx.x / T, q = threadIdx.x - e * T;
    double acc = 0.0;
    if (e < E) {
        const int a = e % s, b = e / s;
        const double *u = U + (long long)a * v.ld, *w = V + (long long)b * v.ld;
        for (long long i = lo + q; i < hi; i += T) acc += u[i] * w[i];
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    if (e < E && q == 0) {
        double sum = 0.0;
        for (int t = 0; t < T; t++) sum += red[threadIdx.x + t];
        v.part[(size_t)blockIdx.x * BCG_MAX_S * BCG_MAX_S + e] = sum;
    }
    __syncthreads();
}

// One warp: G = sum of the partials, entry by entry, as eight interleaved
// sums over the CTAs added pairwise (a fixed order).
__device__ __forceinline__ void gram_reduce(const BcgVecs &v, double *G) {
    const int s = v.s, nc = (int)gridDim.x;
    for (int e = threadIdx.x & 31; e < s * s; e += 32) {
        double t[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        for (int c = 0; c < nc; c++) t[c & 7] += __ldcg(&v.part[(size_t)c * BCG_MAX_S * BCG_MAX_S + e]);
        G[e] = ((t[0] + t[1]) + (t[2] + t[3])) + ((t[4] + t[5]) + (t[6] + t[7]));
    }
    __syncwarp();
}

__device__ __forceinline__ bool all_pass(const BcgVecs &v, const double *rho) {
    bool ok = true;
    for (int j = 0; j < v.s; j++) ok = ok && sqrt(rho[j + j * v.s]) <= v.st->rtol * v.sm->bn[j];
    return ok;
}

// ---- init ----------------------------------------------------------------------------
__global__ void __launch_bounds__(BK) bcg_init_kernel(BcgVecs v, int x0_given, cudaGraphConditionalHandle h_outer,
                                                      cudaGraphConditionalHandle h_inner) {
    __shared__ double G[BCG_MAX_S * BCG_MAX_S];
    State *st = v.st;
    BcgSmall *sm = v.sm;
    count_launch(st);
    long long lo, hi;
    block_range(v.n, blockIdx.x, gridDim.x, lo, hi);
    for (int j = 0; j < v.s; j++)
        for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x) {
            const long long o = (long long)j * v.ld + i;
            if (!x0_given) {
                v.X[o] = 0.0;
                v.R[o] = v.B[o];
            }
            v.P[o] = v.R[o];
        }
    __syncthreads();
    gram_partial(v, v.R, v.R, lo, hi);
    // partial ||B_j||^2
    for (int j = threadIdx.x; j < v.s; j += blockDim.x) {
        const double *b = v.B + (long long)j * v.ld;
        double acc = 0.0;
        for (long long i = lo; i < hi; i++) acc += b[i] * b[i];
        v.part2[(size_t)blockIdx.x * BCG_MAX_S + j] = acc;
    }
    if (!grid_sync(v.bar, st)) return;
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        gram_reduce(v, G);
        const int lane = threadIdx.x;
        if (lane < v.s) {
            double acc = 0.0;
            for (int c = 0; c < (int)gridDim.x; c++) acc += __ldcg(&v.part2[(size_t)c * BCG_MAX_S + lane]);
            sm->bn[lane] = sqrt(acc);
        }
        __syncwarp();
        for (int e = lane; e < v.s * v.s; e += 32) sm->rho[e] = G[e];
        bool nan = false;
        for (int e = 0; e < v.s * v.s; e++) nan = nan || !isfinite(G[e]);
        for (int j = 0; j < v.s; j++) nan = nan || !isfinite(sm->bn[j]);
        const bool pass = !nan && all_pass(v, G);
        bool factored = false;
        if (!nan && !pass) factored = warp_chol(v.s, G);
        for (int e = lane; e < v.s * v.s; e += 32) sm->L[e] = G[e];
        if (lane == 0) {
            int go = 1;
            if (nan) {
                set_err(st, ERRB_NAN);
                go = 0;
            } else if (pass) {
                go = 0;                               // confirm on the true residual
            } else if (!factored) {
                st->status = LS_BREAKDOWN;            // rank-deficient residual block
                go = 0;
            } else if (st->max_iter <= 0) {
                go = 0;
            }
            set_cond(st, h_inner, go);
            set_cond(st, h_outer, 1u);
        }
    }
}

// ---- one step after Q = A P ---------------------------------------------------------------
__global__ void __launch_bounds__(BK) bcg_step_kernel(BcgVecs v, cudaGraphConditionalHandle h_inner) {
    __shared__ double G[BCG_MAX_S * BCG_MAX_S], Y[BCG_MAX_S * BCG_MAX_S];
    __shared__ double coef[BCG_MAX_S * BCG_MAX_S];
    __shared__ int flag_s;
    State *st = v.st;
    BcgSmall *sm = v.sm;
    count_launch(st);
    const int s = v.s;
    if (*(volatile int *)&st->err || *(volatile int *)&st->status == LS_BREAKDOWN) {
        if (blockIdx.x == 0 && threadIdx.x == 0) set_cond(st, h_inner, 0u);
        return;
    }
    long long lo, hi;
    block_range(v.n, blockIdx.x, gridDim.x, lo, hi);
    // gamma = P^T Q
    gram_partial(v, v.P, v.Q, lo, hi);
    if (!grid_sync(v.bar, st)) return;
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        gram_reduce(v, G);
        const bool ok = warp_chol(s, G);
        if (ok) {
            for (int e = threadIdx.x; e < s * s; e += 32) Y[e] = sm->rho[e];
            __syncwarp();
            warp_chol_solve(s, G, Y);                    // alpha = gamma^-1 rho
            for (int e = threadIdx.x; e < s * s; e += 32) sm->alpha[e] = Y[e];
        }
        if (threadIdx.x == 0) {
            sm->ok = ok ? 1 : 0;
            if (!ok) st->status = LS_BREAKDOWN;
        }
    }
    if (!grid_sync(v.bar, st)) return;
    if (threadIdx.x == 0) flag_s = *(volatile int *)&sm->ok;
    __syncthreads();
    if (!flag_s) {
        if (blockIdx.x == 0 && threadIdx.x == 0) set_cond(st, h_inner, 0u);
        return;
    }
    // X += P alpha, R -= Q alpha (row by row, all s columns), partial R^T R
    for (int e = threadIdx.x; e < s * s; e += blockDim.x) coef[e] = __ldcg(&sm->alpha[e]);
    __syncthreads();
    for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x) {
        double p[BCG_MAX_S], q[BCG_MAX_S];
#pragma unroll
        for (int c = 0; c < BCG_MAX_S; c++) {
            p[c] = c < s ? v.P[(long long)c * v.ld + i] : 0.0;
            q[c] = c < s ? v.Q[(long long)c * v.ld + i] : 0.0;
        }
        for (int j = 0; j < s; j++) {
            double dx = 0.0, dr = 0.0;
#pragma unroll
            for (int c = 0; c < BCG_MAX_S; c++)
                if (c < s) {
                    dx += p[c] * coef[c + j * s];
                    dr += q[c] * coef[c + j * s];
                }
            v.X[(long long)j * v.ld + i] += dx;
            v.R[(long long)j * v.ld + i] -= dr;
        }
    }
    __syncthreads();
    gram_partial(v, v.R, v.R, lo, hi);
    if (!grid_sync(v.bar, st)) return;
    // rho' = R^T R: stop test, or beta = rho^-1 rho' and the factor of rho'
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        gram_reduce(v, G);                                // rho'
        bool nan = false;
        for (int e = 0; e < s * s; e++) nan = nan || !isfinite(G[e]);
        const bool pass = !nan && all_pass(v, G);
        int go = 0;
        if (!nan && !pass) {
            for (int e = threadIdx.x; e < s * s; e += 32) Y[e] = G[e];
            for (int e = threadIdx.x; e < s * s; e += 32) coef[e] = sm->L[e];
            __syncwarp();
            warp_chol_solve(s, coef, Y);                  // beta = rho^-1 rho'
            for (int e = threadIdx.x; e < s * s; e += 32) sm->beta[e] = Y[e];
            for (int e = threadIdx.x; e < s * s; e += 32) sm->rho[e] = G[e];
            __syncwarp();
            const bool ok = warp_chol(s, G);              // factor of rho' for the next step
            for (int e = threadIdx.x; e < s * s; e += 32) sm->L[e] = G[e];
            go = ok ? 1 : 0;
            if (threadIdx.x == 0 && !ok) st->status = LS_BREAKDOWN;
        } else {
            for (int e = threadIdx.x; e < s * s; e += 32) sm->rho[e] = G[e];
        }
        if (threadIdx.x == 0) {
            st->iter++;
            if (nan) set_err(st, ERRB_NAN);
            if (go && st->iter >= st->max_iter) go = 0;
            sm->ok = go;
            sm->update_p = (!nan && !pass && *(volatile int *)&st->status != LS_BREAKDOWN) ? 1 : 0;
            set_cond(st, h_inner, go ? 1u : 0u);
        }
    }
    if (!grid_sync(v.bar, st)) return;
    if (threadIdx.x == 0) flag_s = *(volatile int *)&sm->update_p;
    __syncthreads();
    if (!flag_s) return;
    // P = R + P beta (row by row)
    for (int e = threadIdx.x; e < s * s; e += blockDim.x) coef[e] = __ldcg(&sm->beta[e]);
    __syncthreads();
    for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x) {
        double p[BCG_MAX_S];
#pragma unroll
        for (int c = 0; c < BCG_MAX_S; c++) p[c] = c < s ? v.P[(long long)c * v.ld + i] : 0.0;
        for (int j = 0; j < s; j++) {
            double acc = v.R[(long long)j * v.ld + i];
#pragma unroll
            for (int c = 0; c < BCG_MAX_S; c++)
                if (c < s) acc += p[c] * coef[c + j * s];
            v.P[(long long)j * v.ld + i] = acc;
        }
    }
}

// ---- after the loop: the true residual R = B - A X (written by the residual
// GEMVs, with ||R_j||^2 in sm->r2) -----------------------------------------------------------
__global__ void __launch_bounds__(BK) bcg_check_kernel(BcgVecs v, cudaGraphConditionalHandle h_outer,
                                                       cudaGraphConditionalHandle h_inner) {
    __shared__ double G[BCG_MAX_S * BCG_MAX_S];
    __shared__ int restart_s;
    State *st = v.st;
    BcgSmall *sm = v.sm;
    count_launch(st);
    const int s = v.s;
    if (threadIdx.x == 0) {
        bool pass = true, nan = false;
        for (int j = 0; j < s; j++) {
            const double r2 = *(volatile double *)&sm->r2[j];
            nan = nan || !isfinite(r2);
            pass = pass && sqrt(r2) <= v.st->rtol * sm->bn[j];
        }
        int restart = 0;
        if (*(volatile int *)&st->err || nan) {
            if (nan) set_err(st, ERRB_NAN);
        } else if (*(volatile int *)&st->status == LS_BREAKDOWN) {
            // a factor failed: stop with the last iterate
        } else if (pass) {
            if (blockIdx.x == 0) st->status = LS_OK;
        } else if (*(volatile int *)&st->iter >= st->max_iter) {
            if (blockIdx.x == 0) st->status = LS_NOT_CONVERGED;
        } else {
            restart = 1;
        }
        restart_s = restart;
    }
    __syncthreads();
    if (!restart_s) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            set_cond(st, h_outer, 0u);
            set_cond(st, h_inner, 0u);
        }
        return;
    }
    // restart from the true residual: P = R, rho = R^T R and its factor
    long long lo, hi;
    block_range(v.n, blockIdx.x, gridDim.x, lo, hi);
    for (int j = 0; j < s; j++)
        for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x)
            v.P[(long long)j * v.ld + i] = v.R[(long long)j * v.ld + i];
    __syncthreads();
    gram_partial(v, v.R, v.R, lo, hi);
    if (!grid_sync(v.bar, st)) return;
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        gram_reduce(v, G);
        for (int e = threadIdx.x; e < s * s; e += 32) sm->rho[e] = G[e];
        __syncwarp();
        const bool ok = warp_chol(s, G);
        for (int e = threadIdx.x; e < s * s; e += 32) sm->L[e] = G[e];
        if (threadIdx.x == 0) {
            if (!ok) st->status = LS_BREAKDOWN;
            st->cycles++;
            set_cond(st, h_inner, ok ? 1u : 0u);
            set_cond(st, h_outer, 1u);
        }
    }
}

// ============================================================================
// The deflating form: the search directions P are kept orthonormal and of
// full rank r <= s by a rank-revealing orthogonalization, dependent ones
// dropped, so dependent, zero or converged residual columns never make a
// step matrix singular (block CG with orthonormalized directions, as in the
// breakdown-free block CG of Ji and Li):
//   Q = A P;  gamma = P^T Q (r x r);  alpha = gamma^-1 (P^T R);
//   X += P alpha;  R -= Q alpha;  per-column stop test;
//   beta = -gamma^-1 (Q^T R);  P = orth(R + P beta).
// The new directions are A-conjugate to P and span the same block Krylov
// space as O'Leary's, so with a full-rank block the iterates are the same.
// orth(W): W^T W, columns normalized to unit norm, Cholesky with diagonal
// pivoting (largest remaining diagonal first) that stops when the remaining
// diagonal is at most tau^2 = 1e-16 (the column's part outside the span of
// the taken ones is at most 1e-8 of its norm: dependent), then P = W T with
// T = D^-1 Pi L^-T, and a second pass (Gram of P, Cholesky, P = P L2^-T).
// Small matrices use leading dimension BCG_MAX_S; the s x s algebra (at most
// 16 x 16) runs in every CTA, spread over a warp or 16 lanes a column.
// ============================================================================
constexpr int SL = BCG_MAX_S;              // leading dimension of the small matrices
constexpr double BCGD_TAU2 = 1e-16;        // (1e-8)^2 on the normalized diagonal

// Entry e of an nu x nv Gram matrix; sym: of its lower triangle (a >= b).
__device__ __forceinline__ int gram_entries(int nu, int nv, bool sym) { return sym ? nu * (nu + 1) / 2 : nu * nv; }
__device__ __forceinline__ void gram_entry(int e, int nu, bool sym, int &a, int &b) {
    if (!sym) {
        a = e % nu;
        b = e / nu;
        return;
    }
    a = 0;
    while ((a + 1) * (a + 2) / 2 <= e) a++;
    b = e - a * (a + 1) / 2;
}

// This CTA's partial U[:, :nu]^T V[:, :nv] over rows [lo, hi) into
// buf[cta][e].  Every thread of the CTA takes part: T = BK / E threads per
// entry, thread q of an entry summing rows lo + q, lo + q + T, ...; the T sums
// added in q order (a fixed order, so the result does not depend on timing).  A
// warp's FP64 instruction takes about 64 cycles of its scheduler's FP64 unit on
// this GPU, so short chains spread over all four schedulers are what counts.
__device__ __forceinline__ void gram_partial_ld(const BcgVecs &v, double *buf, const double *U, int nu,
                                                const double *V, int nv, bool sym, long long lo, long long hi) {
    __shared__ double red[BK];
    const int E = gram_entries(nu, nv, sym);
    if (E == 0) return;
    const int T = BK / E;
    const int e = threadIdx.x / T, q = threadIdx.x - e * T;
    double acc = 0.0;
    if (e < E) {
        int a, b;
        gram_entry(e, nu, sym, a, b);
        const double *u = U + (long long)a * v.ld, *w = V + (long long)b * v.ld;
#pragma unroll 4
        for (long long i = lo + q; i < hi; i += T) acc += u[i] * w[i];
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    if (e < E && q == 0) {
        double sum = red[threadIdx.x];
        for (int t = 1; t < T; t++) sum += red[threadIdx.x + t];
        buf[(size_t)blockIdx.x * SL * SL + e] = sum;
    }
    __syncthreads();
}
// G = the sum of the CTAs' partials, by threads t0 .. BK - 1 of the calling CTA (t0 a
// multiple of 32; a barrier of those threads inside): T threads an entry, thread q of
// them adding CTAs q, q + T, ..., then the T sums in q order.  The order depends on
// nothing but the sizes, so every CTA that does this gets the same bits.
// A lower triangle is mirrored.
__device__ __forceinline__ void gram_reduce_ld(const double *buf, int nu, int nv, bool sym, double *G, int t0) {
    __shared__ double red[BK];
    const int E = gram_entries(nu, nv, sym), nt = BK - t0, nc = (int)gridDim.x;
    if (E == 0) return;
    const int T = max(1, nt / E), t = (int)threadIdx.x - t0;
    for (int e0 = 0; e0 < E; e0 += nt) {              // more than one round only for 16 x 16 and t0 > 0
        const int e = e0 + t % (T > 1 ? E : nt), q = T > 1 ? t / E : 0;
        double acc = 0.0;
        if (e < E && q < T) {
#pragma unroll 8
            for (int c = q; c < nc; c += T) acc += __ldcg(&buf[(size_t)c * SL * SL + e]);
        }
        red[threadIdx.x] = acc;
        named_bar(2, nt);
        if (e < E && q == 0) {
            for (int i = 1; i < T; i++) acc += red[threadIdx.x + i * E];
            int a, b;
            gram_entry(e, nu, sym, a, b);
            G[a + b * SL] = acc;
            if (sym) G[b + a * SL] = acc;
        }
        named_bar(2, nt);
    }
}

__device__ __forceinline__ bool positive(double x) {   // x > 0 and not NaN, off the FP64 pipe
    const long long b = __double_as_longlong(x);
    return b > 0 && b <= 0x7FF0000000000000ll;
}

// One warp: Cholesky of the leading r x r block (lower triangle, leading
// dimension SL), right-looking, and the reciprocals of its diagonal; false on a pivot
// that is not positive.  One reciprocal square root a column: a square root
// and a division are 0.3 us each on the chain.
__device__ bool warp_chol_ld(int r, double *G, double *dinv) {
    const int lane = threadIdx.x & 31;
    for (int k = 0; k < r; k++) {
        const double d = G[k + k * SL];
        if (!positive(d)) return false;                // the same in every lane
        const double rs = rsqrt(d);
        __syncwarp();
        if (lane >= k && lane < r) G[lane + k * SL] = (lane == k ? d : G[lane + k * SL]) * rs;
        if (lane == 0) dinv[k] = rs;
        __syncwarp();
        const int m = r - 1 - k;
        for (int e = lane; e < m * m; e += 32) {
            const int i = k + 1 + e % m, j = k + 1 + e / m;
            if (i >= j) G[i + j * SL] -= G[i + k * SL] * G[j + k * SL];
        }
        __syncwarp();
    }
    return true;
}

// All threads, thread (k, c) = (tid % 16, tid / 16) holding entry (k, c) of an
// r x 16 block: y = L^-1 y, and with `both` L^-T (L^-1 y).  The 16 lanes of a column
// hand each other the finished entries by shuffles.
__device__ __forceinline__ double team_solve(int r, const double *L, const double *dinv, double y, bool both) {
    const int k = threadIdx.x & 15, base = threadIdx.x & 16;
    for (int i = 0; i < r; i++) {
        const double yi = __shfl_sync(0xffffffffu, y, base | i) * dinv[i];
        if (k == i) y = yi;
        else if (k > i && k < r) y -= L[k + i * SL] * yi;
    }
    if (both)
        for (int i = r - 1; i >= 0; i--) {
            const double yi = __shfl_sync(0xffffffffu, y, base | i) * dinv[i];
            if (k == i) y = yi;
            else if (k < i) y -= L[i + k * SL] * yi;
        }
    return y;
}
// Y (r x c, c <= 16) = (L L^T)^-1 Y.  Warps without a column of Y sit out.
__device__ __forceinline__ void team_chol_solve(int r, int c, const double *L, const double *dinv, double *Y) {
    const int k = threadIdx.x & 15, col = threadIdx.x >> 4;
    if ((int)(threadIdx.x >> 5) * 2 < c) {
        double y = k < r && col < c ? Y[k + col * SL] : 0.0;
        y = team_solve(r, L, dinv, y, true);
        if (k < r && col < c) Y[k + col * SL] = y;
    }
    __syncthreads();
}
// T = scale L^-T in rows perm (scale and perm may be null): T[perm[a] + b SL] = (L^-1)_ba scale[perm[a]].
__device__ __forceinline__ void team_inv_t(int r, const double *L, const double *dinv, const int *perm,
                                           const double *scale, double *T) {
    const int k = threadIdx.x & 15, col = threadIdx.x >> 4;
    T[threadIdx.x] = 0.0;                              // SL * SL = BK entries
    __syncthreads();
    if ((int)(threadIdx.x >> 5) * 2 < r) {
        const double y = team_solve(r, L, dinv, k == col ? 1.0 : 0.0, false);
        if (col < r && k >= col && k < r) {
            const int row = perm ? perm[col] : col;
            T[row + k * SL] = scale ? y * scale[row] : y;
        }
    }
    __syncthreads();
}
static_assert(SL * SL == BK, "a thread an entry of the small matrices");

// First pass of orth, one warp (lane q: column q): from G = W^T W (s x s) the rank r,
// the order of the kept columns, the Cholesky factor Lp of their normalized Gram matrix
// with the reciprocals of its diagonal, and the reciprocal column norms.
// Lc: s x SL scratch.
__device__ int rr_factor(int s, const double *G, double *Lc, double *Lp, double *dinv, double *scale, int *perm) {
    const int q = threadIdx.x & 31;
    const double gq = q < s ? G[q + q * SL] : 0.0;
    const double sq = positive(gq) ? rsqrt(gq) : 0.0;
    if (q < s) scale[q] = sq;
    __syncwarp();
    bool open = positive(gq);                          // not taken, not dropped
    double rem = 1.0;
    int r = 0;
    for (;;) {
        open = open && rem > BCGD_TAU2;
        // the open column with the most left, the first one on ties (bits order as positive values do)
        const long long bits = open ? __double_as_longlong(rem) : -1ll;
        long long best = bits;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
        if (best < 0) break;
        const int p = __ffs(__ballot_sync(0xffffffffu, bits == best)) - 1;
        const double rp = __longlong_as_double(best), linv = rsqrt(rp);
        const double np = scale[p];
        double l = 0.0;
        if (q == p) {
            l = rp * linv;                             // sqrt(rem)
            perm[r] = p;
            dinv[r] = linv;
            open = false;
        } else if (open) {
            double x = G[q + p * SL] * sq * np;
            for (int t = 0; t < r; t++) x -= Lc[q + t * SL] * Lc[p + t * SL];
            l = x * linv;
            rem -= l * l;
        }
        if (q < s) Lc[q + r * SL] = l;
        __syncwarp();
        r++;
    }
    __syncwarp();
    for (int e = q; e < r * r; e += 32) {
        const int i = e % r, t = e / r;
        Lp[i + t * SL] = t <= i ? Lc[perm[i] + t * SL] : 0.0;
    }
    __syncwarp();
    return r;
}

// out[i, b] = (add ? add[i, b] : 0) + sum_{c < nc} in[i, c] T[c, b] for this CTA's rows and b < nb, a thread an
// element.  out may be `in`: a round of elements is formed before any of it is stored,
// and a round holds whole rows.
__device__ __forceinline__ void rows_times(const BcgVecs &v, double *out, const double *add, const double *in, int nc,
                                           const double *T, int nb, long long lo, long long hi) {
    if (nb == 0) return;
    const int per = BK / nb;                           // rows a round
    const int r = threadIdx.x % per, b = threadIdx.x / per;
    for (long long i0 = lo; i0 < hi; i0 += per) {
        const long long i = i0 + r;
        const bool on = b < nb && i < hi;
        double acc = 0.0;
        if (on) {
#pragma unroll 4
            for (int c = 0; c < nc; c++) acc += in[(long long)c * v.ld + i] * T[c + b * SL];
            if (add) acc += add[(long long)b * v.ld + i];
        }
        if (out == in) __syncthreads();
        if (on) out[(long long)b * v.ld + i] = acc;
    }
    __syncthreads();
}

// P = orth(W) over the whole grid (cooperative launch; W and P must differ).
// Every CTA reduces the partial Gram matrices and factors them for itself
// (the same operations, the same bits), so a pass has one barrier of the grid.  On
// return `rank` holds r in every CTA, and sm->rank and sm->w2 (the squared column
// norms of W) are set.  false if a grid barrier gave up or the second pass failed.
__device__ bool coop_orth(const BcgVecs &v, const double *W, long long lo, long long hi, int &rank) {
    __shared__ double G[SL * SL], T[SL * SL], Lc[SL * SL], dinv[SL], scale[SL];
    __shared__ int r_s, perm[SL];
    BcgSmall *sm = v.sm;
    const int s = v.s;
    gram_partial_ld(v, v.part, W, s, W, s, true, lo, hi);
    if (!grid_sync(v.bar, v.st)) return false;
    gram_reduce_ld(v.part, s, s, true, G, 0);
    if (threadIdx.x < 32) {
        bool nan = false;
        for (int j = 0; j < s; j++) nan = nan || !isfinite(G[j + j * SL]);
        const int r = nan ? 0 : rr_factor(s, G, Lc, T, dinv, scale, perm);
        if (threadIdx.x == 0) r_s = r;
        if (blockIdx.x == 0) {
            if ((int)threadIdx.x < s) sm->w2[threadIdx.x] = G[threadIdx.x * (SL + 1)];
            if (threadIdx.x == 0) sm->rank = r;
        }
    }
    __syncthreads();
    const int r = rank = r_s;
    G[threadIdx.x] = T[threadIdx.x];                   // the factor, so that T can take L^-T
    __syncthreads();
    team_inv_t(r, G, dinv, perm, scale, T);
    rows_times(v, v.P, nullptr, W, s, T, s, lo, hi);   // P = W T, zero past column r
    gram_partial_ld(v, v.partb, v.P, r, v.P, r, true, lo, hi);   // second pass
    if (!grid_sync(v.bar, v.st)) return false;
    gram_reduce_ld(v.partb, r, r, true, G, 0);
    if (threadIdx.x < 32) {
        const bool ok = warp_chol_ld(r, G, dinv);
        if (threadIdx.x == 0) r_s = ok;
    }
    __syncthreads();
    if (!r_s) {
        if (blockIdx.x == 0 && threadIdx.x == 0) sm->rank = -1;
        return false;
    }
    team_inv_t(r, G, dinv, nullptr, nullptr, T);
    rows_times(v, v.P, nullptr, v.P, r, T, r, lo, hi);  // P = P L2^-T
    return true;
}

// Every column's ||R_j|| <= rtol ||B_j|| (r2 = the squared norms).
__device__ __forceinline__ bool cols_pass(const BcgVecs &v, const double *r2) {
    bool ok = true;
    for (int j = 0; j < v.s; j++) ok = ok && sqrt(r2[j]) <= v.st->rtol * v.sm->bn[j];
    return ok;
}

// X = 0 and R = B (or R from the residual GEMVs), ||B_j||, P = orth(R), the
// loop conditions.
__global__ void __launch_bounds__(BK) bcgd_init_kernel(BcgVecs v, int x0_given, cudaGraphConditionalHandle h_outer,
                                                       cudaGraphConditionalHandle h_inner) {
    State *st = v.st;
    BcgSmall *sm = v.sm;
    count_launch(st);
    long long lo, hi;
    block_range(v.n, blockIdx.x, gridDim.x, lo, hi);
    for (int j = 0; j < v.s; j++)
        for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x) {
            const long long o = (long long)j * v.ld + i;
            if (!x0_given) {
                v.X[o] = 0.0;
                v.R[o] = v.B[o];
            }
        }
    for (int j = threadIdx.x; j < v.s; j += blockDim.x) {
        const double *b = v.B + (long long)j * v.ld;
        double acc = 0.0;
        for (long long i = lo; i < hi; i++) acc += b[i] * b[i];
        v.part2[(size_t)blockIdx.x * BCG_MAX_S + j] = acc;
    }
    __syncthreads();
    if (!grid_sync(v.bar, st)) return;
    if (blockIdx.x == 0 && threadIdx.x < v.s) {   // eight interleaved sums over the CTAs
        double t[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        for (int c = 0; c < (int)gridDim.x; c++) t[c & 7] += __ldcg(&v.part2[(size_t)c * BCG_MAX_S + threadIdx.x]);
        sm->bn[threadIdx.x] = sqrt(((t[0] + t[1]) + (t[2] + t[3])) + ((t[4] + t[5]) + (t[6] + t[7])));
    }
    int rank = 0;
    const bool ok = coop_orth(v, v.R, lo, hi, rank);    // its first barrier publishes bn too
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        bool nan = false;
        for (int j = 0; j < v.s; j++) nan = nan || !isfinite(sm->w2[j]) || !isfinite(sm->bn[j]);
        const bool pass = !nan && cols_pass(v, sm->w2);
        int go = 1;
        if (!ok) {
            go = 0;
            if (!*(volatile int *)&st->err) st->status = LS_BREAKDOWN;
        } else if (nan) {
            set_err(st, ERRB_NAN);
            go = 0;
        } else if (pass || rank == 0) {
            go = 0;                                     // confirm on the true residual
        } else if (st->max_iter <= 0) {
            go = 0;
        }
        set_cond(st, h_inner, go);
        set_cond(st, h_outer, 1u);
    }
}

// One step after Q = A P.  Four grid barriers: behind each, every CTA reduces the partial
// sums and does the s x s algebra for itself, so nothing waits for one
// CTA's answer.  What bounds it is latency: FP64 chains of the small matrices and
// the barriers.  (One CTA doing the algebra, one thread of it the factorizations,
// with eight barriers: 294 us a step at n = 8192, s = 8.)
__global__ void __launch_bounds__(BK) bcgd_step_kernel(BcgVecs v, cudaGraphConditionalHandle h_inner) {
    __shared__ double G[SL * SL], H[SL * SL], dinv[SL], r2[BCG_MAX_S];
    __shared__ int flag_s;
    State *st = v.st;
    BcgSmall *sm = v.sm;
    count_launch(st);
    const int s = v.s;
    if (*(volatile int *)&st->err || *(volatile int *)&st->status == LS_BREAKDOWN) {
        if (blockIdx.x == 0 && threadIdx.x == 0) set_cond(st, h_inner, 0u);
        return;
    }
    const int r = __ldcg(&sm->rank), iter = __ldcg(&st->iter), max_iter = st->max_iter;
    long long lo, hi;
    block_range(v.n, blockIdx.x, gridDim.x, lo, hi);
    // gamma = P^T Q and P^T R
    gram_partial_ld(v, v.part, v.P, r, v.Q, r, true, lo, hi);
    gram_partial_ld(v, v.partb, v.P, r, v.R, s, false, lo, hi);
    if (!grid_sync(v.bar, st)) return;
    gram_reduce_ld(v.part, r, r, true, G, 0);
    __syncthreads();
    if (threadIdx.x < 32) {
        const bool ok = warp_chol_ld(r, G, dinv);      // positive definite for SPD A
        if (threadIdx.x == 0) flag_s = ok;
    } else {
        gram_reduce_ld(v.partb, r, s, false, H, 32);
    }
    __syncthreads();
    if (!flag_s) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            st->status = LS_BREAKDOWN;
            set_cond(st, h_inner, 0u);
        }
        return;
    }
    team_chol_solve(r, s, G, dinv, H);                 // alpha = gamma^-1 P^T R
    // X += P alpha, R -= Q alpha, then Q^T R and ||R_j||^2
    rows_times(v, v.X, v.X, v.P, r, H, s, lo, hi);
    H[threadIdx.x] = -H[threadIdx.x];
    __syncthreads();
    rows_times(v, v.R, v.R, v.Q, r, H, s, lo, hi);
    gram_partial_ld(v, v.partc, v.Q, r, v.R, s, false, lo, hi);   // others may still read part and partb
    {   // ||R_j||^2 over this CTA's rows: 16 lanes a column
        const int j = threadIdx.x >> 4, q = threadIdx.x & 15;
        double acc = 0.0;
        if (j < s)
            for (long long i = lo + q; i < hi; i += 16) {
                const double x = v.R[(long long)j * v.ld + i];
                acc += x * x;
            }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (j < s && q == 0) v.part2[(size_t)blockIdx.x * BCG_MAX_S + j] = acc;
    }
    if (!grid_sync(v.bar, st)) return;
    gram_reduce_ld(v.partc, r, s, false, H, 0);
    {   // ||R_j||^2 over the CTAs
        const int j = threadIdx.x >> 4, q = threadIdx.x & 15;
        double acc = 0.0;
        if (j < s) {
#pragma unroll 4
            for (int c = q; c < (int)gridDim.x; c += 16) acc += __ldcg(&v.part2[(size_t)c * BCG_MAX_S + j]);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (j < s && q == 0) r2[j] = acc;
    }
    __syncthreads();
    // the stop test, the same in every CTA: lane j tests column j
    if (threadIdx.x < 32) {
        const double x = (int)threadIdx.x < s ? r2[threadIdx.x] : 0.0;
        const bool nan = __any_sync(0xffffffffu, !isfinite(x));
        const bool pass = __all_sync(0xffffffffu, (int)threadIdx.x >= s || sqrt(x) <= v.st->rtol * __ldcg(&sm->bn[threadIdx.x & 15]));
        if (threadIdx.x == 0) flag_s = nan ? -1 : pass ? 0 : 1;
    }
    __syncthreads();
    const int flag = flag_s;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->iter = iter + 1;
        if (flag < 0) set_err(st, ERRB_NAN);
    }
    if (flag <= 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) set_cond(st, h_inner, 0u);
        return;
    }
    team_chol_solve(r, s, G, dinv, H);                 // beta = -gamma^-1 Q^T R
    H[threadIdx.x] = -H[threadIdx.x];
    __syncthreads();
    // W = R + P beta into Q's storage, then P = orth(W)
    rows_times(v, v.Q, v.R, v.P, r, H, s, lo, hi);
    int rank = 0;
    const bool ok = coop_orth(v, v.Q, lo, hi, rank);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        int go = iter + 1 < max_iter;
        if (!ok) {
            go = 0;
            if (!*(volatile int *)&st->err) st->status = LS_BREAKDOWN;
        } else if (rank == 0) {
            go = 0;                                    // nothing left to search: confirm
        }
        set_cond(st, h_inner, go ? 1u : 0u);
    }
}

// After the loop: the true residual (residual GEMVs, ||R_j||^2 in sm->r2);
// accept, stop, or restart from it with P = orth(R).
__global__ void __launch_bounds__(BK) bcgd_check_kernel(BcgVecs v, cudaGraphConditionalHandle h_outer,
                                                        cudaGraphConditionalHandle h_inner) {
    __shared__ int restart_s;
    State *st = v.st;
    BcgSmall *sm = v.sm;
    count_launch(st);
    const int s = v.s;
    if (threadIdx.x == 0) {
        bool pass = true, nan = false;
        for (int j = 0; j < s; j++) {
            const double r2 = *(volatile double *)&sm->r2[j];
            nan = nan || !isfinite(r2);
            pass = pass && sqrt(r2) <= v.st->rtol * sm->bn[j];
        }
        int restart = 0;
        if (*(volatile int *)&st->err || nan) {
            if (nan) set_err(st, ERRB_NAN);
        } else if (*(volatile int *)&st->status == LS_BREAKDOWN) {
        } else if (pass) {
            if (blockIdx.x == 0) st->status = LS_OK;
        } else if (*(volatile int *)&st->iter >= st->max_iter) {
            if (blockIdx.x == 0) st->status = LS_NOT_CONVERGED;
        } else {
            restart = 1;
        }
        restart_s = restart;
    }
    __syncthreads();
    if (!restart_s) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            set_cond(st, h_outer, 0u);
            set_cond(st, h_inner, 0u);
        }
        return;
    }
    long long lo, hi;
    block_range(v.n, blockIdx.x, gridDim.x, lo, hi);
    int rank = 0;
    const bool ok = coop_orth(v, v.R, lo, hi, rank);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        int go = 1;
        if (!ok) {
            go = 0;
            if (!*(volatile int *)&st->err) st->status = LS_BREAKDOWN;
        } else if (rank == 0) {
            go = 0;
            st->status = LS_BREAKDOWN;                  // not converged and nothing left to search
        }
        st->cycles++;
        set_cond(st, h_inner, go ? 1u : 0u);
        set_cond(st, h_outer, go ? 1u : 0u);
    }
}

BcgKernels bcg_kernels() {
    BcgKernels K{};
    K.init = reinterpret_cast<void *>(&bcg_init_kernel);
    K.step = reinterpret_cast<void *>(&bcg_step_kernel);
    K.check = reinterpret_cast<void *>(&bcg_check_kernel);
    K.dinit = reinterpret_cast<void *>(&bcgd_init_kernel);
    K.dstep = reinterpret_cast<void *>(&bcgd_step_kernel);
    K.dcheck = reinterpret_cast<void *>(&bcgd_check_kernel);
    K.block = BK;
    return K;
}

}  // namespace lsi
