// ls_gemv.cuh -- what the matrix-vector products share (k_gemv.cu, k_symv.cu): the
// warp reduction of row sums, the fused epilogues and the solver scalars that
// the last CTA forms.
#pragma once

#include "ls_device.cuh"
#include "ls_ds.cuh"
#include "ls_internal.h"

namespace lsi {

// a + b of two partial sums; SETTLED: of pairs, settled (ls_ds.cuh).  Pairs that stand for
// FP32 sums are left unsettled, so that hi is what FP32 additions alone would give
// (an infinity stays one: pair_value).
template <bool SETTLED, class V>
__device__ __forceinline__ V join(V a, V b) {
    if constexpr (SETTLED) return settled_sum(a, b);
    else return a + b;
}
__device__ __forceinline__ DSV as_sum(float v) { return DSV{v, 0.0f}; }
__device__ __forceinline__ DSV as_sum(DSV v) { return v; }
__device__ __forceinline__ double as_sum(double v) { return v; }
__device__ __forceinline__ double pair_value(double v) { return v; }
__device__ __forceinline__ float pair_value(float v) { return v; }
__device__ __forceinline__ double pair_value(DSV v) { return isfinite(v.h) ? to_double(v) : (double)v.h; }

// Butterfly transpose-reduction of RW per-lane row accumulators over the warp:
// each round a lane keeps half of its rows and adds the partner's copy of
// them, so RW - 1 + (5 - log2 RW) additions replace RW full reductions.
// Afterwards lane l holds the warp total of row (l >> (5 - log2 RW)).
template <int N, int OFF, bool SETTLED, class V, int RW>
__device__ __forceinline__ void butterfly(V (&acc)[RW], int lane) {
    if constexpr (OFF >= 1) {
        if constexpr (N > 1) {
            constexpr int H = N / 2;
            const bool upper = (lane & OFF) != 0;
#pragma unroll
            for (int i = 0; i < H; i++) {
                const V send = upper ? acc[i] : acc[i + H];
                const V keep = upper ? acc[i + H] : acc[i];
                acc[i] = join<SETTLED>(keep, shfl_xor_v(send, OFF));
            }
            butterfly<H, OFF / 2, SETTLED>(acc, lane);
        } else {
            acc[0] = join<SETTLED>(acc[0], shfl_xor_v(acc[0], OFF));
            butterfly<1, OFF / 2, SETTLED>(acc, lane);
        }
    }
}

template <int RW>
__host__ __device__ constexpr int log2i() { return RW <= 1 ? 0 : 1 + log2i<RW / 2>(); }

// ---- epilogue for one finished row ---------------------------------------------------
// V: the vectors' type
template <class V>
__device__ __forceinline__ double epilogue(const GemvArgs &a, int row, V s) {
    V *y = static_cast<V *>(a.y);
    switch (a.epi) {
        case EPI_STORE:
            y[row] = s;
            return 0.0;
        case EPI_DOT:
            y[row] = s;
            return (double)(static_cast<const V *>(a.z)[row] * s);
        case EPI_RESID: {
            V r = (V)(a.b[row] - (double)s);
            y[row] = r;
            return (double)r * (double)r;
        }
        case EPI_JACOBI: {   // y is the next iterate; x and z are read at this row
            const double r = a.b[row] - (double)s;
            y[row] = (V)((double)static_cast<const V *>(a.x)[row] + static_cast<const double *>(a.z)[row] * r);
            return r * r;
        }
        default:  // EPI_NRM
            y[row] = s;
            return (double)s * (double)s;
    }
}

__device__ __forceinline__ void run_finaliser(const GemvArgs &a, double dot) {
    State *st = a.st;
    if (a.dot_out) *a.dot_out = dot;
    switch (a.fin) {
        case FIN_CG_ALPHA:
            st->pq = dot;
            if (!(dot > 0.0)) {
                st->status = LS_BREAKDOWN;
                st->alpha = 0.0;
            } else {
                st->alpha = st->rho / dot;
            }
            break;
        case FIN_TRUE_RES:
            st->true_rnorm = sqrt(dot);
            break;
        case FIN_WNORM0:
            st->wnorm0 = dot;
            break;
        case FIN_INNER_ALPHA:
            st->in_pq = dot;
            if (!(dot > 0.0)) {
                st->in_stop = 2;    // breakdown of the inner solve: keep the iterate
                st->in_alpha = 0.0;
            } else {
                st->in_alpha = st->in_rho / dot;
            }
            break;
        case FIN_FCG_D:
            st->pq = dot;
            break;
        case FIN_BS_ALPHA:
            st->pq = dot;
            if (dot == 0.0 || !isfinite(dot)) {
                st->status = LS_BREAKDOWN;
                st->alpha = 0.0;
            } else {
                st->alpha = st->rho / dot;
            }
            break;
        case FIN_JACOBI: {
            // the residual of the iterate that was just multiplied; the next
            // iterate is already in y, taken (or not) by the next kernel
            const double rn = sqrt(dot);
            st->rnorm = rn;
            st->true_rnorm = rn;
            int stop = 1;
            if (st->status == LS_BREAKDOWN) {
                // zero diagonal entry: this product only measured x
            } else {
                st->iter++;
                if (!isfinite(dot)) set_err(st, ERRB_NAN);
                else if (rn <= st->tol_abs) st->status = LS_OK;
                else if (st->iter >= st->max_iter) st->status = LS_NOT_CONVERGED;
                else stop = 0;
            }
            st->skip = stop;
            break;
        }
        default:
            st->dot = dot;
            break;
    }
}

}  // namespace lsi
