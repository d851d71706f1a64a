// k_lu.cu -- the paper's direct method: LU factorization with partial
// pivoting (right-looking Gaussian elimination), FP64, and the solve.
//
// The paper's right-looking LU: at step k take the row v >= k with the
// largest |a_vk| (the first one on ties), swap rows k and v, divide the
// sub-column by the pivot and subtract the rank-1 update from the trailing
// block.  The right-hand side rides along as column n of the working matrix
// W = [A | b], so the forward substitution L y = P b happens during the
// elimination (y in column n), and U x = y is solved afterwards.
//
// The elimination runs as the paper's block LU factorization (Figures 1-2,
// equations (1)-(4)) with panels of LU_NB = 32 columns, and stays the same
// elimination element by element: every a_ij receives a_ij - l_it u_tj for
// t = 0, 1, ... in order, as a rounded product and a rounded difference.
// Per panel:
// lu_factor_kernel (cooperative, over the panel's steps, its columns only):
//   every CTA owns rows of the panel; per step the CTAs exchange their best
//   pivot candidates (value, row, and that row's entries), pick the same one (a
//   total order) and each divides and updates its rows: l = w_ik / w_kk (IEEE
//   division), w_ij = w_ij - l * w_kj as a separate multiply and subtract (no
//   fused multiply-add), so every element is bit for bit what the same
//   elimination gives in plain FP64 arithmetic.
// lu_laswp_kernel: the panel's row swaps on every other column (a thread a
//   column, the swaps in step order).
// lu_u12_kernel: the panel's pivot rows right of the panel (the paper's
//   triangular solve for U01): the panel's updates t = k0 .. in order, four
//   lanes a column, each holding 8 of the 32 values in registers.
// lu_trail_kernel: the block below and right of the panel, 32 x 32 tiles:
//   each element takes the panel's 32 updates in order from the multipliers
//   and pivot rows staged in shared memory, the product on the integer pipes and
//   the difference on the FP64 pipe (ls_rank.cuh).  This is where the time
//   goes; A crosses DRAM once per panel instead of once per step.
// lu_backsolve_kernel (cooperative): U x = y by blocks of 64 rows from the
//   bottom: CTA 0 solves the diagonal block (one warp, column oriented),
//   then every CTA subtracts the block's contribution from the rows above
//   it (a warp a row).  Two grid barriers per block.
//
// Work: n^3 / 3 updates, a rounded product and a rounded difference each; traffic about 16 n^3 / (3 LU_NB) bytes.
#include <cuda_runtime.h>

#include "ls_device.cuh"
#include "ls_internal.h"
#include "ls_rank.cuh"

namespace lsi {

namespace {

constexpr int LT = 512;            // threads per CTA (16 warps: enough loads in flight)
constexpr int U12_T = 128;         // threads per CTA of lu_u12_kernel (32 columns)
constexpr int LU_NB = 32;          // panel width
constexpr int LW = LT / 32;        // warps per CTA
constexpr int FT = 256, FW = FT / 32;   // threads and warps of a panel CTA
constexpr int SLOTS = 5;           // candidates a lane fetches at a time (152 CTAs)
constexpr int LB = BACK_B;         // rows per back-substitution block
static_assert(LU_NB == RANK_NB, "panel width");

// A pivot candidate: |a| as its bit pattern, which orders as the value does
// (-1 for NaN and for no candidate at all), its row, and the place in its CTA.
// Integer comparisons: one of doubles takes 64 cycles of a scheduler's FP64
// unit, and a step makes dozens (473 -> 421 ms for the whole solve at n = 8192).
struct Cand {
    long long v;
    int i, r;
};
__device__ __forceinline__ Cand make_cand(double x, int i, int r) {
    const long long m = __double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll;
    return Cand{m > 0x7FF0000000000000ll ? -1ll : m, i, r};
}
__device__ __forceinline__ Cand no_cand(int n) { return Cand{-1, n, -1}; }

// The better of two pivot candidates: the larger |a|, the first row on ties.  A
// total order, so the order of a reduction does not change its result.
__device__ __forceinline__ Cand better(Cand a, Cand b) {
    const bool take = b.v > a.v || (b.v == a.v && b.i < a.i);
    return Cand{take ? b.v : a.v, take ? b.i : a.i, take ? b.r : a.r};
}
__device__ __forceinline__ Cand warp_better(Cand c) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        c = better(c, Cand{__shfl_xor_sync(0xffffffffu, c.v, o), __shfl_xor_sync(0xffffffffu, c.i, o),
                           __shfl_xor_sync(0xffffffffu, c.r, o)});
    return c;
}

// What the CTAs tell each other travels as 16-byte words: a value, an index and
// the step + 1.
__device__ __forceinline__ void st_word(LuWord *p, long long v, int i, unsigned seq) {
    st_word128(p, (unsigned long long)v, ((unsigned long long)seq << 32) | (unsigned)i);
}
__device__ __forceinline__ unsigned ld_word(const LuWord *p, long long &v, int &i) {
    unsigned long long lo, hi;
    ld_word128(p, lo, hi);
    v = (long long)lo;
    i = (int)(unsigned)hi;
    return (unsigned)(hi >> 32);
}
// Waits for the word of step seq; false after the library's limit.
__device__ __forceinline__ bool wait_word(const LuWord *p, unsigned seq, long long &v, int &i) {
    if (ld_word(p, v, i) == seq) return true;
    const unsigned long long t0 = gtimer();
    while (ld_word(p, v, i) != seq)
        if (gtimer() - t0 > WAIT_LIMIT_NS) return false;
    return true;
}

}  // namespace

// The panel's steps k0 .. k1 - 1 on its own columns.  A CTA owns `R` rows of the
// panel for all of its steps, in shared memory (or, when they do not fit, in a
// buffer in global memory), so a row crosses HBM twice a panel.  Rows stay where
// they are and only their positions change with the swaps; at the end each
// row is written to its position.
//
// A step is one exchange, made by warp 0: it publishes the CTA's best candidate and that
// row's entries, waits for every CTA's candidate, and fetches the winner's
// row.  Then, a thread a row: the swap of positions, l_i = w_ik / w_kk, the
// update of column k + 1 and the next candidate; the columns right of it are updated by
// the other warps while warp 0 makes the next exchange (which finishes the
// candidate's row itself).  The words are double buffered by the parity of k: a
// CTA writes step k + 2's only after it has seen every CTA's step k + 1, which
// each publishes after it has read step k's.
//
// What bounds it is the chain of a step: the exchange (two L2 round trips), a division,
// an update and two barriers of the CTA.  Two barriers of the grid and all rows read
// from L2 in every step took 15 us a step at n = 8192; whole solve 477 -> 393 ms,
// n = 1500 21.8 -> 9.4 ms.
template <bool SMEM>
__global__ void __launch_bounds__(FT, 1) lu_factor_kernel(LuArgs a, int k0, int k1, int R) {
    extern __shared__ __align__(16) double sm[];
    __shared__ Cand red[FW];
    __shared__ double prow_s[2][LU_NB];
    __shared__ int v_s, ok_s;                    // the pivot's position (-1: no comparable candidate); no timeout
    State *st = a.st;
    count_launch(st);
    if (*(volatile int *)&st->status == LS_BREAKDOWN) return;
    constexpr int P = SMEM ? LU_NB + 1 : LU_NB;
    const int n = a.n, nb = k1 - k0, G = gridDim.x, cta = blockIdx.x;
    const long long ld = a.ld;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int first = k0 + cta * R, mine = max(0, min(R, n - first));
    int *pos = reinterpret_cast<int *>(sm);                           // [R] current position of each row
    double *w = SMEM ? sm + (R + 1) / 2 : a.rowbuf + (size_t)cta * R * LU_NB;
    for (int e = threadIdx.x; e < mine * LU_NB; e += FT) {
        const int r = e / LU_NB, t = e % LU_NB;
        w[r * P + t] = t < nb ? a.W[(long long)(first + r) * ld + k0 + t] : 0.0;
    }
    for (int r = threadIdx.x; r < mine; r += FT) pos[r] = first + r;
    if (threadIdx.x == 0) ok_s = 1;
    __syncthreads();
    Cand best = no_cand(n);
    for (int r = threadIdx.x; r < mine; r += FT) best = better(best, make_cand(w[r * P], pos[r], r));
    best = warp_better(best);
    if (lane == 0) red[warp] = best;
    __syncthreads();

    for (int k = k0; k < k1; k++) {
        const int t = k - k0, par = k & 1;
        const unsigned seq = (unsigned)k + 1;
        LuWord *slots = a.slots + (size_t)par * G;
        LuWord *rows = a.xrows + (size_t)par * (G + 1) * LU_NB;
        double *prow = prow_s[par];
        const double *last = prow_s[par ^ 1];    // step k - 1's pivot row
        Cand mycand = red[0];
#pragma unroll
        for (int i = 1; i < FW; i++) mycand = better(mycand, red[i]);
        if (mycand.v < 0) mycand.r = -1;         // no row is left out below
        if (warp == 0) {
            // ---- publish the candidate, its row finished with step k - 1
            if (mycand.v >= 0) {
                double *wr = w + (size_t)mycand.r * P;
                double x = wr[lane];
                if (t > 0 && lane > t && lane < nb) {
                    x = __dsub_rn(x, __dmul_rn(wr[t - 1], last[lane]));
                    wr[lane] = x;
                }
                st_word(&rows[(size_t)cta * LU_NB + lane], __double_as_longlong(x), 0, seq);
            }
            if (lane == 0) st_word(&slots[cta], mycand.v, mycand.i, seq);
            // ---- everybody's candidates; the winner's row
            Cand c = no_cand(n);
            bool ok = true;
            for (int b0 = 0; b0 < G && ok; b0 += 32 * SLOTS) {
                // a lane's words all requested before the first is looked at
                Cand o[SLOTS];
                unsigned got[SLOTS];
#pragma unroll
                for (int i = 0; i < SLOTS; i++) {
                    o[i] = no_cand(n);
                    got[i] = seq;
                    const int b = b0 + 32 * i + lane;
                    if (b < G) got[i] = ld_word(&slots[b], o[i].v, o[i].i);
                }
#pragma unroll
                for (int i = 0; i < SLOTS; i++) {
                    const int b = b0 + 32 * i + lane;
                    if (got[i] != seq) ok = wait_word(&slots[b], seq, o[i].v, o[i].i) && ok;
                    o[i].r = b;
                    c = better(c, o[i]);
                }
            }
            c = warp_better(c);
            ok = __all_sync(0xffffffffu, ok);
            if (ok && c.v >= 0) {
                long long x;
                int unused;
                ok = __all_sync(0xffffffffu, wait_word(&rows[(size_t)c.r * LU_NB + lane], seq, x, unused));
                prow[lane] = __longlong_as_double(x);
            }
            if (lane == 0) {
                v_s = c.v >= 0 ? c.i : -1;
                if (!ok) {
                    set_err(st, ERRB_TIMEOUT);
                    ok_s = 0;
                }
            }
        } else if (t > 0) {
            // ---- step k - 1 on the columns right of k
            const int nc = nb - 1 - t;
            for (int e = threadIdx.x - 32; e < nc * mine; e += FT - 32) {
                const int r = e / nc, j = t + 1 + e % nc;
                if (r != mycand.r && pos[r] > k - 1)
                    w[r * P + j] = __dsub_rn(w[r * P + j], __dmul_rn(w[r * P + t - 1], last[j]));
            }
        }
        __syncthreads();
        if (!ok_s) return;
        int v = v_s;
        if (v < 0) {
            // no comparable candidate (all NaN): row k stays the pivot, as the sequential
            // scan that starts from it would leave it; its owner publishes it now
            v = k;
            if (warp == 0) {
                for (int r = 0; r < mine; r++)
                    if (pos[r] == k)
                        st_word(&rows[(size_t)G * LU_NB + lane], __double_as_longlong(w[r * P + lane]), 0, seq);
                long long x;
                int unused;
                const bool ok = __all_sync(0xffffffffu, wait_word(&rows[(size_t)G * LU_NB + lane], seq, x, unused));
                prow[lane] = __longlong_as_double(x);
                if (lane == 0 && !ok) {
                    set_err(st, ERRB_TIMEOUT);
                    ok_s = 0;
                }
            }
            __syncthreads();
            if (!ok_s) return;
        }
        if (cta == 0 && threadIdx.x == 0) a.ipiv[k] = v;
        const double piv = prow[t];
        if ((__double_as_longlong(piv) << 1) == 0) {   // a zero pivot, the same in every CTA
            if (cta == 0 && threadIdx.x == 0) st->status = LS_BREAKDOWN;
            return;
        }
        // ---- a thread a row: the swap (the row at position k moves to v, the pivot row to k),
        // the multiplier, column k + 1, the next candidate
        best = no_cand(n);
        for (int r = threadIdx.x; r < mine; r += FT) {
            int p = pos[r];
            if (p == k) p = v;
            else if (p == v) p = k;
            pos[r] = p;
            if (p > k) {
                const double l = w[r * P + t] / piv;
                w[r * P + t] = l;
                if (t + 1 < nb) {
                    const double x = __dsub_rn(w[r * P + t + 1], __dmul_rn(l, prow[t + 1]));
                    w[r * P + t + 1] = x;
                    best = better(best, make_cand(x, p, r));
                }
            }
        }
        best = warp_better(best);
        if (lane == 0) red[warp] = best;
        __syncthreads();
    }
    // every CTA has loaded its rows (it took part in an exchange), so they can be overwritten
    for (int e = threadIdx.x; e < mine * LU_NB; e += FT) {
        const int r = e / LU_NB, t = e % LU_NB;
        if (t < nb) a.W[(long long)pos[r] * ld + k0 + t] = w[r * P + t];
    }
}

// The panel's swaps (steps k0 .. k0 + nb - 1) on the columns outside it.
__global__ void __launch_bounds__(256) lu_laswp_kernel(LuArgs a, int k0, int nb) {
    State *st = a.st;
    count_launch(st);
    if (*(volatile int *)&st->status == LS_BREAKDOWN) return;
    const int n = a.n;
    const long long ld = a.ld;
    double *W = a.W;
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c <= n; c += (long long)gridDim.x * blockDim.x) {
        if (c >= k0 && c < k0 + nb) continue;
        for (int t = k0; t < k0 + nb; t++) {
            const int v = a.ipiv[t];
            if (v != t) {
                const double x = W[(long long)t * ld + c];
                W[(long long)t * ld + c] = W[(long long)v * ld + c];
                W[(long long)v * ld + c] = x;
            }
        }
    }
}

// The pivot rows k0 .. k0 + nb - 1 right of the panel: u_rj -= l_rt u_tj for
// t = k0 .. r - 1 in order.  Four lanes a column (lane q of the quad holds
// rows q, q + 4, ...; the owner of row t hands u_tj to the others by a
// shuffle once it is final), so there are enough warps to keep the FP64
// pipes of every SM busy.
__global__ void __launch_bounds__(U12_T) lu_u12_kernel(LuArgs a, int k0, int nb) {
    __shared__ double Lp[LU_NB][LU_NB + 1];   // the panel's multipliers l_rt, zero past nb
    State *st = a.st;
    count_launch(st);
    if (*(volatile int *)&st->status == LS_BREAKDOWN) return;
    const int n = a.n;
    const long long ld = a.ld;
    double *W = a.W;
    for (int e = threadIdx.x; e < LU_NB * LU_NB; e += blockDim.x) {
        const int r = e / LU_NB, t = e % LU_NB;
        Lp[r][t] = (r < nb && t < r) ? W[(long long)(k0 + r) * ld + k0 + t] : 0.0;
    }
    __syncthreads();
    const int q = threadIdx.x & 3, lane = threadIdx.x & 31;
    const long long ncols = (long long)n + 1 - (k0 + nb);
    const int cpb = U12_T / 4;   // columns a CTA takes at a time
    // the loop bound is the same for the whole CTA, so every lane reaches the shuffles
    for (long long c0 = (long long)blockIdx.x * cpb; c0 < ncols; c0 += (long long)gridDim.x * cpb) {
        const long long jj = c0 + threadIdx.x / 4;
        const bool on = jj < ncols;
        const long long j = k0 + nb + jj;
        // rows past the panel's nb (a short last panel) stay zero and are not stored
        double u[LU_NB / 4];
#pragma unroll
        for (int x = 0; x < LU_NB / 4; x++) {
            const int r = q + 4 * x;
            u[x] = (on && r < nb) ? W[(long long)(k0 + r) * ld + j] : 0.0;
        }
#pragma unroll
        for (int t = 0; t < LU_NB - 1; t++) {
            const double ut = __shfl_sync(0xffffffffu, u[t / 4], (lane & ~3) | (t & 3));
#pragma unroll
            for (int x = 0; x < LU_NB / 4; x++)
                if (q + 4 * x > t) u[x] = __dsub_rn(u[x], __dmul_rn(Lp[q + 4 * x][t], ut));
        }
#pragma unroll
        for (int x = 0; x < LU_NB / 4; x++) {
            const int r = q + 4 * x;
            if (on && r < nb) W[(long long)(k0 + r) * ld + j] = u[x];
        }
    }
}

// The block below and right of the panel (rows k0 + LU_NB .. n - 1, columns
// k0 + LU_NB .. n): a_ij -= l_it u_tj for the panel's steps t in order.
__global__ void __launch_bounds__(RANK_T, 4) lu_trail_kernel(LuArgs a, int k0) {
    constexpr int RT = RANK_R, TT = RANK_TT, PITCH = RANK_PITCH;
    __shared__ Op53 Ls[LU_NB * PITCH], Us[LU_NB * PITCH];
    State *st = a.st;
    count_launch(st);
    if (*(volatile int *)&st->status == LS_BREAKDOWN) return;
    const int n = a.n;
    const long long ld = a.ld;
    double *W = a.W;
    const int r0 = k0 + LU_NB + blockIdx.y * TT, c0 = k0 + LU_NB + blockIdx.x * TT;
    // rows and columns past the block are staged as ones and not stored
    RankRange range;
    for (int e = threadIdx.x; e < TT * LU_NB; e += RANK_T) {
        const int r = e / LU_NB, t = e % LU_NB;
        const Op53 l = op53_a(r0 + r < n ? W[(long long)(r0 + r) * ld + k0 + t] : 1.0);
        const int tt = e / TT, c = e % TT;
        const Op53 u = op53_b(c0 + c <= n ? W[(long long)(k0 + tt) * ld + c0 + c] : 1.0);
        range.a(l);
        range.b(u);
        Ls[t * PITCH + r] = l;
        Us[tt * PITCH + c] = u;
    }
    const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
    double acc[RT][RT];
#pragma unroll
    for (int p = 0; p < RT; p++)
#pragma unroll
        for (int q = 0; q < RT; q++) {
            const int r = r0 + ty + 16 * p, c = c0 + tx + 16 * q;
            acc[p][q] = (r < n && c <= n) ? W[(long long)r * ld + c] : 0.0;
        }
    rank_tile(acc, Ls, Us, LU_NB, range.all_in_range(), ty, tx);
#pragma unroll
    for (int p = 0; p < RT; p++)
#pragma unroll
        for (int q = 0; q < RT; q++) {
            const int r = r0 + ty + 16 * p, c = c0 + tx + 16 * q;
            if (r < n && c <= n) W[(long long)r * ld + c] = acc[p][q];
        }
}

__global__ void __launch_bounds__(LT, 1) lu_backsolve_kernel(LuArgs a) {
    __shared__ double s[LB], xs[LB], T[LB][LB + 1];
    State *st = a.st;
    count_launch(st);
    const int n = a.n;
    const long long ld = a.ld;
    double *W = a.W;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gw = blockIdx.x * LW + warp, nw = gridDim.x * LW;
    if (*(volatile int *)&st->status == LS_BREAKDOWN) return;
#define Y(i) W[(long long)(i) * ld + n]   // y = L^-1 P b, column n of the working matrix
    for (int r1 = n; r1 > 0; r1 -= LB) {
        const int r0 = r1 > LB ? r1 - LB : 0, nb = r1 - r0;
        if (blockIdx.x == 0) {   // the diagonal block
            for (int e = threadIdx.x; e < LB * LB; e += LT) {
                const int r = e / LB, c = e % LB;
                T[r][c] = r < nb && c < nb ? W[(long long)(r0 + r) * ld + r0 + c] : 0.0;
            }
            for (int r = threadIdx.x; r < nb; r += LT) s[r] = __ldcg(&Y(r0 + r));
            __syncthreads();
            if (warp == 0) back_solve_block(nb, T, s, xs);
            __syncthreads();
            for (int r = threadIdx.x; r < nb; r += LT) a.x[r0 + r] = xs[r];
        }
        if (!grid_sync(a.bar, st)) return;
        // rows above the block: y_i -= sum_{j in block} u_ij x_j (a warp a row)
        for (int i = gw; i < r0; i += nw) {
            const double *wi = W + (long long)i * ld + r0;
            double acc = 0.0;
            for (int j = lane; j < nb; j += 32) acc += wi[j] * __ldcg(&a.x[r0 + j]);
            acc = warp_sum(acc);
            if (lane == 0) Y(i) = __ldcg(&Y(i)) - acc;
        }
        if (!grid_sync(a.bar, st)) return;
    }
#undef Y
}

LuKernels lu_kernels() {
    LuKernels K{};
    K.factor = reinterpret_cast<void *>(&lu_factor_kernel<true>);
    K.factor_global = reinterpret_cast<void *>(&lu_factor_kernel<false>);
    K.backsolve = reinterpret_cast<void *>(&lu_backsolve_kernel);
    K.laswp = reinterpret_cast<void *>(&lu_laswp_kernel);
    K.u12 = reinterpret_cast<void *>(&lu_u12_kernel);
    K.trail = reinterpret_cast<void *>(&lu_trail_kernel);
    set_smem_limit(K.factor, LU_FACTOR_SMEM_MAX);
    K.nb = LU_NB;
    K.tile = RANK_TT;
    K.u12_block = U12_T;
    K.block = LT;
    K.factor_block = FT;
    return K;
}

}  // namespace lsi
