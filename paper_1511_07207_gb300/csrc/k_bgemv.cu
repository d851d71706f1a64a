// k_bgemv.cu -- Q = A P for an n x s block P (the block product of block CG),
// A read once as its FP32 pair hi + lo, double-single arithmetic.
//
// One CTA per SM: a producer lane streams, for each of the CTA's 16-row x
// 256-column tiles, the A tile (hi and lo, the solvers' 2-D TMA map) and the matching 256-row chunk of P (pre-split into FP32 pairs,
// column panels padded with zeros to a multiple of 256, one 1-D bulk copy
// per column and part) through a ring of shared-memory stages (mbarrier
// full/empty).  Consumer warps: for S <= 8 sixteen warps, warp w owning row
// w of the 16-row block (enough warps to hide the latency of the
// double-single chains); for S = 16 eight warps of two rows each (w and
// w + 8: registers); lane g takes the 4-column chunks g and g + 32 of each
// tile.  A thread accumulates all S columns of P for its rows in
// double-single (two-sum of the high parts, the low parts and rounding
// errors summed apart, as the GEMV does), and the 32 lanes of a row add
// their sums by shuffles at the end of the row block.  The (row block, column
// tile) sequence is cut into equal pieces, one per CTA (whole row blocks leave up to
// a fifth of the SMs idle in the last turn: n = 8192 has 512 of them), and the last of
// the CTAs that share a row block adds their sums in CTA order, so results are
// deterministic; where meeting costs more than that, and for S = 16, a CTA takes whole
// row blocks (gemv_split.h).  Two kernels: with both forms in one, the whole row
// blocks took up to half as long again.  Work per element of A is 12 FP32 operations per column of
// P: compute-bound for S >= 4 (HBM-bound below).
#include <cuda_runtime.h>

#include "gemv_split.h"
#include "ls_device.cuh"
#include "ls_internal.h"
#include "split_pair.h"

namespace lsi {

namespace {

constexpr int BG_TR = 16, BG_TC = 256;
constexpr int BG_A_B = BG_TR * BG_TC * 4;   // one part of an A tile (16 KB)

struct F2 {
    float h, l;
};

// acc += (mh + ml)(vh + vl), terms below ml*vl kept, low part unnormalised
__device__ __forceinline__ void f2_mac(F2 &acc, float mh, float ml, float vh, float vl) {
    const float p = __fmul_rn(mh, vh);
    float e = __fmaf_rn(mh, vh, -p);
    e = __fmaf_rn(mh, vl, e);
    e = __fmaf_rn(ml, vh, e);
    const float s = __fadd_rn(acc.h, p);
    const float bb = __fsub_rn(s, acc.h);
    const float err = __fadd_rn(__fsub_rn(acc.h, __fsub_rn(s, bb)), __fsub_rn(p, bb));
    acc.h = s;
    acc.l = __fadd_rn(acc.l, __fadd_rn(e, err));
}

// a + b with Knuth's two-sum on the high parts, renormalised
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    const float s = __fadd_rn(a.h, b.h);
    const float bb = __fsub_rn(s, a.h);
    const float err = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, bb)), __fsub_rn(b.h, bb));
    const float l = __fadd_rn(__fadd_rn(a.l, b.l), err);
    const float h = __fadd_rn(s, l);
    return {h, __fsub_rn(l, __fsub_rn(h, s))};
}

// Rows of a 16-row block per consumer warp: one for S <= 8 (sixteen warps,
// to hide the latency of the double-single chains), two for S = 16 (eight
// warps: registers).  Plus the producer warp.
template <int S>
__host__ __device__ constexpr int bg_rows_per_warp() {
    return S <= 8 ? 1 : 2;
}
// Accumulators a column: one row per warp (S <= 8) keeps the two column chunks apart (two
// independent chains per column of P), added at the end of the row block; two rows have one each.
constexpr int BG_ACCS = 2;
template <int S>
__host__ __device__ constexpr int bg_consumers() {
    return 32 * 16 / bg_rows_per_warp<S>();
}
template <int S>
__host__ __device__ constexpr int bg_threads() {
    return bg_consumers<S>() + 32;
}

template <int S>
__host__ __device__ constexpr int stages() {
    return S >= 16 ? 3 : 4;
}
__device__ __forceinline__ long long bg_start(long long T, int c, int G) { return T * c / G; }
__device__ __forceinline__ int bg_owner(long long t, long long T, int G) {
    return (int)(((long long)G * (t + 1) + T - 1) / T) - 1;
}

template <int S>
__host__ __device__ constexpr size_t stage_bytes() {
    return (size_t)2 * BG_A_B + (size_t)2 * S * BG_TC * 4;
}

// A warp's share of one 16 x 256 tile in a ring stage: rows w, w + WS, ..., lane g's 4-column chunks.
template <int S>
__device__ __forceinline__ void bg_tile(F2 (&acc)[BG_ACCS][S], const unsigned char *base, int w, int g) {
    constexpr int RPW = bg_rows_per_warp<S>(), WS = 16 / RPW, NA = BG_ACCS / RPW;
    const float *Ah = reinterpret_cast<const float *>(base);
    const float *Al = reinterpret_cast<const float *>(base + BG_A_B);
    const float *Xh = reinterpret_cast<const float *>(base + 2 * BG_A_B);
    const float *Xl = Xh + S * BG_TC;
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const int c0 = (k * 32 + g) * 4;
        float4 ah[RPW], al[RPW];
#pragma unroll
        for (int q = 0; q < RPW; q++) {
            ah[q] = *reinterpret_cast<const float4 *>(Ah + (w + WS * q) * BG_TC + c0);
            al[q] = *reinterpret_cast<const float4 *>(Al + (w + WS * q) * BG_TC + c0);
        }
#pragma unroll
        for (int j = 0; j < S; j++) {
            const float4 xh = *reinterpret_cast<const float4 *>(Xh + j * BG_TC + c0);
            const float4 xl = *reinterpret_cast<const float4 *>(Xl + j * BG_TC + c0);
#pragma unroll
            for (int q = 0; q < RPW; q++) {
                F2 &a2 = acc[NA == 2 ? k : q][j];
                f2_mac(a2, ah[q].x, al[q].x, xh.x, xl.x);
                f2_mac(a2, ah[q].y, al[q].y, xh.y, xl.y);
                f2_mac(a2, ah[q].z, al[q].z, xh.z, xl.z);
                f2_mac(a2, ah[q].w, al[q].w, xh.w, xl.w);
            }
        }
    }
}

}  // namespace

// P (column-major n x s, FP64) -> Ph, Pl (column panels of ldp floats, S of
// them; zero past n and for columns >= s).  With kptr set, P starts at
// P + (*kptr) * kstride (a graph node walking the blocks of a basis).
__global__ void bgemv_split_kernel(int n, int s, int S, const double *__restrict__ P, long long ld,
                                   float *__restrict__ Ph, float *__restrict__ Pl, long long ldp, State *st,
                                   const int *kptr, long long kstride) {
    count_launch(st);
    if (kptr) P += (long long)(*kptr) * kstride;
    const long long total = (long long)S * ldp;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int j = (int)(e / ldp);
        const long long c = e % ldp;
        const double v = (j < s && c < n) ? P[(long long)j * ld + c] : 0.0;
        split_pair(v, Ph[e], Pl[e]);
    }
}

// WHOLE: whole row blocks, CTA c: c, c + G, ...; else equal pieces (gemv_split.h).
template <int S, bool WHOLE>
__global__ void __launch_bounds__(bg_threads<S>(), 1) bgemv_kernel(const MatDesc *__restrict__ dA, BgemvArgs a) {
    constexpr int BG_C = bg_consumers<S>();
    constexpr int RPW = bg_rows_per_warp<S>(), WS = 16 / RPW;   // rows per warp, their stride
    constexpr int NST = stages<S>();
    constexpr size_t SB = stage_bytes<S>();
    extern __shared__ __align__(1024) unsigned char bg_dyn[];
    unsigned char *ring =
        reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(bg_dyn) + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t full[NST], empty[NST];
    State *st = a.st;
    count_launch(st);
    const int n = a.n;
    const int RB = (n + BG_TR - 1) / BG_TR, CT = (n + BG_TC - 1) / BG_TC;
    const long long T = (long long)RB * CT;
    const int G = gridDim.x, cta = blockIdx.x;
    const long long t0 = WHOLE ? (long long)cta * CT : bg_start(T, cta, G);
    const int ntiles = WHOLE ? (cta < RB ? (RB - cta + G - 1) / G * CT : 0) : (int)(bg_start(T, cta + 1, G) - t0);
    const int first_rb = WHOLE ? cta : (int)(t0 / CT), rb_step = WHOLE ? G : 1;
    __shared__ int ca_s, cb_s, fin_s;
    if (threadIdx.x == 0) {
        for (int i = 0; i < NST; i++) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], BG_C / 32);
        }
        fence_mbar_init();
    }
    __syncthreads();

    if (threadIdx.x >= BG_C) {
        // ---- producer lane ----
        if ((threadIdx.x & 31) != 0) return;
        const MatDesc &M = *dA;
        tmap_acquire(&M.tmap);
        tmap_acquire(&M.tmap_lo);
        int seq = 0;
        int rb = first_rb, t = (int)(t0 - (long long)rb * CT);
        for (; seq < ntiles; seq++) {
            const int sl = seq % NST;
            if (seq >= NST && !mbar_wait(&empty[sl], ((seq / NST) - 1) & 1)) {
                set_err(st, ERRB_TIMEOUT);
                break;
            }
            unsigned char *dst = ring + (size_t)sl * SB;
            mbar_arrive_expect_tx(&full[sl], (unsigned)SB);
            tma_load_2d(dst, &M.tmap, t * BG_TC, rb * BG_TR, &full[sl]);
            tma_load_2d(dst + BG_A_B, &M.tmap_lo, t * BG_TC, rb * BG_TR, &full[sl]);
            for (int j = 0; j < S; j++) {
                const long long off = (long long)j * a.ldp + (long long)t * BG_TC;
                bulk_load_1d(dst + 2 * BG_A_B + (size_t)j * BG_TC * 4, a.Ph + off, BG_TC * 4, &full[sl]);
                bulk_load_1d(dst + 2 * BG_A_B + (size_t)(S + j) * BG_TC * 4, a.Pl + off, BG_TC * 4, &full[sl]);
            }
            if (++t == CT) {
                t = 0;
                rb += rb_step;
            }
        }
        // no copy may be in flight when the CTA exits
        for (int k = seq > NST ? seq - NST : 0; k < seq; k++)
            if (!mbar_wait(&full[k % NST], (k / NST) & 1)) set_err(st, ERRB_TIMEOUT);
        return;
    }

    // ---- consumers ----
    // warp w: rows w, w + WS, ... of the block (RPW of them); lane g: the
    // 4-column chunks g and g + 32 of each tile
    const int w = threadIdx.x >> 5, g = threadIdx.x & 31;
    constexpr int NA = BG_ACCS / RPW;
    int seq = 0;
    bool ok = true;
    for (int rb = first_rb; seq < ntiles; rb += rb_step) {
        F2 acc[RPW * NA][S];
#pragma unroll
        for (int q = 0; q < RPW * NA; q++)
#pragma unroll
            for (int j = 0; j < S; j++) acc[q][j] = {0.f, 0.f};
        const long long rfirst = (long long)rb * CT;
        const int end = WHOLE ? seq + CT : (int)min((long long)ntiles, rfirst + CT - t0);
        for (; seq < end; seq++) {
            const int sl = seq % NST;
            // on a timeout the warp stops waiting and computing but keeps walking
            // its tiles, so it still meets the others where a row block is shared
            ok = ok && mbar_wait(&full[sl], (seq / NST) & 1);
            if (!__all_sync(0xffffffffu, ok)) {
                set_err(st, ERRB_TIMEOUT);
                ok = false;
            }
            if (ok) bg_tile<S>(acc, ring + (size_t)sl * SB, w, g);
            __syncwarp();
            if (g == 0) mbar_arrive(&empty[sl]);
        }
        // this CTA's share of row block rb
        if constexpr (NA == 2)
#pragma unroll
            for (int j = 0; j < S; j++) acc[0][j] = f2_add(acc[0][j], acc[1][j]);
        // the 32 lanes of a row
#pragma unroll
        for (int q = 0; q < RPW; q++)
#pragma unroll
            for (int j = 0; j < S; j++) {
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    F2 b;
                    b.h = __shfl_xor_sync(0xffffffffu, acc[q][j].h, o);
                    b.l = __shfl_xor_sync(0xffffffffu, acc[q][j].l, o);
                    acc[q][j] = f2_add(acc[q][j], b);
                }
            }
        if (WHOLE || (t0 <= rfirst && rfirst + CT <= t0 + ntiles)) {
            if (g == 0)
#pragma unroll
                for (int q = 0; q < RPW; q++) {
                    const int row = rb * BG_TR + w + WS * q;
                    if (row < n)
#pragma unroll
                        for (int j = 0; j < S; j++)
                            if (j < a.s) a.Q[(long long)j * a.ldq + row] = (double)acc[q][j].h + (double)acc[q][j].l;
                }
        } else if constexpr (!WHOLE) {
            // shared with neighbouring CTAs: publish the partial sums; the last of
            // the sharing CTAs adds them in CTA order
            double *fix = a.scr->fix + (size_t)(2 * blockIdx.x + (rb == first_rb ? 0 : 1)) * BG_TR * S;
            if (g == 0) {
#pragma unroll
                for (int q = 0; q < RPW; q++)
#pragma unroll
                    for (int j = 0; j < S; j++)
                        fix[(w + WS * q) * S + j] = (double)acc[q][j].h + (double)acc[q][j].l;
                __threadfence();
            }
            named_bar(1, BG_C);
            if (threadIdx.x == 0) {
                ca_s = bg_owner(rfirst, T, gridDim.x);
                cb_s = bg_owner(rfirst + CT - 1, T, gridDim.x);
                int ncov = 0;
                for (int c = ca_s; c <= cb_s; c++) ncov += bg_start(T, c, gridDim.x) < bg_start(T, c + 1, gridDim.x);
                fin_s = atomicAdd(&a.scr->bticket[ca_s], 1u) == (unsigned)ncov - 1;
                if (fin_s) atomicExch(&a.scr->bticket[ca_s], 0u);
            }
            named_bar(1, BG_C);
            if (fin_s) {
                __threadfence();
                for (int e = threadIdx.x; e < BG_TR * S; e += BG_C) {
                    const int row = rb * BG_TR + e / S, j = e % S;
                    double sum = 0.0;
                    for (int c = ca_s; c <= cb_s; c++) {
                        const long long a0 = bg_start(T, c, gridDim.x);
                        if (bg_start(T, c + 1, gridDim.x) <= a0) continue;   // empty CTA
                        const int slot = rb == (int)(a0 / CT) ? 0 : 1;
                        sum += __ldcg(&a.scr->fix[(size_t)(2 * c + slot) * BG_TR * S + e]);
                    }
                    if (row < n && j < a.s) a.Q[(long long)j * a.ldq + row] = sum;
                }
            }
        }
    }
}

namespace {
// Sixteen columns keep whole row blocks, by measurement (block GMRES, s = 16: n = 8192
// 40.4 ms a solve with whole blocks, 42.1 with pieces; n = 6000, s = 12 24.7 and 26.5).
template <int S>
void bg_set(BgemvLaunch &L, int n) {
    L.smem = stages<S>() * stage_bytes<S>() + 1024;
    if constexpr (S < 16) {
        if (!bgemv_whole_blocks(bgemv_costs(S), (n + BG_TR - 1) / BG_TR, (n + BG_TC - 1) / BG_TC, L.grid)) {
            L.func = reinterpret_cast<void *>(&bgemv_kernel<S, false>);
            return;
        }
    }
    L.func = reinterpret_cast<void *>(&bgemv_kernel<S, true>);
}
}  // namespace

BgemvLaunch bgemv_plan(int n, int s, int num_sms) {
    BgemvLaunch L{};
    L.split = reinterpret_cast<void *>(&bgemv_split_kernel);
    L.grid = num_sms;
    L.S = s <= 1 ? 1 : s <= 2 ? 2 : s <= 4 ? 4 : s <= 8 ? 8 : 16;
    L.block = L.S <= 8 ? bg_threads<8>() : bg_threads<16>();
    switch (L.S) {
        case 1: bg_set<1>(L, n); break;
        case 2: bg_set<2>(L, n); break;
        case 4: bg_set<4>(L, n); break;
        case 8: bg_set<8>(L, n); break;
        default: bg_set<16>(L, n); break;
    }
    set_smem_limit(L.func, L.smem);
    return L;
}

}  // namespace lsi
