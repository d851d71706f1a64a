// k_symv.cu -- y = A x for an exactly symmetric A, from its lower triangle.
//
// CG's matrices are symmetric, and its product is bound by HBM (k_gemv.cu):
// reading one triangle halves the bytes of a step.  An element a_ij below the
// diagonal is used twice, y_i += a_ij x_j and y_j += a_ij x_i, so the arithmetic
// is that of the full product.  The triangle is packed once per solve
// (sym_pack_kernel), which also compares every a_ij with a_ji bit for bit: a
// matrix that is not exactly symmetric keeps the general product.
//
// Layout: row blocks of TR = 128 rows; row block I holds the column tiles J = 0, 1,
// ... up to its diagonal, each 128 x TC, contiguous in the order the product
// reads them (one bulk copy a tile; FP32 pairs: the hi tile, then the lo tile).  Above
// the diagonal and past n the tiles hold zeros; a diagonal entry is halved (exactly),
// so that using it twice is using it once.
//
// The tile sequence is cut into equal pieces, one per CTA (one CTA per SM):
//  * a producer lane streams the tiles through a shared-memory ring;
//  * eight consumer warps own 16 rows each; a lane holds VEC columns.  Row sums stay
//    in registers over a row block's tiles (the FP32 pair's settled every fourth tile, ls_ds.cuh:
//    up to 430 additions in a row); column sums cover the tile's 128 rows:
//    a warp's 16 in registers, the eight warps' through shared memory
//    (one barrier a tile, two buffers), then one partial vector of the tile in global
//    memory (TC sums for 128 x TC elements: 0.8 % of the pair's bytes);
//  * after a barrier of the grid, y_i = the row sums of its row block (from the CTAs
//    that share it, in order) + the column sums of the tiles below it (in order),
//    then the same epilogues and scalars as the general product.  All orders are
//    fixed, so results are deterministic for a given n.
//
// Bound: HBM above about n = 6000 (4 n^2 bytes of the pair: 6.6 TB/s in the slope from
// n = 4000 to 16384), below it the tile loop (1.3 us a tile and SM, the FP32 pipe 44 %
// busy) and the latency of the barrier and the final sums.  A CG step (product and
// update) at n = 16384 took 317 us with the general product and takes 187; n = 4000
// 48 -> 28, n = 1024 28 -> 19; BF16 inside the flexible CG at n = 32768 331 -> 192 ms
// a solve.  Packing: 0.70 ms at n = 16384, the split of all of A 0.68.  Error against FP64, relative
// root mean square: 9.2e-15 at n = 16384 (2.7e-14 without settling; equal pieces of the general
// product 2.2e-14), 5.0e-15 at n = 1024 (8.2e-15; 6.0e-15), for 1 % of a solve at n = 4000.  Tried and
// no faster: mbarrier hand-over to reducing warps instead of the barrier a tile (192 us
// a step where this form took 191), 16 consumer warps of 8 rows (193), fetching the
// next product's first tiles into L2 during the update (191 to 196).
#include <cuda_bf16.h>

#include "ls_device.cuh"
#include "ls_ds.cuh"
#include "ls_gemv.cuh"
#include "ls_internal.h"
#include "split_pair.h"

namespace lsi {

namespace {

constexpr int SW = 8;                        // consumer warps
constexpr int S_T = (SW + 1) * 32;           // threads: consumers and the producer warp
constexpr int S_RW = 16;                     // rows a warp
constexpr int S_TR = SW * S_RW;              // rows a tile
constexpr int S_CB = 64;                     // rows of y formed at a time

template <int DT>
struct SymCfg;
template <>
struct SymCfg<DT_DS> {
    using T = float;
    using V = DSV;
    using X = double;
    static constexpr int VEC = 2, PARTS = 2, STAGES = 3;
};
template <>
struct SymCfg<DT_BF16> {
    using T = uint16_t;
    using V = float;
    using X = float;
    static constexpr int VEC = 4, PARTS = 1, STAGES = 6;
};
template <>
struct SymCfg<DT_F32> {
    using T = float;
    using V = float;
    using X = float;
    static constexpr int VEC = 2, PARTS = 1, STAGES = 6;
};
template <int DT>
struct SymGeo {
    using C = SymCfg<DT>;
    static constexpr int TC = 32 * C::VEC;
    static constexpr int CPR = S_TR / TC;    // column tiles per 128 columns
    static constexpr int ELEMS = S_TR * TC;
    static constexpr int BYTES = ELEMS * (int)sizeof(typename C::T) * C::PARTS;
    static constexpr int NXW = TC / 32;      // warps that cover a tile's columns, a column a lane
    static constexpr int GROUPS = SW / NXW;
    static constexpr size_t SMEM = (size_t)C::STAGES * BYTES +
                                   ((size_t)2 * SW * TC + 2 * TC + S_TR) * sizeof(typename C::V) +
                                   2 * C::STAGES * sizeof(uint64_t);
    static_assert(S_TR % TC == 0 && GROUPS >= 2, "tile shape");
};

// First tile of row block I, in units of CPR tiles.
__host__ __device__ __forceinline__ long long tri(long long I) { return I * (I + 1) / 2; }
// The row block of tile t / CPR = u: the largest I with tri(I) <= u.
__device__ __forceinline__ int tri_row(long long u) {
    int I = (int)((sqrtf(8.0f * (float)u + 1.0f) - 1.0f) * 0.5f);
    while (tri(I) > u) I--;
    while (tri(I + 1) <= u) I++;
    return I;
}
__device__ __forceinline__ long long piece_start(long long T, int c, int G) { return T * c / G; }
__device__ __forceinline__ int piece_owner(long long t, long long T, int G) {
    return (int)(((long long)G * (t + 1) + T - 1) / T) - 1;
}

__device__ __forceinline__ void sym_consumers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(SW * 32) : "memory"); }

// An entry of x as the operand of the products.
__device__ __forceinline__ void to_operand(double x, DSV &v) { split_pair(x, v.h, v.l); }
__device__ __forceinline__ void to_operand(float x, float &v) { v = x; }
// A partial sum as a double-single one.
__device__ __forceinline__ DSV wide(DSV v) { return v; }
__device__ __forceinline__ DSV wide(float v) { return DSV{v, 0.0f}; }

// row += a . p over the lane's VEC columns and col[v] += a_v xr, for VEC
// consecutive stored elements at `a`.
template <int DT>
__device__ __forceinline__ void both(const typename SymCfg<DT>::T *a, const typename SymCfg<DT>::V (&p)[SymCfg<DT>::VEC],
                                     typename SymCfg<DT>::V xr, typename SymCfg<DT>::V &row,
                                     typename SymCfg<DT>::V (&col)[SymCfg<DT>::VEC]) {
    if constexpr (DT == DT_DS) {
        const float2 h = *reinterpret_cast<const float2 *>(a);
        const float2 l = *reinterpret_cast<const float2 *>(a + SymGeo<DT>::ELEMS);
        ds_fma(h.x, l.x, xr, col[0]);
        ds_fma(h.y, l.y, xr, col[1]);
        ds_fma(h.x, l.x, p[0], row);
        ds_fma(h.y, l.y, p[1], row);
    } else if constexpr (DT == DT_BF16) {
        const uint2 w = *reinterpret_cast<const uint2 *>(a);
        const float e[4] = {__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                            __uint_as_float(w.y & 0xffff0000u)};
#pragma unroll
        for (int v = 0; v < 4; v++) {
            col[v] = fmaf(e[v], xr, col[v]);
            row = fmaf(e[v], p[v], row);
        }
    } else {
        const float2 e = *reinterpret_cast<const float2 *>(a);
        col[0] = fmaf(e.x, xr, col[0]);
        col[1] = fmaf(e.y, xr, col[1]);
        row = fmaf(e.x, p[0], row);
        row = fmaf(e.y, p[1], row);
    }
}

}  // namespace

template <int DT>
__global__ void __launch_bounds__(S_T, 1) symv_kernel(SymMat M, GemvArgs args) {
    using C = SymCfg<DT>;
    using G_ = SymGeo<DT>;
    using T = typename C::T;
    using V = typename C::V;
    using X = typename C::X;
    constexpr int VEC = C::VEC, TC = G_::TC, CPR = G_::CPR, ST = C::STAGES;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    T *ring = reinterpret_cast<T *>(smem_raw);
    V *colbuf = reinterpret_cast<V *>(smem_raw + (size_t)ST * G_::BYTES);      // [2][SW][TC]
    V *xbuf = colbuf + 2 * SW * TC;                                            // [2][TC]
    V *xrow = xbuf + 2 * TC;                                                   // [S_TR]
    uint64_t *full = reinterpret_cast<uint64_t *>(xrow + S_TR), *empty = full + ST;
    DSV (*comb)[SW][S_CB] = reinterpret_cast<DSV (*)[SW][S_CB]>(smem_raw);     // [2], in the ring once it is idle
    __shared__ double dred[S_T / 32];
    __shared__ int abort_s, last_s;
    State *st = args.st;
    count_launch(st);
    if (args.kptr) {   // walk a stored basis: x = column k, y = column k + kyoff
        const long long k = *args.kptr;
        args.x = static_cast<const X *>(args.x) + k * args.kstride;
        args.y = static_cast<X *>(args.y) + (k + args.kyoff) * args.kstride;
    }
    if (args.z_is_x) args.z = args.x;
    const int n = M.n, NI = M.blocks, G = gridDim.x, cta = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long tiles = CPR * tri(NI);
    const long long t0 = piece_start(tiles, cta, G), t1 = piece_start(tiles, cta + 1, G);
    const int nt = (int)(t1 - t0);
    V *pcol = static_cast<V *>(M.pcol), *prow = static_cast<V *>(M.prow);
    if (threadIdx.x == 0) {
        abort_s = 0;
        for (int s = 0; s < ST; s++) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], SW);
        }
        fence_mbar_init();
    }
    __syncthreads();

    if (warp == SW) {
        // ---------------- producer ----------------
        if (lane == 0) {
            int issued = 0;
            for (int i = 0; i < nt; i++) {
                const int s = i % ST;
                if (i >= ST && !mbar_wait(&empty[s], ((i / ST) - 1) & 1)) {
                    set_err(st, ERRB_TIMEOUT);
                    abort_s = 1;
                    break;
                }
                if (*(volatile int *)&abort_s) break;
                mbar_arrive_expect_tx(&full[s], G_::BYTES);
                bulk_load_1d(smem_raw + (size_t)s * G_::BYTES, M.tiles + (size_t)(t0 + i) * G_::BYTES, G_::BYTES, &full[s]);
                issued = i + 1;
            }
            // never leave with copies in flight: wait for the last stages
            for (int i = issued > ST ? issued - ST : 0; i < issued; i++)
                if (!mbar_wait(&full[i % ST], (i / ST) & 1)) set_err(st, ERRB_TIMEOUT);
        }
    } else if (nt > 0) {
        // ---------------- consumers ----------------
        const X *x = static_cast<const X *>(args.x);
        const int xg = warp / G_::NXW, xc = (warp % G_::NXW) * 32 + lane;   // the column a thread serves, and its group
        int I = tri_row(t0 / CPR);
        int J = (int)(t0 - CPR * tri(I));
        for (int e = threadIdx.x; e < S_TR + TC; e += SW * 32) {
            const int i = e < S_TR ? I * S_TR + e : J * TC + e - S_TR;
            to_operand(i < n ? x[i] : X(0), e < S_TR ? xrow[e] : xbuf[e - S_TR]);
        }
        V acc[S_RW];
#pragma unroll
        for (int r = 0; r < S_RW; r++) acc[r] = V{};
        sym_consumers_sync();
        for (int i = 0; i < nt; i++) {
            const int s = i % ST, par = i & 1;
            const bool row_ends = J == CPR * (I + 1) - 1;
            // the next tile's x, asked for before the tile is worked on
            X xn = X(0);
            const bool fetches = xg == (i + G_::GROUPS / 2) % G_::GROUPS && i + 1 < nt;
            if (fetches) {
                const int j = (row_ends ? 0 : J + 1) * TC + xc;
                if (j < n) xn = __ldg(&x[j]);
            }
            V p[VEC], col[VEC];
#pragma unroll
            for (int v = 0; v < VEC; v++) {
                p[v] = xbuf[par * TC + lane * VEC + v];
                col[v] = V{};
            }
            // on a timeout the warp stops waiting and computing but keeps
            // walking the tiles, so it still meets the others at the barriers
            if (!*(volatile int *)&abort_s && !mbar_wait(&full[s], (i / ST) & 1)) {
                set_err(st, ERRB_TIMEOUT);
                abort_s = 1;
            }
            if (!*(volatile int *)&abort_s) {
                const T *tile = ring + (size_t)s * (G_::BYTES / sizeof(T)) + (warp * S_RW) * TC + lane * VEC;
#pragma unroll
                for (int r = 0; r < S_RW; r++) both<DT>(tile + r * TC, p, xrow[warp * S_RW + r], acc[r], col);
                if (DT == DT_DS && (J & 3) == 3) {
#pragma unroll
                    for (int r = 0; r < S_RW; r++) acc[r] = settled(acc[r]);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[s]);
#pragma unroll
            for (int v = 0; v < VEC; v++) colbuf[(par * SW + warp) * TC + lane * VEC + v] = col[v];
            if (fetches) to_operand(xn, xbuf[(par ^ 1) * TC + xc]);
            sym_consumers_sync();
            if (xg == i % G_::GROUPS) {   // one group adds the eight warps' column sums
                V c = colbuf[(par * SW) * TC + xc];
#pragma unroll
                for (int w = 1; w < SW; w++) c = settled_sum(c, colbuf[(par * SW + w) * TC + xc]);
                pcol[(t0 + i) * TC + xc] = c;
            }
            if (row_ends || i == nt - 1) {
                // this CTA's share of row block I
                constexpr int LGR = log2i<S_RW>();
                butterfly<S_RW, 16, true>(acc, lane);
                if ((lane & ((32 >> LGR) - 1)) == 0)
                    prow[(size_t)(cta + I) * S_TR + warp * S_RW + (lane >> (5 - LGR))] = acc[0];
#pragma unroll
                for (int r = 0; r < S_RW; r++) acc[r] = V{};
                if (row_ends && i + 1 < nt) {   // every warp has read xrow: it passed the barrier above
                    if (threadIdx.x < S_TR) {
                        const int ii = (I + 1) * S_TR + threadIdx.x;
                        to_operand(ii < n ? x[ii] : X(0), xrow[threadIdx.x]);
                    }
                    sym_consumers_sync();
                }
            }
            if (row_ends) {
                I++;
                J = 0;
            } else {
                J++;
            }
        }
    }
    if (!grid_sync(M.bar, st)) return;

    // ---------------- y, 64 rows at a time ----------------
    double mydot = 0.0;
    int it = 0;
    for (int q = cta; q * S_CB < n; q += G, it++) {
        const int i0 = q * S_CB, I0 = i0 / S_TR, J0 = i0 / TC;
        DSV s0 = {0.0f, 0.0f}, s1 = {0.0f, 0.0f};
        if (warp < SW) {
            // the row sums of row block I0 (CTAs ca .. cb), then the column sums of
            // row blocks I0 .. NI - 1: term e by warp e mod 8
            const int ca = piece_owner(CPR * tri(I0), tiles, G), cb = piece_owner(CPR * tri(I0 + 1) - 1, tiles, G);
            const int nr = cb - ca + 1, terms = nr + NI - I0;
            constexpr int U = 4;
            for (int e0 = warp; e0 < terms; e0 += SW * U) {
                V a0[U], a1[U];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int e = e0 + SW * u;
                    a0[u] = a1[u] = V{};
                    if (e < nr) {
                        const int c = ca + e;
                        if (piece_start(tiles, c, G) < piece_start(tiles, c + 1, G)) {   // not an empty CTA
                            const V *src = prow + (size_t)(c + I0) * S_TR + (i0 - I0 * S_TR) + 2 * lane;
                            a0[u] = ldcg_v(src);
                            a1[u] = ldcg_v(src + 1);
                        }
                    } else if (e < terms) {
                        const V *src = pcol + (CPR * tri(I0 + e - nr) + J0) * TC + (i0 - J0 * TC) + 2 * lane;
                        a0[u] = ldcg_v(src);
                        a1[u] = ldcg_v(src + 1);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
                    s0 = settled_sum(s0, wide(a0[u]));
                    s1 = settled_sum(s1, wide(a1[u]));
                }
            }
            comb[it & 1][warp][2 * lane] = s0;
            comb[it & 1][warp][2 * lane + 1] = s1;
            sym_consumers_sync();
            const int row = i0 + threadIdx.x;
            if (threadIdx.x < S_CB && row < n) {
                DSV s = comb[it & 1][0][threadIdx.x];
#pragma unroll
                for (int w = 1; w < SW; w++) s = settled_sum(s, comb[it & 1][w][threadIdx.x]);
                mydot += epilogue<X>(args, row, (X)to_double(s));
            }
        }
    }
    // ---- the fused dot: per CTA, then the last CTA in a fixed order ----
    const double cd = block_sum(mydot, dred);
    if (threadIdx.x == 0) {
        args.scr->cta_dot[cta] = cd;
        __threadfence();
        last_s = atomicAdd(&args.scr->ticket, 1u) == (unsigned)G - 1;
    }
    __syncthreads();
    if (!last_s) return;
    __threadfence();
    double part = 0.0;
    for (int c = threadIdx.x; c < G; c += S_T) part += __ldcg(&args.scr->cta_dot[c]);
    const double tot = block_sum(part, dred);
    if (threadIdx.x == 0) {
        run_finaliser(args, tot);
        atomicExch(&args.scr->ticket, 0u);
    }
}

// ---- packing ---------------------------------------------------------------------
// Tile (I, J) of the packed triangle from A's rows; CHECK: every a_ij of the
// tile is compared with a_ji, and State::asym set (and the rest of the matrix left out) on a
// difference of bits.  Reads all of A once with CHECK, its lower half without.
template <int DT, bool CHECK>
__global__ void __launch_bounds__(256) sym_pack_kernel(int n, int blocks, const double *__restrict__ A, long long lda,
                                                       unsigned char *__restrict__ tiles, State *st) {
    using G_ = SymGeo<DT>;
    using T = typename SymCfg<DT>::T;
    constexpr int TC = G_::TC, CPR = G_::CPR, U = 8;
    extern __shared__ __align__(16) unsigned long long low[];   // CHECK: [S_TR][TC + 1] the tile's bits
    count_launch(st);
    const long long total = CPR * tri(blocks);
    for (long long t = blockIdx.x; t < total; t += gridDim.x) {
        if (CHECK && *(volatile int *)&st->asym) return;
        const int I = tri_row(t / CPR), J = (int)(t - CPR * tri(I));
        const int i0 = I * S_TR, j0 = J * TC;
        const bool diag = j0 + TC > i0;                          // the tile meets the diagonal
        T *dst = reinterpret_cast<T *>(tiles + (size_t)t * G_::BYTES);
        for (int e0 = threadIdx.x; e0 < G_::ELEMS; e0 += 256 * U) {
            double v[U];
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int e = e0 + 256 * u, i = i0 + e / TC, j = j0 + e % TC;
                v[u] = (i < n && j <= i) ? __ldcs(&A[(long long)i * lda + j]) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < U; u++) {
                const int e = e0 + 256 * u;
                if (CHECK) low[(e / TC) * (TC + 1) + e % TC] = (unsigned long long)__double_as_longlong(v[u]);
                if constexpr (DT == DT_DS) {
                    float h, l;
                    split_pair(v[u], h, l);
                    if (diag && i0 + e / TC == j0 + e % TC) {
                        h *= 0.5f;
                        l *= 0.5f;
                    }
                    dst[e] = h;
                    dst[G_::ELEMS + e] = l;
                } else {
                    const float half = diag && i0 + e / TC == j0 + e % TC ? 0.5f : 1.0f;
                    if constexpr (DT == DT_BF16)
                        dst[e] = (uint16_t)(__float_as_uint(__bfloat162float(__double2bfloat16(v[u])) * half) >> 16);
                    else
                        dst[e] = __double2float_rn(v[u]) * half;
                }
            }
        }
        if (CHECK) {
            __syncthreads();
            bool bad = false;
            for (int e0 = threadIdx.x; e0 < G_::ELEMS; e0 += 256 * U) {
                unsigned long long v[U];
                bool in[U];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int e = e0 + 256 * u, i = i0 + e % S_TR, j = j0 + e / S_TR;
                    in[u] = i < n && j < i;
                    v[u] = in[u] ? (unsigned long long)__double_as_longlong(__ldcs(&A[(long long)j * lda + i])) : 0ull;
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int e = e0 + 256 * u;
                    bad |= in[u] && v[u] != low[(e % S_TR) * (TC + 1) + e / S_TR];
                }
            }
            if (__syncthreads_or(bad)) {
                if (threadIdx.x == 0) st->asym = 1;
                return;
            }
        }
    }
}

// ---- host side -----------------------------------------------------------------------
template <int DT>
static SymLaunch sym_launch(int num_sms) {
    SymLaunch L{};
    L.func = reinterpret_cast<void *>(&symv_kernel<DT>);
    L.grid = num_sms;
    L.block = S_T;
    L.smem = SymGeo<DT>::SMEM;
    set_smem_limit(L.func, L.smem);
    return L;
}
SymLaunch symv_plan(int dtype, int num_sms) {
    return dtype == DT_DS ? sym_launch<DT_DS>(num_sms)
           : dtype == DT_BF16 ? sym_launch<DT_BF16>(num_sms) : sym_launch<DT_F32>(num_sms);
}

template <int DT>
static size_t sym_carve(SymMat *M, unsigned char *base, int n, int num_sms) {
    using G_ = SymGeo<DT>;
    const int blocks = (n + S_TR - 1) / S_TR;
    const size_t t = (size_t)G_::CPR * tri(blocks);
    const size_t at_col = t * G_::BYTES, at_row = at_col + t * G_::TC * sizeof(typename SymCfg<DT>::V);
    const size_t end = at_row + (size_t)(num_sms + blocks) * S_TR * sizeof(typename SymCfg<DT>::V);
    if (M) {
        M->n = n;
        M->blocks = blocks;
        M->tiles = base;
        M->pcol = base + at_col;
        M->prow = base + at_row;
    }
    return end;
}
size_t symv_carve(int dtype, SymMat *M, void *base, int n, int num_sms) {
    unsigned char *b = static_cast<unsigned char *>(base);
    return dtype == DT_DS ? sym_carve<DT_DS>(M, b, n, num_sms)
           : dtype == DT_BF16 ? sym_carve<DT_BF16>(M, b, n, num_sms) : sym_carve<DT_F32>(M, b, n, num_sms);
}

template <int DT, bool CHECK>
static cudaError_t pack(const SymMat &M, const double *A, long long lda, State *st, int num_sms, cudaStream_t s) {
    const size_t smem = CHECK ? (size_t)S_TR * (SymGeo<DT>::TC + 1) * 8 : 0;
    const void *f = reinterpret_cast<const void *>(&sym_pack_kernel<DT, CHECK>);
    cudaError_t e = CHECK ? set_smem_limit(f, smem) : cudaSuccess;
    if (e != cudaSuccess) return e;
    const long long t = SymGeo<DT>::CPR * tri(M.blocks);
    const int grid = (int)(t < 8ll * num_sms ? t : 8ll * num_sms);
    sym_pack_kernel<DT, CHECK><<<grid, 256, smem, s>>>(M.n, M.blocks, A, lda, const_cast<unsigned char *>(M.tiles), st);
    return cudaGetLastError();
}
cudaError_t symv_pack(int dtype, const SymMat &M, const double *A, long long lda, State *st, int num_sms, cudaStream_t s) {
    return dtype == DT_DS     ? pack<DT_DS, true>(M, A, lda, st, num_sms, s)
           : dtype == DT_BF16 ? pack<DT_BF16, false>(M, A, lda, st, num_sms, s)
                              : pack<DT_F32, false>(M, A, lda, st, num_sms, s);
}

}  // namespace lsi
