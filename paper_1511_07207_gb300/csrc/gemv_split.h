// gemv_split.h -- how the products (k_gemv.cu, k_bgemv.cu) deal their tiles to the
// CTAs: whole row tiles, or equal pieces of the tile sequence.  Host code, which the
// CPU tests compile too.
#pragma once

namespace lsi {

// Times in ns that the rule weighs: a tile of a CTA that walks a whole row tile; a tile of
// equal pieces, per SM (two CTAs share it); the fixed part of adding partial sums with the
// neighbours, and the part for each of the CTAs that share a row tile.
struct GemvCosts {
    int tile, piece, meet, sharer;
};

// Row tiles (RT) that fit the grid of G CTAs (two an SM) may go to one CTA each, which
// then adds nothing up with its neighbours.  The longest CTA has CT tiles to
// walk, whatever RT is; in equal pieces all SMs share RT x CT tiles and the
// meeting costs 6 to 13 us.  So whole row tiles win while CT is small: few tiles altogether, or
// nearly as many row tiles as CTAs.  Taking them by RT alone left the chip to RT CTAs
// however wide the matrix: 64 x 1000000 took 2679 us for the FP32 pair, 1863 us for BF16,
// 1935 us for FP8 and 1987 us for FP32; 141, 135, 220 and 102 us in equal pieces.
//
// The costs are fitted to both forms measured at 116 shapes a format (16 to 19400
// rows, 256 to 250000 columns, squares from 128 to 19000): at none of them is the form
// that is chosen slower than equal pieces by more than 2 % or half a microsecond.  Whole
// row tiles against equal pieces: n = 1024 10.3 and 16.4 us (pair), 10.3 and 20.5 (FP8);
// n = 4000 28.9 and 35.9 (pair), 14.7 and 18.5 (BF16), 14.4 and 20.5 (FP32); n = 9500
// 39.4 and 41.7 (BF16), but 35.4 and 29.1 for FP8, which takes pieces there.
inline bool gemv_whole_tiles(GemvCosts c, int RT, int CT, int G) {
    if (RT < 1 || RT > G) return false;
    const long long share = G / RT < CT ? G / RT : CT;
    return (long long)CT * c.tile * G <= 2ll * RT * CT * c.piece + (c.meet + c.sharer * share) * G;
}

constexpr GemvCosts GEMV_COSTS_PAIR = {900, 540, 13000, 1000};
constexpr GemvCosts GEMV_COSTS_BF16 = {560, 440, 6000, 950};
constexpr GemvCosts GEMV_COSTS_FP8 = {920, 250, 13000, 1000};
constexpr GemvCosts GEMV_COSTS_F32 = {520, 250, 5300, 1300};

// ---- the block product -----------------------------------------------------------------
// One CTA an SM; whole row blocks go to CTA c, c + G, ..., so the longest CTA has
// ceil(RB / G) CT tiles, in equal pieces RB CT / G.  Pieces win when the tiles they
// save take longer than the meeting of the CTAs that share a row block.
struct BgemvCosts {
    int tile, meet;   // ns
};
inline bool bgemv_whole_blocks(BgemvCosts c, long long RB, long long CT, long long G) {
    const long long idle = (RB + G - 1) / G * CT * G - RB * CT;   // over all CTAs
    return idle * c.tile < c.meet * G;
}
// Fitted to both forms at 20 sizes from n = 300 to 9801 (caches cold): the form chosen is
// within 2 % of the faster one.  Eight columns: n = 1000 16.9 us whole, 23.8 in pieces; 2001
// 26.2 and 34.3; 2450 53.2 and 42.0; 4500 87.3 and 92.3; 8000 287.9 and 249.7.
inline BgemvCosts bgemv_costs(int S) {
    return S <= 1 ? BgemvCosts{650, 8500} : S <= 2 ? BgemvCosts{870, 6500} : S <= 4 ? BgemvCosts{1370, 10400} : BgemvCosts{2400, 12800};
}

}  // namespace lsi
