// Host check of csrc/gemv_split.h: which matrices are dealt out as whole row tiles.
#include <cstdio>

#include "gemv_split.h"

using namespace lsi;

static int bad = 0;
static void expect(bool whole, GemvCosts c, const char *name, int tr, int rows, long long cols, int G = 304) {
    const int RT = (rows + tr - 1) / tr, CT = (int)((cols + 255) / 256);
    if (gemv_whole_tiles(c, RT, CT, G) != whole) {
        std::printf("%s %d x %lld: expected %s\n", name, rows, cols, whole ? "whole row tiles" : "equal pieces");
        bad++;
    }
}

int main() {
    struct {
        const char *name;
        GemvCosts c;
        int tr;
    } F[] = {{"pair", GEMV_COSTS_PAIR, 16}, {"bf16", GEMV_COSTS_BF16, 32}, {"fp8", GEMV_COSTS_FP8, 64}, {"f32", GEMV_COSTS_F32, 16}};
    for (auto &f : F) {
        // wide: few CTAs would walk the whole matrix
        expect(false, f.c, f.name, f.tr, 64, 1000000);
        expect(false, f.c, f.name, f.tr, 64, 250000);
        expect(false, f.c, f.name, f.tr, 300, 40000);
        expect(false, f.c, f.name, f.tr, 1000, 100000);
        // small: the meetings would be most of the time
        expect(true, f.c, f.name, f.tr, 1, 1);
        expect(true, f.c, f.name, f.tr, 512, 512);
        expect(true, f.c, f.name, f.tr, 1024, 1024);
        expect(true, f.c, f.name, f.tr, 4000, 4000);
        // more row tiles than CTAs
        expect(false, f.c, f.name, f.tr, 304 * f.tr + 1, 100);
        expect(false, f.c, f.name, f.tr, 304 * f.tr + 1, 20000);
        // a chosen form never changes back as the matrix gets wider
        for (int RT = 1; RT <= 304; RT++) {
            bool was = true;
            for (int CT = 1; CT < 40000; CT += 1 + CT / 8) {
                const bool w = gemv_whole_tiles(f.c, RT, CT, 304);
                if (w && !was) {
                    std::printf("%s RT %d CT %d: whole again\n", f.name, RT, CT);
                    bad++;
                }
                was = w;
            }
        }
        if (gemv_whole_tiles(f.c, 0, 5, 304)) bad++;
        // no overflow at the largest sizes an int takes
        if (gemv_whole_tiles(f.c, 1, 8388608, 304)) bad++;
    }
    expect(false, GEMV_COSTS_FP8, "fp8", 64, 9500, 9500);   // 149 of 304 CTAs: 34.5 us against 28.8
    expect(true, GEMV_COSTS_PAIR, "pair", 16, 4800, 4800);
    std::printf("mismatches %d\n", bad);
    return bad != 0;
}
