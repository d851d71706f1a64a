// Host check of the block product's rule in csrc/gemv_split.h against sizes at which both forms
// were measured and differ by more than 5 %.
#include <cstdio>

#include "gemv_split.h"

using namespace lsi;

int main() {
    struct {
        int S, n;
        bool whole;
    } T[] = {{8, 300, true},   {8, 1000, true},  {8, 1500, true},  {8, 2001, true},  {8, 2300, true},  {8, 2450, false},
             {8, 2700, false}, {8, 3500, false}, {8, 4500, true},  {8, 5000, false}, {8, 6000, false}, {8, 8000, false},
             {8, 9801, false}, {4, 300, true},   {4, 2001, true},  {4, 2450, false}, {4, 3000, false}, {4, 4500, true},
             {4, 5000, false}, {4, 6000, false}, {4, 8000, false}, {2, 1000, true},  {2, 2300, true},  {2, 2450, false},
             {2, 4500, true},  {2, 5000, false}, {2, 6000, false}, {2, 9801, false}, {1, 800, true},   {1, 2001, true},
             {1, 3500, true},  {1, 4500, true},  {1, 5000, false}, {1, 7000, true},  {1, 9801, false}};
    int bad = 0;
    for (auto &t : T)
        if (bgemv_whole_blocks(bgemv_costs(t.S), (t.n + 15) / 16, (t.n + 255) / 256, 152) != t.whole) {
            std::printf("S %d, n %d: expected %s\n", t.S, t.n, t.whole ? "whole row blocks" : "equal pieces");
            bad++;
        }
    for (int S = 1; S <= 8; S *= 2)   // a full turn leaves no SM idle
        if (!bgemv_whole_blocks(bgemv_costs(S), 304, 19, 152)) bad++;
    std::printf("mismatches %d\n", bad);
    return bad != 0;
}
