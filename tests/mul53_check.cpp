// Host check of the integer-pipe product: where mul53 does not report a tie it
// must give the bits of the rounded FP64 product, for normal operands with a
// normal product.  Prints "checked N mismatches M ties T"; exit 1 on a mismatch.
#include <cstdint>
#include <cstdio>
#include <cstring>

#include "mul53.h"

static uint64_t rng_state = 0x9E3779B97F4A7C15ull;
static uint64_t next_u64() {   // xorshift64*
    rng_state ^= rng_state >> 12;
    rng_state ^= rng_state << 25;
    rng_state ^= rng_state >> 27;
    return rng_state * 0x2545F4914F6CDD1Dull;
}
static double make(uint64_t sign, int field, uint64_t frac) {
    const uint64_t b = (sign << 63) | ((uint64_t)field << 52) | (frac & ((1ull << 52) - 1));
    double d;
    memcpy(&d, &b, 8);
    return d;
}

static long long checked = 0, bad = 0, ties = 0;
static void check(double x, double y) {
    bool tie = false;
    const lsi::Op53 a = lsi::op53_a(x), b = lsi::op53_b(y);
    const double p = lsi::mul53(a, b, tie), q = x * y;
    const double xa = lsi::op53_value(a, 5), yb = lsi::op53_value(b, 6);
    checked++;
    ties += tie;
    if (memcmp(&xa, &x, 8) || memcmp(&yb, &y, 8) || (!tie && memcmp(&p, &q, 8))) {
        if (bad < 10) printf("mismatch %a * %a: %a, %a\n", x, y, p, q);
        bad++;
    }
}

int main() {
    // random significands at every pair of exponent fields near the borders of the range, and anywhere
    const int fields[] = {1, 2, 3, 511, 512, 513, 1000, 1022, 1023, 1024, 1025, 1534, 2044, 2045, 2046};
    for (int fa : fields)
        for (int fb : fields)
            if (lsi::mul53_in_range(fa, fa, fb, fb))
                for (int i = 0; i < 20000; i++)
                    check(make(next_u64() & 1, fa, next_u64()), make(next_u64() & 1, fb, next_u64()));
    for (int i = 0; i < 3000000; i++)
        check(make(next_u64() & 1, 600 + (int)(next_u64() % 800), next_u64()),
              make(next_u64() & 1, 600 + (int)(next_u64() % 800), next_u64()));
    // few significant bits (exact products and real ties), all ones, borders of the one-bit shift
    const uint64_t fr[] = {0, 1, 2, 3, 1ull << 51, (1ull << 51) + 1, (1ull << 52) - 1, (1ull << 52) - 2,
                           0x6A09E667F3BCCull, 0x6A09E667F3BCDull, 0x5555555555555ull, 0xAAAAAAAAAAAAAull,
                           1ull << 26, (1ull << 26) + 1, (1ull << 25) - 1, 0xFFFFFFFFull, 0x100000000ull};
    for (uint64_t f : fr)
        for (uint64_t g : fr)
            for (uint64_t s = 0; s < 2; s++) check(make(s, 1020, f), make(0, 1030, g));
    for (int x = 1; x < 3000; x++)
        for (int y = 1; y < 300; y++) check((double)x, -(double)y);
    for (int i = 0; i < 2000000; i++) {   // products of 54 bits whose last bit is set: exact ties
        const uint64_t f = (next_u64() & 0x7FFFFFFull) | 1, g = (next_u64() & 0x7FFFFFFull) | 1;
        check((double)f, (double)g);
    }
    printf("checked %lld mismatches %lld ties %lld\n", checked, bad, ties);
    return bad || ties == 0 ? 1 : 0;
}
