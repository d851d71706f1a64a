// mul53.h -- the correctly rounded FP64 product (round to nearest, ties to
// even) formed with 32-bit integer operations, for the direct methods' rank
// updates a_ij - l_it u_tj.
//
// Those updates keep the product and the difference apart, each rounded (so
// that the factors are bit for bit the plain elimination's), which is two
// instructions on the FP64 pipe an element and step; that pipe issues a warp
// instruction every 64 cycles per scheduler on this GPU and is what bounds
// the factorizations.  The integer pipes idle meanwhile, so the product moves
// there and the FP64 pipe keeps the difference alone.
//
// An operand v = (-1)^s 2^(e-1075) m, m its 53-bit integer significand, is kept
// as m shifted left (by 5 in the first factor, by 6 in the second: the two
// shifts together put the product's top 64 bits where a 53-bit significand
// ends) and as its sign and exponent field.  With (a1 a0) and (b1 b0) the 32-bit
// halves of the shifted significands,
//     2^11 m_a m_b = a1 b1 2^64 + (a1 b0 + a0 b1) 2^32 + a0 b0
// (a1 < 2^26, b1 < 2^27, so the middle sum does not overflow 64 bits).  The
// high 64 bits of it are the product's significand, in [2^51, 2^53); when they are
// below 2^52 everything moves up one bit.  The 32 bits below the significand
// decide the rounding except when they are exactly one half: then the rest
// of a0 b0 and the parity of the significand matter, and mul53 only reports
// the case (`tie`); the caller takes the product from the FP64 pipe.  A carry out
// of the rounded significand raises the exponent field by itself.
//
// Valid for normal operands whose product is normal: the caller checks the
// exponent fields (mul53_in_range on the extremes of a tile).
#pragma once

#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define LS_MUL53_FN __host__ __device__ __forceinline__
#else
#define LS_MUL53_FN inline
#endif

namespace lsi {

// One operand: the shifted significand (hi, lo), the sign and exponent field
// (the second factor's without the exponent bias), and the value's high word.
struct alignas(16) Op53 {
    uint32_t lo, hi, e, raw;
};

LS_MUL53_FN Op53 op53_split(uint32_t lw, uint32_t hw, int shift, uint32_t bias) {
    Op53 o;
    const uint32_t m1 = (hw & 0xFFFFFu) | 0x100000u;
    o.lo = lw << shift;
    o.hi = (m1 << shift) | (lw >> (32 - shift));
    o.e = (hw & 0xFFF00000u) - bias;
    o.raw = hw;
    return o;
}
LS_MUL53_FN Op53 op53_a(double v) {
    uint64_t u;
    memcpy(&u, &v, 8);
    return op53_split((uint32_t)u, (uint32_t)(u >> 32), 5, 0u);
}
LS_MUL53_FN Op53 op53_b(double v) {
    uint64_t u;
    memcpy(&u, &v, 8);
    return op53_split((uint32_t)u, (uint32_t)(u >> 32), 6, 1023u << 20);
}
// The value an operand was made from (any value, the out-of-range ones included).
LS_MUL53_FN double op53_value(const Op53 &o, int shift) {
    const uint32_t lw = (o.lo >> shift) | (o.hi << (32 - shift));
    const uint64_t u = ((uint64_t)o.raw << 32) | lw;
    double v;
    memcpy(&v, &u, 8);
    return v;
}
LS_MUL53_FN int op53_field(const Op53 &o) { return (int)((o.raw >> 20) & 0x7FFu); }

// Every product of a first factor with exponent field in [amin, amax] and a
// second one with [bmin, bmax] can be formed by mul53.
LS_MUL53_FN bool mul53_in_range(int amin, int amax, int bmin, int bmax) {
    return amin >= 1 && bmin >= 1 && amax <= 2046 && bmax <= 2046 && amin + bmin >= 1025 && amax + bmax <= 3068;
}

// a b rounded to nearest even; tie is set (never cleared) when the rounding
// needs more than the bits formed here.
LS_MUL53_FN double mul53(const Op53 &a, const Op53 &b, bool &tie) {
    uint32_t r, ml, mh;
#if defined(__CUDA_ARCH__)
    uint32_t tl, hl, hh;
    asm("{\n\t"
        ".reg .u32 c, th;\n\t"
        ".reg .u64 t, h;\n\t"
        "mul.hi.u32 c, %3, %5;\n\t"
        "mul.wide.u32 t, %4, %5;\n\t"
        "mad.wide.u32 t, %3, %6, t;\n\t"
        "mul.wide.u32 h, %4, %6;\n\t"
        "mov.b64 {%0, th}, t;\n\t"
        "mov.b64 {%1, %2}, h;\n\t"
        "add.cc.u32 %0, %0, c;\n\t"
        "addc.cc.u32 %1, %1, th;\n\t"
        "addc.u32 %2, %2, 0;\n\t}"
        : "=r"(tl), "=r"(hl), "=r"(hh)
        : "r"(a.lo), "r"(a.hi), "r"(b.lo), "r"(b.hi));
    const uint32_t s20 = ~hh & 0x100000u, s = s20 >> 20;   // one when the significand starts a bit lower
    ml = __funnelshift_l(tl, hl, s);
    mh = __funnelshift_l(hl, hh, s);
    r = tl << s;
    const uint32_t e = a.e + b.e - s20;
    uint32_t r2;
    asm("add.cc.u32 %0, %3, 0x80000000;\n\t"
        "addc.cc.u32 %1, %1, 0;\n\t"
        "addc.u32 %2, %2, %4;"
        : "=&r"(r2), "+r"(ml), "+r"(mh)
        : "r"(r), "r"(e));
    tie |= r2 == 0u;
    return __hiloint2double((int)mh, (int)ml);
#else
    const uint32_t c = (uint32_t)(((uint64_t)a.lo * b.lo) >> 32);
    uint64_t t = (uint64_t)a.hi * b.lo + (uint64_t)a.lo * b.hi;
    t += c;
    uint64_t h = (uint64_t)a.hi * b.hi + (t >> 32);
    const uint32_t s20 = ~(uint32_t)(h >> 32) & 0x100000u, s = s20 >> 20;
    r = (uint32_t)t << s;
    h = s ? (h << 1) | ((uint32_t)t >> 31) : h;
    h += r >> 31;
    ml = (uint32_t)h;
    mh = (uint32_t)(h >> 32) + a.e + b.e - s20;
    tie |= r == 0x80000000u;
    const uint64_t u = ((uint64_t)mh << 32) | ml;
    double v;
    memcpy(&v, &u, 8);
    return v;
#endif
}

}  // namespace lsi
