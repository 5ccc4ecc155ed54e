// cls_fixed.h -- the 96-bit fixed point in which the FP64 walk sums its flights'
// track lengths bin by bin.
//
// A flight scores in units of 2^-F bin widths.  F is 64 where a mean flight is a
// bin width or longer, down to 2^-8 of one, and grows with the bin width over the
// mean flight beyond that (fixed_bits), so a mean flight is worth 2^56 units and
// more and is rounded below the last place of a double.  Flights of 2^(90 - F)
// bin widths and more (2^34 mean flights, or 2^26 bin widths) score into the global
// bins in FP64.  So a deposit is kept to all the bits that a double sum has, and
// the sums lose none.  (64 bits, 48 of them fractions of a bin width whatever the
// flights' length, lost 1% of a bin of 1e14 flights' width and all of one of 1e16,
// and four bits of a bin with a single flight.)  The third word costs the FP64 walk
// 1 to 4%: box L = 10, 1e7 histories, 33.1 -> 34.5 ms; slab 1e6 552 -> 571 us;
// extruded 3e5 1019 -> 1039 us; FP64 additions to shared memory, compare-and-swap
// loops, cost the box 13% before the steps that followed.
//
// Host and device compile the same code (the host build serves tests).
#pragma once

#include <algorithm>
#include <cmath>

#include "cls_intmath.h"

namespace cls {

struct Fix96 {
    uint32_t w0, w1, w2;  // low word first
};

// One deposit is below 2^kFixedDepositBits units.
constexpr int kFixedDepositBits = 90;
// F of a case whose flights all score in FP64: no double is below 2^(90 - F).
constexpr int kFixedNone = 4000;

// Fraction bits of a bin width dx for a case whose materials' mean flights are
// 1/(Sigma + 1/Lambda): the shortest, or where a chord ends before the material
// collides, the share of the other material's flights that its histories take.
inline int fixed_bits(double dx, const double *sigma, const double *lambda) {
    const double t[2] = {1.0 / (sigma[0] + 1.0 / lambda[0]), 1.0 / (sigma[1] + 1.0 / lambda[1])};
    double flight = INFINITY;
    for (int m = 0; m < 2; ++m)
        flight = std::min(flight, std::max(t[m], t[1 - m] / (1.0 + sigma[m] * lambda[m])));
    if (!(flight > 0.0) || !std::isfinite(1.0 / dx)) return kFixedNone;
    int ed, ef;
    const double md = std::frexp(dx, &ed), mf = std::frexp(flight, &ef);
    const int over = ed - ef + (md > mf ? 1 : 0);  // dx <= 2^over flights
    const int bits = 64 + std::max(0, over - 8);
    return ed - bits < -960 ? kFixedNone : bits;  // the unit dx 2^-F stays a normal double
}

// x >> t for t >= 0, 0 from t = 64 on (as the GPU shifts)
CLS_HD uint64_t shift_right(uint64_t x, int t) {
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(t));
    return r;
#else
    return t < 64 ? x >> t : 0ull;
#endif
}

// floor(v 2^F) for 0 <= v < 2^(kFixedDepositBits - F)
CLS_HD Fix96 fixed96(double v, int F) {
    uint64_t b;
#ifdef __CUDA_ARCH__
    b = (uint64_t)__double_as_longlong(v);
#else
    memcpy(&b, &v, sizeof b);
#endif
    // the significand at the top of 96 bits, shifted right by t >= 6
    const uint64_t N = ((b << 11) & 0x7FFFFFFFFFFFFFFFull) | (1ull << 63);
    const int t = 95 + 1023 - F - (int)(b >> 52);
    const uint64_t hi = shift_right(N, t);
    const uint32_t lo = (uint32_t)shift_right(t < 32 ? N << 32 : N, t < 32 ? t : t - 32);
    return Fix96{lo, (uint32_t)hi, (uint32_t)(hi >> 32)};
}

// a - b modulo 2^96
CLS_HD Fix96 sub96(const Fix96 &a, const Fix96 &b) {
    Fix96 r;
#ifdef __CUDA_ARCH__
    asm("sub.cc.u32 %0, %3, %6;\n\tsubc.cc.u32 %1, %4, %7;\n\tsubc.u32 %2, %5, %8;"
        : "=r"(r.w0), "=r"(r.w1), "=r"(r.w2)
        : "r"(a.w0), "r"(a.w1), "r"(a.w2), "r"(b.w0), "r"(b.w1), "r"(b.w2));
#else
    const uint64_t al = (uint64_t)a.w1 << 32 | a.w0, bl = (uint64_t)b.w1 << 32 | b.w0, l = al - bl;
    r = Fix96{(uint32_t)l, (uint32_t)(l >> 32), a.w2 - b.w2 - (al < bl ? 1u : 0u)};
#endif
    return r;
}

// a + b modulo 2^96
CLS_HD Fix96 add96(const Fix96 &a, const Fix96 &b) {
    Fix96 r;
#ifdef __CUDA_ARCH__
    asm("add.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, %7;\n\taddc.u32 %2, %5, %8;"
        : "=r"(r.w0), "=r"(r.w1), "=r"(r.w2)
        : "r"(a.w0), "r"(a.w1), "r"(a.w2), "r"(b.w0), "r"(b.w1), "r"(b.w2));
#else
    const uint64_t al = (uint64_t)a.w1 << 32 | a.w0, bl = (uint64_t)b.w1 << 32 | b.w0, l = al + bl;
    r = Fix96{(uint32_t)l, (uint32_t)(l >> 32), a.w2 + b.w2 + (l < al ? 1u : 0u)};
#endif
    return r;
}

// f 2^-64 of q, for q < 2^kFixedDepositBits: at most 3 units below the product,
// never above it (the low words' products of 2^-64 and the fractions of the two
// of 2^-32 are left out)
CLS_HD Fix96 fraction96(uint64_t f, const Fix96 &q) {
    const uint32_t fh = (uint32_t)(f >> 32), fl = (uint32_t)f;
    const uint64_t m = (uint64_t)fh * q.w1 + umulhi32(fl, q.w1) + umulhi32(fh, q.w0);  // at most 2^64 - 3
    const uint64_t a = (uint64_t)fl * q.w2 + (uint32_t)m;                              // below 2^59
    const uint64_t u = (uint64_t)fh * q.w2 + (m >> 32) + (a >> 32);                    // below 2^59
    return Fix96{(uint32_t)a, (uint32_t)u, (uint32_t)(u >> 32)};
}

// the sum as a double, in units, rounded twice at most (once below 2^85 units)
CLS_HD double fix96_to_double(const Fix96 &q) {
    return (double)((uint64_t)q.w2 << 32 | q.w1) * 0x1p32 + (double)q.w0;
}

}  // namespace cls
