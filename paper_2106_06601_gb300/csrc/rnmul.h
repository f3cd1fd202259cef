// RN(c * v), the product of two doubles rounded to nearest even, on the
// integer pipes: the bits of the FP64 multiply for a normal factor c and every
// v that is zero or normal with a product certain to be normal (or to overflow
// by rounding).  GB300's FP64 pipe takes 2 thread-instructions per SM and
// cycle, so kernels at memory speed have it form only some of their products.
//
// With the operands split as in fxdot.h, p = floor(significand product / 2^44)
// and the words dropped on the way tell whether it was exact.  The bits below
// the 53 of the result, with that sticky bit in the lowest, decide the
// rounding.
//
// The same code compiles for the host.
#pragma once

#include "fxdot.h"

namespace costa {
namespace rn {

struct Factor {
    uint32_t h, l;     // as fx::Op
    uint32_t sign;     // sign bit in a high word
    int32_t e;         // biased exponent - 1024: added to v's, one below the product's
    uint32_t lo, span; // admissible biased exponents of v: lo + [0, span]
};

COSTA_FX_HD Factor factor(double c) {
    const fx::Op o = fx::unpack(c);
    Factor f;
    f.h = o.h;
    f.l = o.l;
    f.sign = o.s & 0x80000000u;
    f.e = o.e - 1024;
    // v normal, and its product's exponent v + c - 1023 (+ 1) in [1, 2046]
    const int32_t lo = 1 > 1024 - o.e ? 1 : 1024 - o.e, hi = 2046 < 3068 - o.e ? 2046 : 3068 - o.e;
    const bool some = o.e >= 1 && o.e <= 2046 && hi >= lo;
    f.lo = some ? static_cast<uint32_t>(lo) : 4096u;
    f.span = some ? static_cast<uint32_t>(hi - lo) : 0u;
    return f;
}

COSTA_FX_HD bool admits(const Factor &f, double v) {
    const uint64_t u = fx::bits_of(v);
    const uint32_t hi = static_cast<uint32_t>(u >> 32), lo = static_cast<uint32_t>(u);
    return ((hi >> 20) & 0x7FFu) - f.lo <= f.span || (((hi & 0x7FFFFFFFu) | lo) == 0u && f.lo < 4096u);
}

// RN(c * v) for an admitted v.
COSTA_FX_HD double mul(const Factor &f, double v) {
    const uint64_t u = fx::bits_of(v);
    const uint32_t hi = static_cast<uint32_t>(u >> 32), lo = static_cast<uint32_t>(u);
    const uint32_t e = (hi >> 20) & 0x7FFu;
    const uint32_t h = (((hi & 0xFFFFFu) | 0x100000u) << 10) | (lo >> 22), l = lo << 10;
    const uint64_t low = fx::mad_wide(f.l, l, 0);
    const uint64_t mid = fx::mad_wide(f.l, h, fx::mad_wide(f.h, l, low >> 32));
    uint64_t p = fx::mad_wide(f.h, h, mid >> 32);  // in [2^60, 2^62)
    const uint32_t below = static_cast<uint32_t>(mid) | static_cast<uint32_t>(low);
    p |= below ? 1u : 0u;
    const uint32_t two = static_cast<uint32_t>(p >> 61);  // 1 when the significands' product is at least 2
    p <<= 1u - two;                                       // the result's bits are now 61 .. 9
    p += 0xFFu + (static_cast<uint32_t>(p >> 9) & 1u);    // to nearest, ties to even
    const uint64_t sig = p >> 9;  // in [2^52, 2^53]: its hidden bit adds 1 to the exponent below
    const uint32_t rh = static_cast<uint32_t>(sig >> 32) + ((e + static_cast<uint32_t>(f.e) + two) << 20);
    const uint32_t sign = (hi & 0x80000000u) ^ f.sign;
    const uint64_t r = (static_cast<uint64_t>(sign | rh) << 32) | static_cast<uint32_t>(sig);
    return fx::from_bits(e ? r : static_cast<uint64_t>(sign) << 32);
}

}  // namespace rn
}  // namespace costa
