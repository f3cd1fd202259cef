// Sum of 2 or 4 products of doubles in fixed point on the integer pipes:
// one component of alpha * b + beta * a with complex scalars (Eq. 1, Sec. 5)
// for double data, where GB300's FP64 pipe is too narrow for a compensated
// floating-point evaluation at memory speed.
//
// Every operand must be zero or of magnitude in [2^-480, 2^480) (no
// subnormal, infinite or NaN operand; callers test this and take another
// evaluation otherwise).  Then:
//   1. each product's significand product is formed from the two 53-bit
//      significands, split into their top 31 and low 22 bits (these shifted
//      to the top of a word), by four 32 x 32 -> 64-bit multiply-adds, of
//      which the bits below 2^44 are dropped: the floor, in [2^60, 2^62);
//   2. the products are aligned to the largest exponent, with one bit of
//      headroom, and summed exactly as signed 64-bit integers in units
//      U = 2^-7 ulp(M) or finer (M the largest product): dropping and
//      alignment together truncate less than one U per product;
//   3. the integer sum is rounded once to double, to nearest even, by the
//      hardware's conversion (dot2_mid: with integer instructions), and the
//      exponent added to its exponent field.
// The result is within 0.5 ulp(x) + n U of the exact sum x of the n exact
// products: n U <= 2^-5 ulp(M), so at most 0.5 ulp(x) + 0.032 ulp(M).  Where
// products cancel, that is far above an ulp of x; sums of two products, whose
// alternative is Kahan's algorithm with 2u|x|, carry 32 bits more (dot2_mid).  All
// intermediate magnitudes stay in the normal range: a product lies in
// [2^-960, 2^960), the sum below 2^962, and a nonzero result is a multiple of
// U >= 2^-1019.
//
// The ALU pipe bounds the kernels that use it.  This split keeps every
// partial sum inside 64 bits, so that there are no carries, and drops whole
// words, so that there are no shifts (one 64 x 64 -> high 64 multiply takes
// about twice the instructions); the conversion replaces
// the count of leading zeros, the shifts and the rounding: 4096^2 c128 T,
// complex beta, BC64 -> BC128: 2340 -> 3450 GB/s (430 -> 320
// instructions per element).
//
// The same code compiles for the host (costa_debug_fxdot uses it), so the
// arithmetic can be checked without a GPU.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define COSTA_FX_HD __host__ __device__ __forceinline__
#define COSTA_FX_HD_CALL static __host__ __device__ __noinline__
#else
#define COSTA_FX_HD inline
#define COSTA_FX_HD_CALL inline
#endif

namespace costa {
namespace fx {

COSTA_FX_HD uint64_t bits_of(double v) {
#ifdef __CUDA_ARCH__
    return static_cast<uint64_t>(__double_as_longlong(v));
#else
    uint64_t u;
    std::memcpy(&u, &v, sizeof u);
    return u;
#endif
}

COSTA_FX_HD double from_bits(uint64_t u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(static_cast<long long>(u));
#else
    double v;
    std::memcpy(&v, &u, sizeof v);
    return v;
#endif
}

// x * y + a without overflow checks (one multiply-add on the GPU).
COSTA_FX_HD uint64_t mad_wide(uint32_t x, uint32_t y, uint64_t a) {
    return static_cast<uint64_t>(x) * y + a;
}

// v >> n, 0 for n >= 64 (the GPU's shift clamps its count).
COSTA_FX_HD uint64_t shr_clamp(uint64_t v, uint32_t n) {
#ifdef __CUDA_ARCH__
    uint64_t r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
    return r;
#else
    return n < 64u ? v >> n : 0;
#endif
}

COSTA_FX_HD uint32_t leading_zeros(uint64_t v) {
#ifdef __CUDA_ARCH__
    return static_cast<uint32_t>(__clzll(static_cast<long long>(v)));
#else
    return static_cast<uint32_t>(__builtin_clzll(v));
#endif
}

// The integer rounded to the nearest double, ties to even.
COSTA_FX_HD double round_to_double(int64_t v) {
#ifdef __CUDA_ARCH__
    return __ll2double_rn(v);
#else
    return static_cast<double>(v);  // the default rounding mode is to nearest even
#endif
}

// An operand: its 53-bit significand as 31 top bits (h) and 22 low bits at the
// top of a word (l = low bits * 2^10), both 0 for a zero; its biased exponent (kZeroExp for a zero, so that a zero
// product never is the largest); its sign as a mask.
constexpr int32_t kZeroExp = -8192;
struct Op {
    uint32_t h, l;
    int32_t e;
    uint32_t s;
};

// Zero, or a magnitude in [2^-480, 2^480): the range in which unpack and
// sum below are exact as stated.
COSTA_FX_HD bool in_range(double v) {
    const uint64_t u = bits_of(v);
    const uint32_t e = static_cast<uint32_t>(u >> 52) & 0x7FFu;
    return (u << 1) == 0 || (e - (1023u - 480u)) < 960u;
}

COSTA_FX_HD Op unpack(double v) {
    const uint64_t u = bits_of(v);
    const uint32_t hi = static_cast<uint32_t>(u >> 32), lo = static_cast<uint32_t>(u);
    const uint32_t e = (hi >> 20) & 0x7FFu;
    const uint32_t top = e ? (hi & 0xFFFFFu) | 0x100000u : 0u;
    Op o;
    o.h = (top << 10) | (lo >> 22);
    o.l = lo << 10;
    o.e = e ? static_cast<int32_t>(e) : kZeroExp;
    o.s = static_cast<uint32_t>(static_cast<int32_t>(hi) >> 31);
    return o;
}

// One product x * y, negated when neg = 1: floor(significand product / 2^44)
// (in [2^60, 2^62), or 0), the next 32 bits of that quotient, the sum of the
// biased exponents and the sign as a mask.
struct Term {
    uint64_t p;
    uint32_t r;
    int32_t e;
    uint32_t s;
};

COSTA_FX_HD Term mul(const Op &x, const Op &y, uint32_t neg) {
    Term t;
    const uint64_t low = mad_wide(x.l, y.l, 0) >> 32;
    const uint64_t mid = mad_wide(x.l, y.h, mad_wide(x.h, y.l, low));  // below 2^64 (h < 2^31)
    t.p = mad_wide(x.h, y.h, mid >> 32);
    t.r = static_cast<uint32_t>(mid);
    t.e = x.e + y.e;
    t.s = x.s ^ y.s ^ (neg ? 0xFFFFFFFFu : 0u);
    return t;
}

// bits * 2^(emax - 2105) for the bits of a nonzero double: a sum's unit (a
// significand product has unit 2^(emax - 2150), and this is 2^45 of it).
COSTA_FX_HD double scaled(uint64_t bits, int32_t emax) {
    return from_bits(bits + (static_cast<uint64_t>(static_cast<int64_t>(emax - 2105)) << 52));
}

// The sum of n <= 4 terms, rounded once to double (to nearest, ties to even).
// A zero sum gives +0.
template <int N>
COSTA_FX_HD double sum(const Term (&t)[N]) {
    int32_t emax = t[0].e;
#pragma unroll
    for (int i = 1; i < N; ++i) emax = t[i].e > emax ? t[i].e : emax;
    uint64_t acc = 0;
    uint32_t neg = 0;  // minus the number of negative terms: v ^ mask = -v - 1
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const uint64_t v = shr_clamp(t[i].p, static_cast<uint32_t>(emax - t[i].e + 1));  // < 2^61: |sum| < 2^63
        const uint64_t mask = (static_cast<uint64_t>(t[i].s) << 32) | t[i].s;
        acc += v ^ mask;
        neg += t[i].s;
    }
    acc -= static_cast<uint64_t>(static_cast<int64_t>(static_cast<int32_t>(neg)));
    if (acc == 0) return 0.0;
    return scaled(bits_of(round_to_double(static_cast<int64_t>(acc))), emax);
}

// ---- sums of two products ----

COSTA_FX_HD double fma_rn(double x, double y, double z) {
#ifdef __CUDA_ARCH__
    return __fma_rn(x, y, z);
#else
    return std::fma(x, y, z);
#endif
}
COSTA_FX_HD double mul_rn(double x, double y) {
#ifdef __CUDA_ARCH__
    return __dmul_rn(x, y);
#else
    return x * y;
#endif
}
COSTA_FX_HD double add_rn(double x, double y) {
#ifdef __CUDA_ARCH__
    return __dadd_rn(x, y);
#else
    return x + y;
#endif
}

// x * y + z * t, or x * y - z * t (minus), with Kahan's algorithm for 2 x 2
// determinants: w = z * t rounded, its error e exactly by one fma, then (x * y
// +- w) rounded by a second fma and +- e added.  Jeannerod, Louvet and Muller
// ("Further analysis of Kahan's algorithm for the accurate computation of
// 2 x 2 determinants", Math. Comp. 82, 2013) bound its error by 2u|exact|
// when nothing overflows or underflows: within 2 ulps of the exact value,
// and so of the oracle's compensated result.  4 FP64 operations instead of
// Dot2's 13.
COSTA_FX_HD double kahan2(double x, double y, double z, double t, bool minus) {
    const double w = mul_rn(z, t);
    const double e = fma_rn(z, t, -w);  // z * t = w + e exactly
    return minus ? add_rn(fma_rn(x, y, -w), -e) : add_rn(fma_rn(x, y, w), e);
}

// A call of its own, so that the FP64 pipe is not held by instructions that are
// predicated off.
COSTA_FX_HD_CALL double kahan2_far(double x, double y, double z, double t) { return kahan2(x, y, z, t, false); }

// The low 32 bits of (hi:lo) >> n, hi for n >= 32; the high 32 of (hi:lo) << n, n < 32.
COSTA_FX_HD uint32_t funnel_shr(uint32_t lo, uint32_t hi, uint32_t n) {
#ifdef __CUDA_ARCH__
    return __funnelshift_rc(lo, hi, n);
#else
    return n < 32u ? static_cast<uint32_t>(((static_cast<uint64_t>(hi) << 32) | lo) >> n) : hi;
#endif
}
COSTA_FX_HD uint32_t funnel_shl(uint32_t lo, uint32_t hi, uint32_t n) {
#ifdef __CUDA_ARCH__
    return __funnelshift_l(lo, hi, n);
#else
    return static_cast<uint32_t>(((static_cast<uint64_t>(hi) << 32 | lo) << n) >> 32);
#endif
}

// x * y + z * t for operands in range, within 2u of the exact value (u =
// 2^-53), the bound of Kahan's algorithm, whatever cancels: a sum in fixed
// point with 32 bits more than `sum` has, so that it is within 1.02u wherever
// it has at least 2^31 of sum's units (the larger product has at least 2^59):
// terms of nearly the same exponent are off by less than 2^-32 of a unit each;
// one that is shifted by more than 32 bits is off by less than a unit, but
// then nothing cancels.  Below, Kahan's algorithm.  Rounded without the
// hardware's conversion: the other component of the complex-alpha kind is
// formed on the FP64 pipe, and the conversions' rate is as low (without the 32
// bits 173 -> 148 us).  GB300, c128 4096^2 T, complex alpha, BC64 -> BC128, us
// per call: 157; Kahan's algorithm for both components 212; no more bits than
// `sum`, and Kahan's algorithm below 2^54 units (a third of the warps) 173;
// never Kahan's algorithm, thousands of ulps off where the products cancel, 148.
COSTA_FX_HD double dot2_mid(double x, double y, double z, double t) {
    const Term a = mul(unpack(x), unpack(y), 0u), b = mul(unpack(z), unpack(t), 0u);
    const int32_t emax = a.e > b.e ? a.e : b.e;
    const uint32_t na = static_cast<uint32_t>(emax - a.e + 1), nb = static_cast<uint32_t>(emax - b.e + 1);
    // two's complement, the 32 bits below the unit in `low`
    const uint64_t low = static_cast<uint64_t>(funnel_shr(a.r, static_cast<uint32_t>(a.p), na) ^ a.s) +
                         (funnel_shr(b.r, static_cast<uint32_t>(b.p), nb) ^ b.s) + ((a.s & 1u) + (b.s & 1u));
    const uint64_t acc = (shr_clamp(a.p, na) ^ (static_cast<uint64_t>(a.s) << 32 | a.s)) +
                         (shr_clamp(b.p, nb) ^ (static_cast<uint64_t>(b.s) << 32 | b.s)) + (low >> 32);
    const uint32_t sgn = static_cast<uint32_t>(static_cast<int64_t>(acc) >> 63);
    const uint64_t rest = static_cast<uint64_t>(static_cast<uint32_t>(low) ^ sgn) + (sgn & 1u);
    const uint64_t mag = (acc ^ (static_cast<uint64_t>(sgn) << 32 | sgn)) + (rest >> 32);
    if (mag < (uint64_t(1) << 31)) return (a.p | b.p) ? kahan2_far(x, y, z, t) : 0.0;
    const uint32_t lz = leading_zeros(mag), up = lz - 1u;  // up < 32
    const uint32_t mid = static_cast<uint32_t>(mag);
    const uint64_t m = static_cast<uint64_t>(funnel_shl(mid, static_cast<uint32_t>(mag >> 32), up)) << 32 |
                       funnel_shl(static_cast<uint32_t>(rest), mid, up);  // leading bit at 62
    const uint64_t q = (m + 0x1FFu + ((m >> 10) & 1u)) >> 10;  // 53 bits, ties to even; a carry moves on to the exponent
    return scaled((static_cast<uint64_t>(sgn) << 63) + (static_cast<uint64_t>(1085u - lz) << 52) + q, emax);
}

}  // namespace fx
}  // namespace costa
