// Float64 operations on the integer pipe, bit for bit those of the float64 one.
//
// GB300 issues float64 at 1/74 of the float32 rate -- comparisons and
// conversions included -- so in a kernel bound by the float64 pipe every such
// instruction that a few integer instructions can stand for is better done by
// them.
//
// Quotients.  A float64 quotient is a dozen dependent float64 instructions, and
// the kernels that form face conductances, face velocities and pressures spent
// most of their float64 time on divisions.  With both mantissas as 53-bit
// integers A and B:
//
//   y0 = 24 bits of 1/B from the float32 reciprocal approximation of B's
//        leading 24 bits,
//   y  = y0 (1 + e + e^2), e = 1 - B y0 exactly: Newton's series for the
//        reciprocal to third order, 60 bits in fixed point,
//   Q  = A y truncated, biased down so that it is the quotient's integer part or
//        one less,
//   and the exact remainder A 2^s - Q B (mod 2^64, since it fits) rounds it.
//
// A quotient of two 53-bit integers is never halfway between two 53-bit
// results, so the remainder's comparison with B / 2 is the rounding to nearest
// (Markstein's and every remainder-based division's last step): the bits are
// those of the hardware's a / b and __drcp_rn, checked exhaustively at the
// mantissas' corners and on random pairs.  Operands or results outside the
// normal range (subnormals, infinities, NaN, a zero divisor) take the
// hardware's path; a zero dividend, common in fields at rest, is a zero.
//
// About 65 integer instructions, against seven (reciprocal) and eleven
// (quotient) issue slots of the float64 pipe at 18.5 cycles an SM each.
//
// Sign, finiteness and order of float64 values are those of their bits; a
// conversion between normal float32 and float64 values shifts the mantissa.
#pragma once

#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#define LM_HD __host__ __device__ __forceinline__
#else
#define LM_HD inline
#endif

namespace lm {

// 2^63 / m for m = B / 2^52 in [1, 2), off by less than 2^4, from the bits of
// y0 in [1/2, 1], off from 1 / m by less than 2^-21.
LM_HD uint64_t idiv_recip(uint64_t B, uint32_t y0_bits) {
    // y0 as an integer at scale 2^24
    const uint32_t Y0 = ((y0_bits & 0x7fffffu) | 0x800000u) << ((y0_bits >> 23) - 126u);
    const uint64_t P = (uint64_t)(uint32_t)B * Y0 + ((uint64_t)((uint32_t)(B >> 32) * Y0) << 32);
    const int64_t E = -(int64_t)P;                             // (1 - m y0) 2^76, |E| < 2^55
    const int32_t eh = (int32_t)(E >> 24);
    const int64_t F = E + (((int64_t)eh * eh) >> 28);          // (e + e^2) 2^76
    const int64_t T = ((int64_t)(int32_t)Y0 * (int32_t)(F >> 32) + (int64_t)(((uint64_t)Y0 * (uint32_t)F) >> 32)) >> 5;
    return ((uint64_t)Y0 << 39) + (uint64_t)T;
}

LM_HD uint64_t idiv_mulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
    return __umul64hi(a, b);
#else
    return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}

// Mantissa and exponent of the rounded quotient of normal operands as one
// integer: e 2^52 + Q - 2^52 (Q = 2^53 carries into the exponent); e is the
// biased exponent, valid when 1 <= e <= 2046 before and after.
LM_HD int64_t idiv_core(uint64_t ma, uint64_t mb, int e, uint64_t y) {
    const uint64_t A = ma | (1ull << 52), B = mb | (1ull << 52);
    const int less = A < B;                                    // quotient in (1/2, 1): one more bit
    const uint64_t q62 = idiv_mulhi(A << 11, y) - 16;          // A / B at scale 2^62, low by less than 2^6
    uint64_t Q = q62 >> (10 - less);
    const int64_t rem2 = 2 * (int64_t)((A << (52 + less)) - Q * B);   // twice the remainder, in [0, 4 B)
    Q += (rem2 > (int64_t)B) + (rem2 > (int64_t)(3 * B));
    return ((int64_t)(e - less) << 52) + (int64_t)(Q - (1ull << 52));
}

#ifdef __CUDACC__
// the bits of a computed value, opaque to the compiler, which makes float64
// comparisons of tests on bits that it sees come from float64 arithmetic
__device__ __forceinline__ uint64_t dbits(double v) {
    uint64_t u;
    asm("mov.b64 %0, %1;" : "=l"(u) : "d"(v));
    return u;
}

__device__ __forceinline__ uint32_t idiv_seed(uint64_t m) {
    const float f = __uint_as_float(0x3f800000u | (uint32_t)(m >> 29));
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f));
    return __float_as_uint(fmaxf(r, 0.5f));
}

// a / b, rounded to nearest
__device__ __forceinline__ double idiv(double a, double b) {
    const uint64_t ua = dbits(a), ub = dbits(b);
    const int ea = (int)(ua >> 52) & 0x7ff, eb = (int)(ub >> 52) & 0x7ff, e = ea - eb + 1023;
    const uint64_t M = (1ull << 52) - 1;
    // normal operands and a result that stays normal whichever way it rounds
    if ((unsigned)(ea - 1) < 2046u && (unsigned)(eb - 1) < 2046u && (unsigned)(e - 2) < 2044u) {
        const uint64_t mb = ub & M;
        const int64_t r = idiv_core(ua & M, mb, e, idiv_recip(mb | (1ull << 52), idiv_seed(mb)));
        return __longlong_as_double(r | (int64_t)((ua ^ ub) & (1ull << 63)));
    }
    if (!(ua << 1) && (unsigned)(eb - 1) < 2046u) return __longlong_as_double((long long)((ua ^ ub) & (1ull << 63)));
    return a / b;
}
// 1 / b, rounded to nearest
__device__ __forceinline__ double ircp(double b) { return idiv(1.0, b); }

// v > 0 and finite
__device__ __forceinline__ bool pos_finite(double v) {
    return dbits(v) - 1 < 0x7ff0000000000000ull - 1;
}

// (float)v, rounded to nearest even
__device__ __forceinline__ float to_f32(double v) {
    const uint64_t u = dbits(v), m = u & 0x7fffffffffffffffull;
    // exponents of normal float32 values, one short of the largest so that a
    // carry is one too
    if (m - (897ull << 52) < (1149ull - 897ull + 1) << 52) {
        const uint32_t r = (uint32_t)((m + 0x0fffffffull + ((m >> 29) & 1)) >> 29) - (896u << 23);
        return __uint_as_float(r | (uint32_t)(u >> 32 & 0x80000000u));
    }
    if (!(u << 1)) return __uint_as_float((uint32_t)(u >> 32));
    return (float)v;
}
// (double)v
__device__ __forceinline__ double to_f64(float v) {
    const uint32_t u = __float_as_uint(v), e = u >> 23 & 255u;
    if (e - 1u < 254u)
        return __longlong_as_double((long long)((((uint64_t)(u & 0x7fffffffu) << 29) + (896ull << 52)) |
                                                ((uint64_t)(u & 0x80000000u) << 32)));
    if (!(u << 1)) return __longlong_as_double((long long)((uint64_t)u << 32));
    return (double)v;
}

// v times a factor that is 2^k, or no such power (k = POW2_NONE)
constexpr int POW2_NONE = 0x7fffffff;
// (a call: as an inlined alternative it would be executed, predicated off, for all)
static __device__ __noinline__ double mul_call(double v, double factor) { return v * factor; }
__device__ __forceinline__ double mul_pow2(double v, double factor, int k) {
    const uint64_t u = dbits(v);
    const int e = (int)(u >> 52) & 0x7ff;
    if (k != POW2_NONE && (unsigned)(e - 1) < 2046u && (unsigned)(e + k - 1) < 2046u)
        return __longlong_as_double((long long)u + ((long long)k << 52));
    if (!(u << 1) && k != POW2_NONE) return v;
    return mul_call(v, factor);
}
#endif

// a b > 0 ? (|a| < |b| ? a : b) : 0 on the bits of a and b, the product rounded to
// float64 as the comparison with it would have it (so zero below 2^-1075).  No
// float64 instruction even in the rare case, which a compiler would run for all.
LM_HD uint64_t minmod_bits(uint64_t a, uint64_t b) {
    const uint64_t M = 0x7fffffffffffffffull, ma = a & M, mb = b & M;
    if (!(a << 1) || !(b << 1) || (int64_t)(a ^ b) < 0) return 0;
    if ((uint32_t)(ma >> 32) - 0x20000000u >= 0x5ff00000u || (uint32_t)(mb >> 32) - 0x20000000u >= 0x5ff00000u) {
        const uint64_t inf = 0x7ffull << 52;
        if (ma > inf || mb > inf) return 0;                    // NaN
        if (ma < inf && mb < inf) {
            const int ea = (int)(ma >> 52), eb = (int)(mb >> 52);
            const uint64_t A = (ma & ((1ull << 52) - 1)) | (ea ? 1ull << 52 : 0),
                           B = (mb & ((1ull << 52) - 1)) | (eb ? 1ull << 52 : 0);
            const int t = 1075 - (ea ? ea : 1) - (eb ? eb : 1);   // a b = A B 2^(-1075 - t)
            if (t > 106) return 0;
            if (t >= 0 && (unsigned __int128)A * B <= (unsigned __int128)1 << t) return 0;
        }
    }
    return ma < mb ? a : b;
}

// ---- exact stencil sums ---------------------------------------------------------
//
// sum_o g_o (x_c - x_o) over neighbours of a cell, in integers.  The x become
// integers at one scale, of 53 + XB bits where the largest x has its leading one,
// and the weights likewise with GB; both as limbs h 2^29 + l, the x with their sign
// on both limbs, so that differences and sums of weights need no carry.  Products
// accumulate exactly in three 64-bit sums, four widening multiply-adds a term, and
// the total is rounded once to float64.
//
// Precision.  Where the nonzero x lie within 2^XB of each other and the weights
// within 2^GB the sum is exact before its one rounding; float64 rounds every
// difference, product and partial sum.  An x further down is cut off at 2^-(52 + XB)
// of the largest, E: a term is off by less than 2^-(51 + XB) g E.  Then some
// difference is at least E / 2 in magnitude, and the float64 form rounds it, its
// product and the partial sums after that by up to 2^-53 of them each -- with XB = 5
// 8 times the cut for as large a weight.  So x of any spread are taken where the
// weights lie within a factor of four; all else takes the float64 form.  E has to
// be the centre's or one that some weight meets: the centre's value stands for a
// neighbour without weight (past a wall), whose size would cut the others off.
// Where classes of neighbours have factors of their own, E has to be, but for one
// bit, the centre's or one of a strong class, with a factor within four of the
// largest: if it is the centre's, a cut x is in a difference of about E itself;
// if not, the difference that holds E has a factor to match every cut one's.
//
// Room: |xl|, |xh| < 2^29 with XB <= 5, so differences < 2^30; gl < 2^29 and
// gh < 2^(24 + GB) <= 2^28.  Six single weights, or FE's sums of two (four terms) and
// four (two terms) with GB = 3, keep each sum below 2^62.5.

// range of the nonzero magnitudes, by their high words
struct ExpRange {
    uint32_t hi = 0, lo = 0xffffffffu;      // largest; smallest nonzero, less one
    LM_HD void add(uint32_t h) {            // h: high word without its sign
        hi = h > hi ? h : hi;
        lo = h - 1u < lo ? h - 1u : lo;
    }
    LM_HD int top() const { return (int)(hi >> 20); }
    LM_HD int spread() const { return (int)(hi >> 20) - (int)((lo + 1u) >> 20); }
};
// both ranges in reach, and the sum's exponent in the normal range however far
// its terms cancel (zeros are below every scale: 2^200 over the smallest normal);
// strong: the range of the centre and the strong classes
LM_HD bool fix_ok(const ExpRange& x, int xb, const ExpRange& g, int gb, const ExpRange& strong) {
    const int ex = x.top(), eg = g.top(), sg = g.spread();
    return ex >= 200 && ex < 2047 && eg >= 200 && eg < 2047 && sg <= gb &&
           (x.spread() <= xb || (sg <= 1 && strong.top() >= ex - 1)) && (unsigned)(ex + eg - 1023 - 150) < 1880u;
}
LM_HD bool fix_ok(const ExpRange& x, int xb, const ExpRange& g, int gb) { return fix_ok(x, xb, g, gb, x); }
// x of a neighbour of weight w (the bits of one, or of all of several, or-ed), or
// the centre's c where that is zero: the term stays zero.  An infinity or NaN stays:
// it times zero is NaN.
LM_HD uint64_t fix_live(uint64_t x, uint64_t w, uint64_t c) {
    return (w << 1) || (x >> 52 & 0x7ff) == 0x7ff ? x : c;
}
struct Limbs {
    int32_t h, l;
};
// |v| of the value's bits at scale 2^(52 + B) over exponent `top`
template <int B>
LM_HD Limbs fix_abs(uint64_t u, int top) {
    const int sh = top - ((int)(u >> 52) & 0x7ff);
    const uint64_t m = (((u & ((1ull << 52) - 1)) | (1ull << 52)) << B) >> (sh > 63 ? 63 : sh);
    return {(int32_t)(uint32_t)(m >> 29), (int32_t)((uint32_t)m & 0x1fffffffu)};
}
template <int B>
LM_HD Limbs fix(uint64_t u, int top) {
    const Limbs a = fix_abs<B>(u, top);
    const int32_t s = (int32_t)((int64_t)u >> 63) | 1;
    return {a.h * s, a.l * s};
}
// c - v
template <int B>
LM_HD Limbs fix_diff(Limbs c, uint64_t u, int top) {
    const Limbs a = fix_abs<B>(u, top);
    const int32_t s = ~(int32_t)((int64_t)u >> 63) | 1;
    return {c.h + a.h * s, c.l + a.l * s};
}
struct FixSum {
    int64_t a0 = 0, a1 = 0, a2 = 0;         // weights 1, 2^29, 2^58
    LM_HD void mac(Limbs d, Limbs g) {
        a0 += (int64_t)d.l * g.l;
        a1 += (int64_t)d.l * g.h;
        a1 += (int64_t)d.h * g.l;
        a2 += (int64_t)d.h * g.h;
    }
    LM_HD __int128 total() const { return ((__int128)a2 << 58) + ((__int128)a1 << 29) + a0; }
};
// t rounded to float64, as bits; e: the exponent field of 2^0 at t's scale
LM_HD uint64_t fix_round(__int128 t, int e) {
    const uint64_t s = (uint64_t)((int64_t)(t >> 64) >> 63);
    uint64_t lo = (uint64_t)t ^ s, hi = (uint64_t)(t >> 64) ^ s;
    lo -= s;
    hi += s & (uint64_t)(lo == 0);
    if (!hi) {                               // |t| < 2^64
        if (!lo) return 0;
        hi = lo;
        lo = 0;
        e -= 64;
    }
#ifdef __CUDA_ARCH__
    const int z = __clzll((long long)hi);
#else
    const int z = __builtin_clzll(hi);
#endif
    uint64_t m = hi << z | (lo >> 1) >> (63 - z);
    m |= (uint64_t)(lo << z != 0);
    m = (m >> 11) + (((m & 0x7ff) + 0x3ff + ((m >> 11) & 1)) >> 11);
    return (m + ((uint64_t)(e + 126 - z) << 52)) | (s & (1ull << 63));
}
// the exponent field of 2^0 at the scale of a sum of x (top ex) times g (top eg)
template <int XB, int GB>
LM_HD int fix_scale(int ex, int eg) {
    return ex + eg - 1023 - 104 - XB - GB;
}

// the exponent k of a factor 2^k, else POW2_NONE (host)
inline int pow2_of(double f) {
    int e = 0;
    return f > 0.0 && f < 1e300 && frexp(f, &e) == 0.5 && e > -1000 && e < 1000 ? e - 1 : 0x7fffffff;
}

}  // namespace lm
