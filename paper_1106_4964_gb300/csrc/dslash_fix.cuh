// Hopping term of FP64 and double-float fields in block fixed point on the integer pipes.
//
// GB300 issues 2 FP64 operations per clock and SM against 128 FP32 or 64 integer ones, and a
// double-float multiply-add is 18 FP32 operations, so a hop's 72 multiply-adds are its cost.  Here each
// projected half spinor h (12 reals, formed in the field's arithmetic) is written as 64-bit integers in
// units of 2^-60 of the power of two above its largest component, the link as 64-bit integers in units
// of 2^-62, and the colour multiply sums 32 x 32 -> 64-bit products: with x = x1 2^32 + x0, x0 in
// [-2^31, 2^31),
//   u h / 2^64 = u1 h1 + (u1 h0 + u0 h1) / 2^32 + (u0 h0) / 2^64,
// the last term below the unit of the result and dropped, the sum rounded to nearest; zeros stay exactly zero.
// The sum over the eight hops is a 64-bit integer in units of 2^-58 of the power of two above the largest
// component met.  Relative to a hop's largest component, cut conversions cost at most sqrt(6) 2^-59, dropped
// terms 6 x 2^-59 and the rounding 2^-58: below 2^-55 together (2^-58 in the root mean square), where FP64
// rounds every product and partial sum to 2^-53 of itself: relative to the field around the site the sum's
// error is that of the floating-point sum or smaller.
//
// Bounds (|u row| = 1 to 1e-9, |h| < 2^60): sum of |u1 h0| <= sqrt(6) 2^61, sum of |u0 h1| <=
// 6 x 2^59, together below 2^63; the sum of u1 h1 stays below 2^60; a hop's result is below
// 2.45 x 2^58, the sum of eight below 2^62.3.
//
// Where links mix colours, that error lies below the rounding of the larger products in every component.  Where
// they do not (a free field, block-diagonal links, one filled colour) a component can be far below the largest
// one and floating point would still hold it to all its bits.  So a complex component of which the sum and all
// eight hops' parts are below 2^-FIX_KEEP of the scale, exact zeros among them, is formed again from its own
// products in the field's arithmetic with the links in FP64 (fix_small).  (A small sum of larger parts is
// left: floating point rounds the parts as well.)  What stays has an error of at most 8 x 3.6 units of 2^-58
// of the scale, 2^FIX_KEEP times which its largest part is: 2^-47 of that in FP64, 2^-44 in double-float, some
// 2^-51 in the root mean square.  Largest error of a component in units of 2^-53 of its |u| |h|, FP64 sums /
// this form: Gaussian fields on mixing links 1.4 / 0.9, components spread over 2^12 on diagonal links 3.1 / 2.7,
// sites spread over 2^80 there 5.2 / 10.9.  24^3 x 64, us per launch without and with it: FP64 427 / 436,
// double-float (which needs no range checks any more) 613 / 600; 12 point sources' solve at 8^4 with FP64
// residuals, whose fields have such components, 337 / 351 ms (a test of the sum alone would make it 510).
//
// What the format does not hold at all goes to the field's own arithmetic, block by block: infinities, NaN,
// values near the ends of the exponent range.
#pragma once

#include <stdint.h>

namespace ov {

struct Fix {
    int h, l;  // value = h 2^32 + l
};

__host__ __device__ __forceinline__ uint32_t fix_shr(uint32_t hi, uint32_t lo, uint32_t n)
{
    // low word of (hi : lo) >> min(n, 32)
#ifdef __CUDA_ARCH__
    return __funnelshift_rc(lo, hi, n);
#else
    const uint64_t v = ((uint64_t)hi << 32) | lo;
    return (uint32_t)(v >> (n < 32 ? n : 32));
#endif
}

__host__ __device__ __forceinline__ unsigned long long fix_shr64(unsigned long long x, uint32_t n)
{
    // x >> n, 0 for n >= 64
#ifdef __CUDA_ARCH__
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
#else
    return n < 64 ? x >> n : 0;
#endif
}

__host__ __device__ __forceinline__ uint32_t f64_hi(double x)
{
#ifdef __CUDA_ARCH__
    return (uint32_t)__double2hiint(x);
#else
    uint64_t b;
    __builtin_memcpy(&b, &x, 8);
    return (uint32_t)(b >> 32);
#endif
}
__host__ __device__ __forceinline__ uint32_t f64_lo(double x)
{
#ifdef __CUDA_ARCH__
    return (uint32_t)__double2loint(x);
#else
    uint64_t b;
    __builtin_memcpy(&b, &x, 8);
    return (uint32_t)b;
#endif
}
__host__ __device__ __forceinline__ double f64_bits(uint32_t hi, uint32_t lo)
{
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)hi, (int)lo);
#else
    const uint64_t b = ((uint64_t)hi << 32) | lo;
    double x;
    __builtin_memcpy(&x, &b, 8);
    return x;
#endif
}

constexpr uint32_t FIX_EXP = 0x7ff00000u;        // exponent field of a double's high word
constexpr uint32_t FIX_ELO = 200u << 20;         // exponents the fixed-point path takes
constexpr uint32_t FIX_EHI = 1900u << 20;
constexpr int FIX_KEEP = 6, FIXD_KEEP = 9;       // components below 2^-KEEP of the scale are formed again

// x >> n, arithmetic (any n)
__host__ __device__ __forceinline__ long long fix_sar(long long x, uint32_t n)
{
#ifdef __CUDA_ARCH__
    long long r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
    return r;
#else
    return x >> (n < 63 ? n : 63);
#endif
}

// a component of the sum below 2^-keep of the scale (2^58 units), both parts: its high words within 2^(26 - keep)
__host__ __device__ __forceinline__ bool fix_small(long long re, long long im, int keep)
{
    const uint32_t t = 1u << (26 - keep);
    return (uint32_t)(re >> 32) + t < 2 * t && (uint32_t)(im >> 32) + t < 2 * t;
}

// x in units of 2^-60 of the power of two above a component of exponent field emax >= f.  Negative values are
// complemented: one unit low.
__host__ __device__ __forceinline__ Fix to_fix(double x, uint32_t emax)
{
    const uint32_t hw = f64_hi(x), lw = f64_lo(x), f = hw & FIX_EXP;
    uint32_t mh = fix_shr(hw, lw, 21) | 0x80000000u;  // 53-bit mantissa, left-aligned in mh : ml
    uint32_t sg = (uint32_t)((int)hw >> 31);
    const uint32_t ml = lw << 11;
    if (f == 0) mh = sg = 0;  // zero (a subnormal is below any unit the path uses)
    const unsigned long long m = fix_shr64(((unsigned long long)mh << 32) | ml, 4u + ((emax - f) >> 20));
    const uint32_t hi = (uint32_t)(m >> 32) ^ sg, lo = (uint32_t)m ^ sg;
    Fix r;
    r.l = (int)lo;
    r.h = (int)(hi + (lo >> 31));
    return r;
}

// -x, exactly (a low word of -2^31 counts as -2^31 + 1).  Zero stays zero: a complement would leave one unit in
// every vanishing product, and fields that are exactly zero in some colours or spins (a free field's point
// source) would fill with noise there.
__host__ __device__ __forceinline__ Fix fix_neg(Fix x) { return Fix{-x.h, -(x.l > -2147483647 ? x.l : -2147483647)}; }
// x or -x for m = 0 or -1; the low word of a link is never -2^31 (link_to_fix)
__host__ __device__ __forceinline__ Fix fix_sign(Fix x, int m) { return Fix{(x.h ^ m) - m, (x.l ^ m) - m}; }

// links: |u| <= 1 in units of 2^-62
__host__ __device__ __forceinline__ Fix link_to_fix(double u)
{
    const long long q = (long long)rint(u * 4611686018427387904.0);
    Fix r;
    r.l = (int)(uint32_t)q;
    r.h = (int)((q - (long long)r.l) >> 32);
    if (r.l == -2147483647 - 1) r.l = -2147483647;  // one unit: fix_sign
    return r;
}

struct FixProd {
    long long hi, mid;
};
__host__ __device__ __forceinline__ void fix_mac(FixProd& s, Fix a, Fix b)
{
    s.hi += (long long)a.h * b.h;
    s.mid += (long long)a.h * b.l;
    s.mid += (long long)a.l * b.h;
}
__host__ __device__ __forceinline__ long long fix_sum(const FixProd& s)
{
    return s.hi + ((s.mid + 0x80000000ll) >> 32);  // |mid| stays below 2^63 - 2^31
}

// Exponent field of the largest of the 12 components (0: every component is zero or subnormal), FIX_BAD
// when the format does not hold them
constexpr uint32_t FIX_BAD = 0xffffffffu;
__host__ __device__ __forceinline__ uint32_t fix_range(const double h[12])
{
    uint32_t emax = 0;
#pragma unroll
    for (int i = 0; i < 12; ++i) {
        const uint32_t f = f64_hi(h[i]) & FIX_EXP;
        emax = emax > f ? emax : f;
    }
    if (emax == 0) {
        uint32_t any = 0;
#pragma unroll
        for (int i = 0; i < 12; ++i) any |= (f64_hi(h[i]) << 1) | f64_lo(h[i]);
        return any ? FIX_BAD : 0u;
    }
    return emax >= FIX_EHI || emax < FIX_ELO ? FIX_BAD : emax;
}

// v 2^-1080 2^e (e: exponent field >> 20 of the sum's unit), rounded to nearest
__host__ __device__ __forceinline__ int fix_clz(unsigned long long m)
{
#ifdef __CUDA_ARCH__
    return __clzll((long long)m);
#else
    return m ? __builtin_clzll(m) : 64;
#endif
}
__host__ __device__ __forceinline__ double fix_to_f64(long long v, int e)
{
    const unsigned long long sg = (unsigned long long)(v >> 63);
    unsigned long long m = ((unsigned long long)v ^ sg) - sg;
    const int lz = fix_clz(m);
    m = lz < 64 ? m << lz : 0ull;
    // m 2^-63 in [1, 2): exponent of the value 63 - lz + e - 1080
    const unsigned long long r = (m >> 11) + ((m >> 10) & 1ull);
    const unsigned long long bits =
        r + ((unsigned long long)(uint32_t)(63 - lz + e - 1080 + 1023 - 1) << 52);
    return lz < 64 ? f64_bits((uint32_t)(bits >> 32) | ((uint32_t)sg & 0x80000000u), (uint32_t)bits) : 0.0;
}

// ---- double-float: exponent fields are those of the high words (8 bits at bit 23) ----
constexpr uint32_t FIXD_EXP = 0x7f800000u;
constexpr uint32_t FIXD_ELO = 74u << 23;
constexpr uint32_t FIXD_EHI = 250u << 23;

__host__ __device__ __forceinline__ uint32_t f32_bits(float x)
{
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    uint32_t b;
    __builtin_memcpy(&b, &x, 4);
    return b;
#endif
}
__host__ __device__ __forceinline__ float bits_f32(uint32_t b)
{
#ifdef __CUDA_ARCH__
    return __uint_as_float(b);
#else
    float x;
    __builtin_memcpy(&x, &b, 4);
    return x;
#endif
}

__host__ __device__ __forceinline__ uint32_t fixd_range(const float hi[12], const float lo[12])
{
    uint32_t emax = 0;
#pragma unroll
    for (int i = 0; i < 12; ++i) {
        const uint32_t f = f32_bits(hi[i]) & FIXD_EXP;
        emax = emax > f ? emax : f;
    }
    if (emax == 0) {
        uint32_t any = 0;
#pragma unroll
        for (int i = 0; i < 12; ++i) any |= (f32_bits(hi[i]) | f32_bits(lo[i])) << 1;
        return any ? FIX_BAD : 0u;
    }
    return emax >= FIXD_EHI || emax < FIXD_ELO ? FIX_BAD : emax;
}

__host__ __device__ __forceinline__ Fix fixd_to_fix(float xh, float xl, uint32_t emax)
{
    const uint32_t hb = f32_bits(xh), lb = f32_bits(xl), f = hb & FIXD_EXP, fl = lb & FIXD_EXP;
    uint32_t m = ((hb << 4) & 0x07fffff0u) | 0x08000000u;  // 24-bit mantissa, units of 2^32 below 2^60
    uint32_t sg = (uint32_t)((int)hb >> 31);
    if (f == 0) m = sg = 0;
    const unsigned long long mm = fix_shr64((unsigned long long)m << 32, (emax - f) >> 23);
    long long x = (long long)(mm ^ (unsigned long long)(long long)(int)sg);
    // low word: 24 bits from 2^15 units up (2^-21 of the hop's largest component: a pair whose low word exceeds
    // half a unit of its high word by a few bits is taken too), cut at one unit
    // (a zero's exponent field shifts all of it out)
    const unsigned long long l =
        fix_shr64((unsigned long long)((lb & 0x007fffffu) | 0x00800000u) << 15, ((emax - fl) >> 23) - 21u);
    const long long sl = (long long)((int)lb >> 31);
    x += (long long)(l ^ (unsigned long long)sl) - sl;
    Fix r;
    r.l = (int)(uint32_t)x;
    r.h = (int)((uint32_t)(x >> 32) + ((uint32_t)r.l >> 31));
    return r;
}

// v 2^-184 2^e as a normalised pair (24 + 24 significand bits), rounded to nearest
__host__ __device__ __forceinline__ void fixd_from_fix(long long v, int e, float& hi, float& lo)
{
    const unsigned long long sg = (unsigned long long)(v >> 63);
    unsigned long long m = ((unsigned long long)v ^ sg) - sg;
    const int lz = fix_clz(m);
    m = lz < 64 ? m << lz : 0ull;
    const int ex = 63 - lz + e - 184 + 127;  // biased exponent of the value
    const uint32_t s = (uint32_t)sg & 0x80000000u;
    const uint32_t top = (uint32_t)(m >> 32);
    const float h0 = bits_f32(((uint32_t)ex << 23) + ((top >> 8) & 0x007fffffu) | s);
    // the next 32 bits, rounded to nearest as they become a float (cut, every sum would come out short by 2^-48 on
    // average, and a chain of applications shrinks with it)
    const uint32_t rest = (uint32_t)(m >> 8);
    // 2^(value exponent - 23), one unit of h0's last place; below the normal range (a sum far below hops that
    // are themselves near the end of the range) the low word is nothing
    const float u = bits_f32(ex > 23 ? (uint32_t)(ex - 23) << 23 : 0u);
    const float l0 = (float)rest * 2.3283064365386962890625e-10f * (s ? -u : u);
    if (lz >= 64) {
        hi = lo = 0.f;
        return;
    }
    hi = h0 + l0;
    lo = l0 - (hi - h0);
}

}  // namespace ov
