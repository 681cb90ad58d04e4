// FP64-class arithmetic of the full-lattice operator in 64-bit fixed point.
//
// This GPU runs an FP64 multiply-add at 2 lanes per clock and SM and a
// 32x32+64-bit integer multiply-add at about 60.  A value is therefore kept as
// a fixed-point integer of up to 60 bits in two signed limbs, v = hi 2^30 + lo
// with |lo| <= 2^29, and a product is accumulated with three integer
// multiply-adds (hi hi, hi lo + lo hi; the lo lo part, below the last bit kept,
// is dropped):  a b = 2^60 (hi hi + 2^-30 (hi lo + lo hi)).
//
// Scales are powers of two:
//   spinor  x 2^(57 - e), e per site, |x| < 2^e for all 24 reals of the site
//   links   U 2^(60 - u), u per field: |U_ab| < 2^u (u = 0, |U_ab| <= 1, for SU(3)),
//           and |Re| + |Im| summed over a row or a column at most kFxLinkRow 2^u
//           (sqrt 6 for a unitary one)
//   clover  A 2^(60 - a), a per site: |A_ij| < 2^a, and |Re| + |Im| summed over a row
//           at most kFxCloverRow 2^a
// A spinor component thus keeps 57 bits below its site's largest one (FP64 keeps
// 53 below itself).  A half spinor is the sum or difference of two components
// limb by limb, so its limbs are one bit longer, |lo| <= 2^30, and may be
// negated.  The sums stay below 2^63: per component of a colour product
// |sum hi hi| <= 6 2^30 2^28 and |sum cross| <= sqrt(6) 2^30 2^30 + 6 2^29 2^28
// < 3.3 2^60; the hop sum of eight directions, each at most sqrt(6) 2^58, is below
// 19.6 2^58 < 2^62.3; the clover sums of eleven products are below
// 11 (2^59 + 2^56) < 2^62.7.
//
// The error of a component y of D x belongs to these scales.  With E the largest
// exponent of the nine sites and Q = 2^(E + u - 57), a hop's component is off by at
// most sqrt(6) Q (rounded spinors), 0.75 Q (rounded links), 3 Q (products of lower
// limbs left out), 0.5 Q (rounding) and Q (shift to E): eight hops by 62 Q =
// 2^(E + u - 51.05).  The clover sum, with q = 2^(e + a - 57): 0.6 q (spinors), 0.7 q
// (A), 2.75 q (lower limbs), 0.5 q: 2^(e + a - 54.8).  FP64 arithmetic rounds a hop's
// six multiply-adds, the projection before and the sum of eight after them, by up
// to 15 2^-53 S, S the sum of the moduli of the products U h.  So a component is
// as good as FP64's where
//   S >= kFxHop 2^(E + u) + kFxClover 2^(e + a) / |kappa|,
// which the leading bits of links and half spinors show (k_dslash_fx); a site with
// any component below is computed in FP64.  Of 65536 sites the smallest S is 2.1
// times that with Gaussian spinors, and 1.4 times with the Schwarz method's second
// direction, on links of eps = 0.5 and 0.7.
//
// A site with a non-finite component, or with its largest exponent near the
// ends of FP64's range, is marked kFxRaw in place of its exponent, and every site
// that reads one is computed in FP64.
#pragma once

#include "common.cuh"

namespace qdd {

struct fx {
    int hi, lo;
};
struct cfx {
    fx re, im;
};

constexpr int kFxRaw = 1 << 20;     // exponent mark of a site kept in FP64
constexpr int kFxZero = -900;       // exponent of an all-zero site
constexpr int kFxLimb = 30;         // bits of the lower limb
constexpr int kFxSpinorBits = 57, kFxCloverBits = 60, kFxLinkBits = 60;
constexpr float kFxLinkRow = 2.4495f, kFxCloverRow = 1.25f;
constexpr float kFxHop = 0.26f, kFxClover = 0.02f;

// the smallest e with v <= 2^e (v >= 0; infinity and NaN give 128 and more)
__device__ __forceinline__ int fx_ceil_exponent(float v)
{
    const uint32_t b = __float_as_uint(v);
    return (int)(b >> 23) - 127 + ((b & 0x007fffffu) ? 1 : 0);
}

__device__ __forceinline__ fx fx_split(int64_t v)
{
    const int hi = (int)((v + (1ll << (kFxLimb - 1))) >> kFxLimb);
    return {hi, (int)((uint32_t)v - ((uint32_t)hi << kFxLimb))};
}
__device__ __forceinline__ int64_t fx_join(fx v) { return ((int64_t)v.hi << kFxLimb) + v.lo; }

struct fxacc {
    int64_t h, c;
};
__device__ __forceinline__ void fx_mac(fxacc &s, fx a, fx b)
{
    s.h += (int64_t)a.hi * b.hi;
    s.c += (int64_t)a.hi * b.lo;
    s.c += (int64_t)a.lo * b.hi;
}
// s[k] += a x_k for four x
__device__ __forceinline__ void fx_mac4(fxacc *s, fx a, fx x0, fx x1, fx x2, fx x3)
{
    const fx x[4] = {x0, x1, x2, x3};
#pragma unroll
    for (int k = 0; k < 4; k++) s[k].h += (int64_t)a.hi * x[k].hi;
#pragma unroll
    for (int k = 0; k < 4; k++) s[k].c += (int64_t)a.hi * x[k].lo;
#pragma unroll
    for (int k = 0; k < 4; k++) s[k].c += (int64_t)a.lo * x[k].hi;
}
__device__ __forceinline__ void fx_mac2(fxacc &s0, fxacc &s1, fx a, fx x0, fx x1)
{
    s0.h += (int64_t)a.hi * x0.hi;
    s1.h += (int64_t)a.hi * x1.hi;
    s0.c += (int64_t)a.hi * x0.lo;
    s1.c += (int64_t)a.hi * x1.lo;
    s0.c += (int64_t)a.lo * x0.hi;
    s1.c += (int64_t)a.lo * x1.hi;
}
// an empty sum (half a unit of the result, so that fx_value rounds), and the
// sum over 2^60
__device__ __forceinline__ fxacc fx_zero() { return {0, 1ll << (kFxLimb - 1)}; }
__device__ __forceinline__ int64_t fx_value(const fxacc &s) { return s.h + (s.c >> kFxLimb); }

// v 2^ex in FP64 (v's leading 53 bits, rounded; the result is a normal number or
// zero: -1022 <= ex <= 960, which the callers' ranges of scales ensure)
__device__ __forceinline__ double fx_to_double(int64_t v, int ex)
{
    if (v == 0) return 0.0;
    const uint32_t sign = (uint32_t)(v >> 32) & 0x80000000u;
    uint64_t m = (uint64_t)(v < 0 ? -v : v);
    const int lz = __clzll((long long)m);
    m <<= lz;                                     // leading one at bit 63: value m 2^(ex - lz)
    const uint64_t bits = (m >> 11) + ((m >> 10) & 1);  // bit 52 set, or 2^53 after the rounding
    const uint64_t r = bits + ((uint64_t)(uint32_t)(ex - lz + 63 + 1023 - 1) << 52);
    return __hiloint2double((int)((uint32_t)(r >> 32) | sign), (int)(uint32_t)r);
}

// the FP64 number with bits (hi, lo) as an integer with `bits` bits below
// 2^(emax - 1022), rounded, emax an exponent field at least its own
__device__ __forceinline__ int64_t fx_from_bits(uint32_t hi, uint32_t lo, int emax, int bits)
{
    const int ex = (int)((hi >> 20) & 0x7ff);
    // 53-bit mantissa (subnormal numbers, far below any site's scale here, count as zero)
    const uint64_t m = ex ? ((uint64_t)((hi & 0x000fffffu) | 0x00100000u) << 32 | lo) : 0;
    const int d = emax - ex;
    const uint64_t x = d > 63 ? 0 : ((m << (bits - 53)) + ((1ull << d) >> 1)) >> d;  // (bits <= 60: no carry lost)
    return (int32_t)hi < 0 ? -(int64_t)x : (int64_t)x;
}

__device__ __forceinline__ fx fx_from_double(double v, int emax, int bits)
{
    return fx_split(fx_from_bits((uint32_t)__double2hiint(v), (uint32_t)__double2loint(v), emax, bits));
}

__device__ __forceinline__ int fx_exponent(double v) { return (int)(((uint32_t)__double2hiint(v) >> 20) & 0x7ff); }

// ---- FP64 vectors
//
// A group of FP64 numbers that share one scale, the largest exponent field.
// fx_group_done: false unless the group has a fixed-point form whose products
// with another such group are normal FP64 numbers (finite, exponents within
// +-400, or all zero).
struct fxgroup {
    uint32_t top, any;  // largest high word without sign, the bits set in any word
    int emax;
};
__device__ __forceinline__ void fx_group_add(fxgroup &g, double2 v)
{
    const uint32_t a = (uint32_t)__double2hiint(v.x) & 0x7fffffffu, b = (uint32_t)__double2hiint(v.y) & 0x7fffffffu;
    g.top = max(g.top, max(a, b));
    g.any |= (uint32_t)__double2loint(v.x) | (uint32_t)__double2loint(v.y);
}
__device__ __forceinline__ bool fx_group_done(fxgroup &g)
{
    g.emax = (int)(g.top >> 20);
    if ((g.top | g.any) == 0u) g.emax = 1023;  // all zero: every number is far below the scale
    return g.emax > 623 && g.emax < 1423;
}

__device__ __forceinline__ bool fx_group_zero(const fxgroup &g) { return (g.top | g.any) == 0u; }

// shifts by 32 and more give 0
__device__ __forceinline__ uint32_t shr_clamp(uint32_t v, uint32_t n)
{
    uint32_t r;
    asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(n));
    return r;
}

// A number of a group (exponent field at most emax, emax > 600) with `kBits`
// bits below 2^(emax - 1022), 36 < kBits <= 60, rounded towards zero, the limb below
// centred, |lo| <= 2^29 (and |hi| <= 2^(kBits - 30)); lead: its leading six bits.
// (Subnormal numbers and zeros are shifted out.)
template <int kBits>
__device__ __forceinline__ fx fx_centred(double v, int emax, uint32_t &lead)
{
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const uint32_t t = __funnelshift_l(lo, hi, 11) | 0x80000000u, r = lo << 11;  // mantissa, leading one on top
    const uint32_t sh = (uint32_t)(emax + (64 - kBits)) - ((hi >> 20) & 0x7ffu); // magnitude = (t:r) >> sh
    const uint32_t mh = shr_clamp(t, sh - (32 - kFxLimb));
    const uint32_t ml = (sh < 32 ? __funnelshift_r(r, t, sh) : shr_clamp(t, sh - 32)) & ((1u << kFxLimb) - 1);
    const uint32_t up = ml >> (kFxLimb - 1);
    lead = mh >> (kBits - kFxLimb - 6);
    const int sg = ((int)hi >> 31) | 1;
    return {(int)(mh + up) * sg, (int)(ml - (up << kFxLimb)) * sg};
}

// The 12 components v of a site into the fixed-point field f (planes of the
// domain block at blk) and its exponent (a raw site's components are not read).
__device__ __forceinline__ void fx_store_site(int4 *blk, int s, int Vd, int *e_out, const cpx<double> *v)
{
    int emax = 0;
    uint32_t any = 0;
#pragma unroll
    for (int k = 0; k < 12; k++) {
        emax = max(emax, max(fx_exponent(v[k].re), fx_exponent(v[k].im)));
        any |= ((uint32_t)__double2hiint(v[k].re) | (uint32_t)__double2hiint(v[k].im)) & 0x7fffffffu;
        any |= (uint32_t)__double2loint(v[k].re) | (uint32_t)__double2loint(v[k].im);
    }
    const bool zero = any == 0;
    const bool raw = !zero && (emax < 123 || emax > 1923);
    *e_out = zero ? kFxZero : (raw ? kFxRaw : emax - 1022);
#pragma unroll
    for (int k = 0; k < 12; k++) {
        const fx a = fx_from_double(v[k].re, emax, kFxSpinorBits), b = fx_from_double(v[k].im, emax, kFxSpinorBits);
        blk[(int64_t)k * Vd + s] = make_int4(a.hi, a.lo, b.hi, b.lo);
    }
}

}  // namespace qdd
