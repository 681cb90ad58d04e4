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
//   links   U 2^lsh, one scale per field: 60 for SU(3) links (|U_ab| <= 1),
//           58 - u for |U_ab| < 2^u otherwise
//   clover  A 2^(60 - a), a per site, |A_ij| < 2^a
// A spinor component thus keeps 57 bits below its site's largest one (FP64 keeps
// 53 below itself).  A half spinor is the sum or difference of two components
// limb by limb, so its limbs are one bit longer, |lo| <= 2^30, and may be
// negated.  The sums stay below 2^63: per component of a colour product
// |sum hi hi| <= 6 2^30 2^28 and |sum cross| <= sqrt(6) 2^30 2^30 + 6 2^29 2^28
// < 3.3 2^60 for SU(3) rows (less for the other scale); the hop sum of eight
// directions, each at most sqrt(6) 2^58, is below 19.6 2^58 < 2^62.3; the clover
// sums of eleven products are below 11 (2^59 + 2^56) < 2^62.7.
//
// A site with a non-finite component, or with its largest exponent near the
// ends of FP64's range, keeps its FP64 components as they are (its exponent is
// marked kFxRaw), and every site that reads one is computed in FP64.
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
constexpr int kFxSpinorBits = 57, kFxCloverBits = 60;

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
// the sum over 2^60, rounded
__device__ __forceinline__ int64_t fx_value(const fxacc &s) { return s.h + ((s.c + (1ll << (kFxLimb - 1))) >> kFxLimb); }

// v 2^ex in FP64 (v's leading 53 bits, rounded; the result is a normal number or zero)
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
// 2^(emax - 1022), emax an exponent field at least its own
__device__ __forceinline__ int64_t fx_from_bits(uint32_t hi, uint32_t lo, int emax, int bits)
{
    const int ex = (int)((hi >> 20) & 0x7ff);
    // 53-bit mantissa (subnormal numbers, far below any site's scale here, count as zero)
    const uint64_t m = ex ? ((uint64_t)((hi & 0x000fffffu) | 0x00100000u) << 32 | lo) : 0;
    const int d = emax - ex;
    const uint64_t x = d > 63 ? 0 : (m << (bits - 53)) >> d;
    return (int32_t)hi < 0 ? -(int64_t)x : (int64_t)x;
}

__device__ __forceinline__ fx fx_from_double(double v, int emax, int bits)
{
    return fx_split(fx_from_bits((uint32_t)__double2hiint(v), (uint32_t)__double2loint(v), emax, bits));
}

__device__ __forceinline__ int fx_exponent(double v) { return (int)(((uint32_t)__double2hiint(v) >> 20) & 0x7ff); }

// The 12 components v of a site into the fixed-point field f (planes of the
// domain block at blk) and its exponent.
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
        int4 w;
        if (raw) {
            w = make_int4(__double2loint(v[k].re), __double2hiint(v[k].re), __double2loint(v[k].im),
                          __double2hiint(v[k].im));
        } else {
            const fx a = fx_from_double(v[k].re, emax, kFxSpinorBits), b = fx_from_double(v[k].im, emax, kFxSpinorBits);
            w = make_int4(a.hi, a.lo, b.hi, b.lo);
        }
        blk[(int64_t)k * Vd + s] = w;
    }
}

}  // namespace qdd
