// Shared device-side definitions of libqdd: complex arithmetic, storage
// precisions, the domain-blocked field layout and the spin algebra of the
// Wilson-clover operator (arXiv:1502.04025, Sec. 3.1-3.2).
//
// Device layout of every lattice field (Sec. 3.2 chooses a layout for the
// domain-decomposed algorithm; this one is chosen for coalesced GPU access
// and for one contiguous block per domain, so a domain stages with a single
// bulk copy):
//   domain slot d  : colour-major, d = colour*(Nd/2) + (block index >> 1)
//   site slot s    : parity-split within the domain, s = parity*(Vd/2) + (l >> 1),
//                    l the domain-local lexicographic index
//   element        : plane-major per domain, field[(d*planes + p)*Vd + s],
//                    one complex number per plane entry
// Planes: spinor 12 (p = spin*3 + colour); links 36 (p = mu*9 + a*3 + b);
// clover 36 (18 per chirality block: 3 pairs of real diagonal entries, then
// the 15 upper off-diagonal entries row by row).
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace qdd {

// ------------------------------------------------------------------ complex

template <typename R>
struct cpx {
    R re, im;
};

template <typename R>
__host__ __device__ __forceinline__ cpx<R> mk(R a, R b) { return cpx<R>{a, b}; }
template <typename R>
__device__ __forceinline__ cpx<R> operator+(cpx<R> a, cpx<R> b) { return {a.re + b.re, a.im + b.im}; }
template <typename R>
__device__ __forceinline__ cpx<R> operator-(cpx<R> a, cpx<R> b) { return {a.re - b.re, a.im - b.im}; }
template <typename R>
__device__ __forceinline__ cpx<R> operator-(cpx<R> a) { return {-a.re, -a.im}; }
template <typename R>
__device__ __forceinline__ cpx<R> operator*(cpx<R> a, cpx<R> b)
{
    return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
template <typename R>
__device__ __forceinline__ cpx<R> operator*(R s, cpx<R> a) { return {s * a.re, s * a.im}; }
template <typename R>
__device__ __forceinline__ cpx<R> conj(cpx<R> a) { return {a.re, -a.im}; }
// conj(a) * b
template <typename R>
__device__ __forceinline__ cpx<R> cmulc(cpx<R> a, cpx<R> b)
{
    return {a.re * b.re + a.im * b.im, a.re * b.im - a.im * b.re};
}
// i * a and -i * a
template <typename R>
__device__ __forceinline__ cpx<R> ti(cpx<R> a) { return {-a.im, a.re}; }
template <typename R>
__device__ __forceinline__ cpx<R> tmi(cpx<R> a) { return {a.im, -a.re}; }
// acc += a * b
template <typename R>
__device__ __forceinline__ void cfma(cpx<R> &acc, cpx<R> a, cpx<R> b)
{
    acc.re = fma(a.re, b.re, acc.re);
    acc.re = fma(-a.im, b.im, acc.re);
    acc.im = fma(a.re, b.im, acc.im);
    acc.im = fma(a.im, b.re, acc.im);
}
// acc += conj(a) * b
template <typename R>
__device__ __forceinline__ void cfmac(cpx<R> &acc, cpx<R> a, cpx<R> b)
{
    acc.re = fma(a.re, b.re, acc.re);
    acc.re = fma(a.im, b.im, acc.re);
    acc.im = fma(a.re, b.im, acc.im);
    acc.im = fma(-a.im, b.re, acc.im);
}

// ------------------------------------------- FP64 <-> FP32 by integer operations
//
// The conversion instructions between FP64 and FP32 (or integers) run at 2
// lanes per clock and SM on this GPU, as slowly as FP64 arithmetic (measured:
// 1.99 against 64-90 for integer operations), so a pass that converts every
// component of a field is bound by them and not by memory.  These forms give
// the conversion instructions' results bit for bit: the exponent and mantissa
// bits are moved by integer operations, and the rare values outside FP32's
// normal range (subnormal results, overflow, infinities, NaN) take the
// instruction.

// round to nearest even
__device__ __forceinline__ float d2f(double v)
{
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const uint32_t mag = hi & 0x7fffffffu, sign = hi & 0x80000000u;
    const uint32_t e = mag - 0x38000000u;  // the exponent rebased to FP32's
    uint32_t f = __funnelshift_l(lo, e, 3);
    const uint32_t r = lo << 3;  // the 29 dropped bits, at the top of the word
    f += (r > 0x80000000u || (r == 0x80000000u && (f & 1u))) ? 1u : 0u;
    // normal results: rebased exponent 1..253 (254 may round up to infinity)
    if (e - 0x00100000u < 0x0fd00000u) return __uint_as_float(f | sign);
    if ((mag | lo) == 0u) return __uint_as_float(sign);
    return __double2float_rn(v);
}

// exact
__device__ __forceinline__ double f2d(float v)
{
    const uint32_t b = __float_as_uint(v), mag = b & 0x7fffffffu, sign = b & 0x80000000u;
    if (mag - 0x00800000u < 0x7f000000u)
        return __hiloint2double((int)(((mag >> 3) + 0x38000000u) | sign), (int)(b << 29));
    if (mag == 0u) return __hiloint2double((int)sign, 0);
    return (double)v;
}

// a * b in FP64 (the product of two 24-bit mantissas is exact)
__device__ __forceinline__ double mul_f2d(float a, float b)
{
    const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
    const uint32_t ma = ua & 0x7fffffffu, mb = ub & 0x7fffffffu, sign = (ua ^ ub) & 0x80000000u;
    if (ma - 0x00800000u < 0x7f000000u && mb - 0x00800000u < 0x7f000000u) {
        uint64_t p = (uint64_t)((ma & 0x007fffffu) | 0x00800000u) * ((mb & 0x007fffffu) | 0x00800000u);
        const uint32_t top = (uint32_t)(p >> 47);  // 1 when the product of the mantissas is >= 2
        p <<= 6u - top;                            // leading one at bit 52
        const uint32_t e = (ma >> 23) + (mb >> 23) + (1023u - 254u) + top;
        return __hiloint2double((int)((((uint32_t)(p >> 32)) - 0x00100000u + (e << 20)) | sign), (int)(uint32_t)p);
    }
    return (double)a * (double)b;
}

// Four doubles (32 bytes) with one access; p on a 32-byte boundary.
__device__ __forceinline__ void ld_global_x4(const double2 *p, double2 &a, double2 &b)
{
    asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(a.x), "=d"(a.y), "=d"(b.x), "=d"(b.y) : "l"(p));
}
__device__ __forceinline__ void st_global_x4(double2 *p, double2 a, double2 b)
{
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(a.x), "d"(a.y), "d"(b.x), "d"(b.y) : "memory");
}

// --------------------------------------------------------- storage formats

// One complex number per plane entry.  16-bit formats of spinors and clover
// carry one FP32 scale per site (stored value = value / scale); links are
// stored unscaled (unitary, |U_ab| <= 1).
struct StF64 {
    using T2 = double2;
    static constexpr bool kScaled = false;
    static constexpr int kBytes = 16;
    static constexpr bool kQuad = false;  // spinor fields in quad planes
};
struct StF32 {
    using T2 = float2;
    static constexpr bool kScaled = false;
    static constexpr int kBytes = 8;
    static constexpr bool kQuad = false;  // spinor fields in quad planes
};
struct StF16 {
    using T2 = __half2;
    static constexpr bool kScaled = true;
    static constexpr int kBytes = 4;
    static constexpr bool kQuad = true;  // spinor fields in quad planes
};
struct StBF16 {
    using T2 = __nv_bfloat162;
    static constexpr bool kScaled = true;
    static constexpr int kBytes = 4;
    static constexpr bool kQuad = false;  // spinor fields in quad planes
};

template <typename R>
__device__ __forceinline__ cpx<R> ld_c(const double2 *p) { double2 v = __ldg(p); return {(R)v.x, (R)v.y}; }
template <typename R>
__device__ __forceinline__ cpx<R> ld_c(const float2 *p) { float2 v = __ldg(p); return {(R)v.x, (R)v.y}; }
template <typename R>
__device__ __forceinline__ cpx<R> ld_c(const __half2 *p)
{
    float2 v = __half22float2(__ldg(p));
    return {(R)v.x, (R)v.y};
}
template <typename R>
__device__ __forceinline__ cpx<R> ld_c(const __nv_bfloat162 *p)
{
    float2 v = __bfloat1622float2(__ldg(p));
    return {(R)v.x, (R)v.y};
}

// plain (coherent) loads, for shared memory or buffers written in the same kernel
template <typename R>
__device__ __forceinline__ cpx<R> ld_s(const double2 *p) { double2 v = *p; return {(R)v.x, (R)v.y}; }
template <typename R>
__device__ __forceinline__ cpx<R> ld_s(const float2 *p) { float2 v = *p; return {(R)v.x, (R)v.y}; }
template <typename R>
__device__ __forceinline__ cpx<R> ld_s(const __half2 *p) { float2 v = __half22float2(*p); return {(R)v.x, (R)v.y}; }
template <typename R>
__device__ __forceinline__ cpx<R> ld_s(const __nv_bfloat162 *p)
{
    float2 v = __bfloat1622float2(*p);
    return {(R)v.x, (R)v.y};
}

template <typename R>
__device__ __forceinline__ void st_c(double2 *p, cpx<R> v) { *p = make_double2((double)v.re, (double)v.im); }
template <typename R>
__device__ __forceinline__ void st_c(float2 *p, cpx<R> v) { *p = make_float2((float)v.re, (float)v.im); }
template <typename R>
__device__ __forceinline__ void st_c(__half2 *p, cpx<R> v) { *p = __floats2half2_rn((float)v.re, (float)v.im); }
template <typename R>
__device__ __forceinline__ void st_c(__nv_bfloat162 *p, cpx<R> v)
{
    *p = __floats2bfloat162_rn((float)v.re, (float)v.im);
}

// A field in device memory: planes of Vd complex per domain, optional scale.
template <typename S>
struct Field {
    typename S::T2 *p;
    float *scale;  // [Nd*Vd], only for S::kScaled
};

// Spinor fields: per right-hand side and domain, a block of 12*Vd complex
// components.  Plane storage (FP64, FP32, BF16) keeps plane k of the block for
// component k of the domain's sites (offset k*Vd + s).  FP16 storage keeps
// quad planes: components 4q..4q+3 of a site side by side (16 bytes, one
// vector access), quad q of all the domain's sites before quad q+1 (offset
// (k/4)*4*Vd + 4s + k%4).  A 16-bit field's per-site scale is indexed by site.
// (Quad planes took the FP16 operator on 32^3x64 from 173.0 to 165.7 us; the
// BF16 operator measured 177.7 us in planes and 180.3 us in quads, so it keeps
// planes.)
__device__ __forceinline__ float2 word_f2(uint32_t w, const __half2 *)
{
    __half2 h;
    memcpy(&h, &w, 4);
    return __half22float2(h);
}
__device__ __forceinline__ float2 word_f2(uint32_t w, const __nv_bfloat162 *)
{
    __nv_bfloat162 h;
    memcpy(&h, &w, 4);
    return __bfloat1622float2(h);
}
__device__ __forceinline__ uint32_t f2_word(float a, float b, const __half2 *)
{
    __half2 h = __floats2half2_rn(a, b);
    uint32_t w;
    memcpy(&w, &h, 4);
    return w;
}
__device__ __forceinline__ uint32_t f2_word(float a, float b, const __nv_bfloat162 *)
{
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    uint32_t w;
    memcpy(&w, &h, 4);
    return w;
}

// The 12 stored components of site s of a spinor domain block blk (unscaled).
// NC: through the read-only path (the kernel does not write the field).
template <typename R, typename S, bool NC = true>
__device__ __forceinline__ void ld_sp_site(const typename S::T2 *blk, int s, int Vd, cpx<R> *x)
{
    if constexpr (S::kQuad) {
        const uint4 *q = reinterpret_cast<const uint4 *>(blk) + s;
        const typename S::T2 *tag = nullptr;
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const uint4 w = NC ? __ldg(q + (int64_t)j * Vd) : q[(int64_t)j * Vd];
            const float2 a = word_f2(w.x, tag), b = word_f2(w.y, tag), c = word_f2(w.z, tag), e = word_f2(w.w, tag);
            x[4 * j + 0] = {(R)a.x, (R)a.y};
            x[4 * j + 1] = {(R)b.x, (R)b.y};
            x[4 * j + 2] = {(R)c.x, (R)c.y};
            x[4 * j + 3] = {(R)e.x, (R)e.y};
        }
    } else {
        const typename S::T2 *p = blk + s;
#pragma unroll
        for (int k = 0; k < 12; k++) x[k] = NC ? ld_c<R>(p + (int64_t)k * Vd) : ld_s<R>(p + (int64_t)k * Vd);
    }
}

// Store the 12 components x (already divided by the site's scale for 16-bit
// storage) of site s of a spinor domain block blk.
template <typename R, typename S>
__device__ __forceinline__ void st_sp_site(typename S::T2 *blk, int s, int Vd, const cpx<R> *x)
{
    if constexpr (S::kQuad) {
        uint4 *q = reinterpret_cast<uint4 *>(blk) + s;
        const typename S::T2 *tag = nullptr;
#pragma unroll
        for (int j = 0; j < 3; j++) {
            uint4 w;
            w.x = f2_word((float)x[4 * j + 0].re, (float)x[4 * j + 0].im, tag);
            w.y = f2_word((float)x[4 * j + 1].re, (float)x[4 * j + 1].im, tag);
            w.z = f2_word((float)x[4 * j + 2].re, (float)x[4 * j + 2].im, tag);
            w.w = f2_word((float)x[4 * j + 3].re, (float)x[4 * j + 3].im, tag);
            q[(int64_t)j * Vd] = w;
        }
    } else {
        typename S::T2 *p = blk + s;
#pragma unroll
        for (int k = 0; k < 12; k++) st_c<R>(p + (int64_t)k * Vd, x[k]);
    }
}

// The 9 entries of a link and the 18 of a clover block in the copies that the
// Schwarz kernel stages, from the domain's planes blk (36 per site).  FP64 keeps
// planes.  FP32 keeps pairs (entries 2q and 2q+1 of a site side by side, element
// 2*Vd*q + 2*s + k%2; a link's entry 8 a plane): one 16-byte access for two.
// 16-bit storage keeps entries of a site side by side, so that
// one access brings several: a link's entries 0-3 and 4-7 as two quads (element
// 4*Vd*q + 4*s + k%4 of its nine planes), entry 8 as a plane; a clover block's
// entries 0-15 as four quads, 16 and 17 as a pair.  3 and 5 accesses for 9 and 18
// (us per half-sweep, planes against this: H16, 6x4^3 domains on 24x16x16x24 69.5 ->
// 65.0; BF16 on 24x32^3 291 -> 277; 4^4 domains on 32^4 within 0.3 %, and 165 -> 156 on
// 24^3x48 with the three-CTA form, whose clover reads go through the cache).
template <typename S>
__host__ __device__ constexpr int clover_elem(int k, int Vd, int s)
{
    return S::kBytes == 16                ? k * Vd + s
           : S::kBytes == 8 || k >= 16    ? (k / 2) * 2 * Vd + 2 * s + k % 2
                                          : (k / 4) * 4 * Vd + 4 * s + k % 4;
}

// NC: through the read-only path (global memory); else a plain load
template <typename T, bool NC>
__device__ __forceinline__ T ld_as(const void *p)
{
    if (NC) return __ldg(reinterpret_cast<const T *>(p));
    return *reinterpret_cast<const T *>(p);
}
template <typename R, typename T2>
__device__ __forceinline__ cpx<R> word_c(uint32_t w)
{
    const float2 v = word_f2(w, (const T2 *)nullptr);
    return {(R)v.x, (R)v.y};
}
template <typename R, typename S, bool NC>
__device__ __forceinline__ void ld_link(const typename S::T2 *blk, int mu, int s, int Vd, cpx<R> *u)
{
    using T2 = typename S::T2;
    const T2 *p = blk + mu * 9 * Vd;
    if constexpr (S::kBytes == 4) {
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const uint4 w = ld_as<uint4, NC>(p + q * 4 * Vd + 4 * s);
            u[4 * q + 0] = word_c<R, T2>(w.x);
            u[4 * q + 1] = word_c<R, T2>(w.y);
            u[4 * q + 2] = word_c<R, T2>(w.z);
            u[4 * q + 3] = word_c<R, T2>(w.w);
        }
        u[8] = word_c<R, T2>(ld_as<uint32_t, NC>(p + 8 * Vd + s));
    } else if constexpr (S::kBytes == 8) {
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const float4 w = ld_as<float4, NC>(p + q * 2 * Vd + 2 * s);
            u[2 * q] = {(R)w.x, (R)w.y};
            u[2 * q + 1] = {(R)w.z, (R)w.w};
        }
        u[8] = NC ? ld_c<R>(p + 8 * Vd + s) : ld_s<R>(p + 8 * Vd + s);
    } else {
#pragma unroll
        for (int k = 0; k < 9; k++) u[k] = NC ? ld_c<R>(p + k * Vd + s) : ld_s<R>(p + k * Vd + s);
    }
}
template <typename R, typename S, bool NC>
__device__ __forceinline__ void ld_clover_blk(const typename S::T2 *blk, int b, int s, int Vd, cpx<R> *m)
{
    using T2 = typename S::T2;
    const T2 *p = blk + b * 18 * Vd;
    if constexpr (S::kBytes == 4) {
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const uint4 w = ld_as<uint4, NC>(p + q * 4 * Vd + 4 * s);
            m[4 * q + 0] = word_c<R, T2>(w.x);
            m[4 * q + 1] = word_c<R, T2>(w.y);
            m[4 * q + 2] = word_c<R, T2>(w.z);
            m[4 * q + 3] = word_c<R, T2>(w.w);
        }
        const uint2 w = ld_as<uint2, NC>(p + 16 * Vd + 2 * s);
        m[16] = word_c<R, T2>(w.x);
        m[17] = word_c<R, T2>(w.y);
    } else if constexpr (S::kBytes == 8) {
#pragma unroll
        for (int q = 0; q < 9; q++) {
            const float4 w = ld_as<float4, NC>(p + q * 2 * Vd + 2 * s);
            m[2 * q] = {(R)w.x, (R)w.y};
            m[2 * q + 1] = {(R)w.z, (R)w.w};
        }
    } else {
#pragma unroll
        for (int k = 0; k < 18; k++) m[k] = NC ? ld_c<R>(p + k * Vd + s) : ld_s<R>(p + k * Vd + s);
    }
}

// ------------------------------------------------------------------ geometry

// Direction k = 2*mu + b: b = 0 the forward neighbour n+mu, b = 1 the backward n-mu.
struct Geom {
    int L[4], dom[4], nb[4];
    int V, Vd, Vh, Nd, Nd2;
    int vd_shift;          // log2(Vd) when Vd is a power of two, else -1
    const uint16_t *nbl;   // [Vd][8]: neighbour site slot (wrapped into the domain), bit 15 = leaves the domain
    const int *nbd;        // [Nd][8]: neighbour domain slot
    const int *block_slot; // [Nd]: slot of the domain with lexicographic block index b
    // Face slots of a domain (one per hop that leaves it): direction dir's
    // slots start at foff[dir] and are indexed by the site's coordinates
    // transverse to mu = dir/2, which a hop and its reverse share.
    const uint32_t *fcoord;  // [Vd]: byte mu = transverse index of the site for direction mu
    int foff[8];
    int nf;                  // face slots per domain
};

// Site of thread index gi when the lattice is walked domain by domain in
// lexicographic block order (neighbouring domains close together in time, so
// their data is still in L2 when it is read as a neighbour); the storage
// order of the slots is colour-major.
__device__ __forceinline__ void lex_site(const Geom &g, int gi, int &d, int &s)
{
    int b;
    if (g.vd_shift >= 0) {
        b = gi >> g.vd_shift;
        s = gi & (g.Vd - 1);
    } else {
        b = gi / g.Vd;
        s = gi - b * g.Vd;
    }
    d = __ldg(g.block_slot + b);
}

constexpr uint16_t kCross = 0x8000;
constexpr uint16_t kSlotMask = 0x7fff;

__device__ __forceinline__ void split_index(const Geom &g, int gi, int &d, int &s)
{
    if (g.vd_shift >= 0) {
        d = gi >> g.vd_shift;
        s = gi & (g.Vd - 1);
    } else {
        d = gi / g.Vd;
        s = gi - d * g.Vd;
    }
}

// global index of the neighbour of (d, s) in direction k
__device__ __forceinline__ int neighbour(const Geom &g, int d, int s, int k)
{
    uint16_t e = __ldg(g.nbl + s * 8 + k);
    int nd = (e & kCross) ? __ldg(g.nbd + d * 8 + k) : d;
    return nd * g.Vd + (e & kSlotMask);
}

// plane-major address: global index gi = d*Vd + s, plane p of P
__device__ __forceinline__ int64_t paddr(const Geom &g, int gi, int p, int P)
{
    int d, s;
    split_index(g, gi, d, s);
    return ((int64_t)d * P + p) * g.Vd + s;
}

// ------------------------------------------------------------ spin algebra

// Spinor component index: spin*3 + colour.  In the chiral basis
//   gamma_mu = [[0, a_mu], [a_mu^+, 0]] (2x2 spin blocks),
//   a_x = -i sigma_x, a_y = -i sigma_y, a_z = -i sigma_z, a_t = 1.
// (1 - sgn*gamma_mu) psi = (h ; -sgn * a^+ h) with h = u - sgn * a l, where
// u = spins (0,1) and l = spins (2,3) of psi.  The hopping term only needs the
// two-spin vector h per colour (the rank-2 projection), so each hop costs two
// SU(3) products.

// h = u - sgn * (a_mu l): half spinor from a full spinor, per colour c
template <int MU, int SGN, typename R>
__device__ __forceinline__ void project(const cpx<R> *x, cpx<R> *h)
{
#pragma unroll
    for (int c = 0; c < 3; c++) {
        cpx<R> u0 = x[0 * 3 + c], u1 = x[1 * 3 + c], l0 = x[2 * 3 + c], l1 = x[3 * 3 + c];
        cpx<R> al0, al1;
        if (MU == 0) { al0 = tmi(l1); al1 = tmi(l0); }       // -i sigma_x l
        else if (MU == 1) { al0 = -l1; al1 = l0; }           // -i sigma_y l
        else if (MU == 2) { al0 = tmi(l0); al1 = ti(l1); }   // -i sigma_z l
        else { al0 = l0; al1 = l1; }                         // 1 l
        if (SGN > 0) { h[c] = u0 - al0; h[3 + c] = u1 - al1; }
        else { h[c] = u0 + al0; h[3 + c] = u1 + al1; }
    }
}

// acc += (w ; -sgn * a_mu^+ w), w the half spinor after the colour product.
// SWAP: acc holds spins (2,3) in its first six entries and spins (0,1) in
// its last six (the same sums, stored the other way round).
template <int MU, int SGN, bool SWAP = false, typename R>
__device__ __forceinline__ void reconstruct_add(const cpx<R> *w, cpx<R> *acc)
{
    constexpr int up = SWAP ? 6 : 0, lo = SWAP ? 0 : 6;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        cpx<R> w0 = w[c], w1 = w[3 + c];
        cpx<R> b0, b1;  // a^+ w
        if (MU == 0) { b0 = ti(w1); b1 = ti(w0); }          // i sigma_x w
        else if (MU == 1) { b0 = w1; b1 = -w0; }            // i sigma_y w
        else if (MU == 2) { b0 = ti(w0); b1 = tmi(w1); }    // i sigma_z w
        else { b0 = w0; b1 = w1; }
        acc[up + c] = acc[up + c] + w0;
        acc[up + 3 + c] = acc[up + 3 + c] + w1;
        if (SGN > 0) { acc[lo + c] = acc[lo + c] - b0; acc[lo + 3 + c] = acc[lo + 3 + c] - b1; }
        else { acc[lo + c] = acc[lo + c] + b0; acc[lo + 3 + c] = acc[lo + 3 + c] + b1; }
    }
}

// FP32 form of su3_mul_half: the two spins of h share every link entry, so
// their products run as pairs (one paired FMA for the two spins), with the
// scalar form's order of operations in each lane -- the same bits.
template <bool DAG>
__device__ __forceinline__ void su3_mul_half_x2(const cpx<float> *U, const cpx<float> *h, cpx<float> *w)
{
    float2 hr[3], hi[3];
#pragma unroll
    for (int b = 0; b < 3; b++) {
        hr[b] = make_float2(h[b].re, h[3 + b].re);
        hi[b] = make_float2(h[b].im, h[3 + b].im);
    }
#pragma unroll
    for (int a = 0; a < 3; a++) {
        float2 ar = make_float2(0.f, 0.f), ai = make_float2(0.f, 0.f);
#pragma unroll
        for (int b = 0; b < 3; b++) {
            const cpx<float> u = DAG ? U[b * 3 + a] : U[a * 3 + b];
            const float2 ur = make_float2(u.re, u.re);
            const float2 ui = make_float2(DAG ? u.im : -u.im, DAG ? u.im : -u.im);  // enters re
            const float2 uj = make_float2(DAG ? -u.im : u.im, DAG ? -u.im : u.im);  // enters im
            ar = __ffma2_rn(ur, hr[b], ar);
            ar = __ffma2_rn(ui, hi[b], ar);
            ai = __ffma2_rn(ur, hi[b], ai);
            ai = __ffma2_rn(uj, hr[b], ai);
        }
        w[a] = mk(ar.x, ai.x);
        w[3 + a] = mk(ar.y, ai.y);
    }
}

// w = U h (DAG = false) or U^+ h (DAG = true) for the two spins of h;
// PAIRED: the FP32 form runs the two spins as paired FMAs (same bits)
template <bool DAG, typename R, bool PAIRED = true>
__device__ __forceinline__ void su3_mul_half(const cpx<R> *U, const cpx<R> *h, cpx<R> *w)
{
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ >= 1000
    if constexpr (sizeof(R) == 4 && PAIRED) {
        su3_mul_half_x2<DAG>(U, h, w);
        return;
    }
#endif
#pragma unroll
    for (int sp = 0; sp < 2; sp++)
#pragma unroll
        for (int a = 0; a < 3; a++) {
            cpx<R> acc = mk<R>(0, 0);
#pragma unroll
            for (int b = 0; b < 3; b++) {
                if (DAG) cfmac(acc, U[b * 3 + a], h[sp * 3 + b]);
                else cfma(acc, U[a * 3 + b], h[sp * 3 + b]);
            }
            w[sp * 3 + a] = acc;
        }
}

// one hop: acc += (1 - sgn gamma_mu) V x, V = U (forward) or U^+ (backward)
// reconstruct_add with a weight m (1: the same sums, as single-rounded
// fused multiply-adds of 1 * w; 0: acc unchanged), for hops that every lane
// evaluates and only some keep
template <int MU, int SGN, typename R>
__device__ __forceinline__ void reconstruct_fma(R m, const cpx<R> *w, cpx<R> *acc)
{
    const R ms = SGN > 0 ? -m : m;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        cpx<R> w0 = w[c], w1 = w[3 + c];
        cpx<R> b0, b1;  // a^+ w
        if (MU == 0) { b0 = ti(w1); b1 = ti(w0); }
        else if (MU == 1) { b0 = w1; b1 = -w0; }
        else if (MU == 2) { b0 = ti(w0); b1 = tmi(w1); }
        else { b0 = w0; b1 = w1; }
        acc[c] = mk<R>(fma(m, w0.re, acc[c].re), fma(m, w0.im, acc[c].im));
        acc[3 + c] = mk<R>(fma(m, w1.re, acc[3 + c].re), fma(m, w1.im, acc[3 + c].im));
        acc[6 + c] = mk<R>(fma(ms, b0.re, acc[6 + c].re), fma(ms, b0.im, acc[6 + c].im));
        acc[9 + c] = mk<R>(fma(ms, b1.re, acc[9 + c].re), fma(ms, b1.im, acc[9 + c].im));
    }
}

template <int MU, int SGN, bool SWAP = false, typename R>
__device__ __forceinline__ void hop(const cpx<R> *U, const cpx<R> *x, cpx<R> *acc)
{
    cpx<R> h[6], w[6];
    project<MU, SGN>(x, h);
    su3_mul_half<(SGN < 0)>(U, h, w);
    reconstruct_add<MU, SGN, SWAP>(w, acc);
}

// Hermitian 6x6 block from its packed 18 complex slots
template <typename R>
__device__ __forceinline__ void herm6_mul(const cpx<R> *blk, const cpx<R> *in, cpx<R> *out)
{
    R d[6] = {blk[0].re, blk[0].im, blk[1].re, blk[1].im, blk[2].re, blk[2].im};
#pragma unroll
    for (int i = 0; i < 6; i++) out[i] = d[i] * in[i];
    int k = 3;
#pragma unroll
    for (int i = 0; i < 6; i++)
#pragma unroll
        for (int j = i + 1; j < 6; j++) {
            cfma(out[i], blk[k], in[j]);
            cfmac(out[j], blk[k], in[i]);
            k++;
        }
}

// FP32 form of the two clover blocks at once: block 0 (spins 0,1) in lane 0
// and block 1 (spins 2,3) in lane 1 of paired FMAs.  Each lane runs
// herm6_mul's sequence of operations, so the result is the same bits.
__device__ __forceinline__ void herm6_mul_x2(const cpx<float> *b0, const cpx<float> *b1, const cpx<float> *in,
                                             cpx<float> *out)
{
    float2 inr[6], ini[6], ore[6], oim[6];
#pragma unroll
    for (int i = 0; i < 6; i++) {
        inr[i] = make_float2(in[i].re, in[6 + i].re);
        ini[i] = make_float2(in[i].im, in[6 + i].im);
    }
#pragma unroll
    for (int i = 0; i < 6; i++) {
        const float2 dd = make_float2((i & 1) ? b0[i >> 1].im : b0[i >> 1].re, (i & 1) ? b1[i >> 1].im : b1[i >> 1].re);
        ore[i] = __fmul2_rn(dd, inr[i]);
        oim[i] = __fmul2_rn(dd, ini[i]);
    }
    int k = 3;
#pragma unroll
    for (int i = 0; i < 6; i++)
#pragma unroll
        for (int j = i + 1; j < 6; j++) {
            const float2 br = make_float2(b0[k].re, b1[k].re), bi = make_float2(b0[k].im, b1[k].im);
            const float2 nbi = make_float2(-b0[k].im, -b1[k].im);
            ore[i] = __ffma2_rn(br, inr[j], ore[i]);  // out[i] += b in[j]
            ore[i] = __ffma2_rn(nbi, ini[j], ore[i]);
            oim[i] = __ffma2_rn(br, ini[j], oim[i]);
            oim[i] = __ffma2_rn(bi, inr[j], oim[i]);
            ore[j] = __ffma2_rn(br, inr[i], ore[j]);  // out[j] += conj(b) in[i]
            ore[j] = __ffma2_rn(bi, ini[i], ore[j]);
            oim[j] = __ffma2_rn(br, ini[i], oim[j]);
            oim[j] = __ffma2_rn(nbi, inr[i], oim[j]);
            k++;
        }
#pragma unroll
    for (int i = 0; i < 6; i++) {
        out[i] = mk(ore[i].x, oim[i].x);
        out[6 + i] = mk(ore[i].y, oim[i].y);
    }
}

// Runtime-checked device error flags (bounded waits that ran out, etc.).
constexpr int kErrMbarTimeout = 1;

// Range checks of the hot-path kernels' indices.  A library built with
// -DQDD_CHECK tests every guarded index; one out of range is counted in this
// translation unit's counter and its access skipped (no trap, no wait).  In
// the normal build the guard is the constant true and compiles away.
#ifdef QDD_CHECK
static __device__ unsigned long long g_check_hits;
__device__ __forceinline__ bool in_range(long long v, long long lo, long long hi)
{
    if (v >= lo && v < hi) return true;
    atomicAdd(&g_check_hits, 1ull);
    return false;
}
#define QDD_IN_RANGE(v, lo, hi) ::qdd::in_range((long long)(v), (long long)(lo), (long long)(hi))
#else
#define QDD_IN_RANGE(v, lo, hi) true
#endif

}  // namespace qdd
