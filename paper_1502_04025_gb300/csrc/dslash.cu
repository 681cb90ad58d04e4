// Full-lattice Wilson-clover operator  y = D x = A x - kappa H x
// (arXiv:1502.04025, Sec. 3.1 names the operator; Sec. 3.6 counts 1848 flop
// per site: 1320 for the eight spin-projected hops, 504 for the two Hermitian
// 6x6 clover blocks, 24 for the final combination).
//
// One thread per site over the domain-blocked, plane-major layout: a warp
// reads 32 consecutive sites of one plane (256 or 512 contiguous bytes) for
// every link, clover and spinor component.  Domains are visited in
// lexicographic block order, so a domain's neighbours are processed close in
// time and their spinors are read from L2 rather than again from HBM.  Neighbour sites come from a
// per-domain-shape table (the neighbour's slot inside its domain and whether
// the hop leaves the domain) and a per-domain table of neighbouring domains.
// The roofline of this kernel is HBM bandwidth: each link, clover entry and
// input spinor is read once and the output written once when the neighbour
// re-reads hit in L1/L2.  For SU(3) fields the FP32 and 16-bit forms read
// only the first two rows of each link and rebuild the third (96 fewer bytes
// per site in FP32), and their 16-bit link and clover copies are stored with
// planes paired, one 8-byte load per two planes.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "fixed.cuh"
#include "internal.h"

namespace qdd {

// FP16 spinors (quad planes): site s of the domain block at blk_base, scaled
template <typename R, typename S>
__device__ __forceinline__ void load_spinor_quad(const Field<S> &f, int64_t blk_base, int s, int64_t sidx, int Vd,
                                                 cpx<R> *x)
{
    const R sc = (R)__ldg(f.scale + sidx);
    ld_sp_site<R, S>(f.p + blk_base, s, Vd, x);
#pragma unroll
    for (int k = 0; k < 12; k++) x[k] = sc * x[k];
}

// spinors in planes: the site's first component at gi_plane_base
template <typename R, typename S>
__device__ __forceinline__ void load_spinor(const Field<S> &f, int64_t gi_plane_base, int64_t sidx, int Vd,
                                            cpx<R> *x)
{
    const typename S::T2 *p = f.p + gi_plane_base;
    R sc = S::kScaled ? (R)__ldg(f.scale + sidx) : (R)1;
#pragma unroll
    for (int k = 0; k < 12; k++) {
        cpx<R> v = ld_c<R>(p + (int64_t)k * Vd);
        x[k] = S::kScaled ? sc * v : v;
    }
}

// Two adjacent planes of a paired 16-bit field with one 8-byte load.
template <typename R>
__device__ __forceinline__ void ld_pair(const __half2 *p, cpx<R> &a, cpx<R> &b)
{
    uint2 v = __ldg(reinterpret_cast<const uint2 *>(p));
    float2 f0 = __half22float2(*reinterpret_cast<const __half2 *>(&v.x));
    float2 f1 = __half22float2(*reinterpret_cast<const __half2 *>(&v.y));
    a = mk<R>(f0.x, f0.y);
    b = mk<R>(f1.x, f1.y);
}
template <typename R>
__device__ __forceinline__ void ld_pair(const __nv_bfloat162 *p, cpx<R> &a, cpx<R> &b)
{
    uint2 v = __ldg(reinterpret_cast<const uint2 *>(p));
    float2 f0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.x));
    float2 f1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&v.y));
    a = mk<R>(f0.x, f0.y);
    b = mk<R>(f1.x, f1.y);
}

// Link U_mu of site s of domain d.  L12: the field holds the first two rows
// (24 planes per site) and the third is rebuilt as the conjugated cross
// product of the two, i.e. from the cofactors of U = (U^+)^-1 for det U = 1.
template <typename R, typename S, bool L12>
__device__ __forceinline__ void load_link(const Field<S> &U, int d, int s, int mu, int Vd, cpx<R> *u)
{
    if (L12) {
        if constexpr (S::kBytes == 4) {  // 16-bit: paired planes
            const typename S::T2 *p = U.p + pair_index(d, 24, mu * 6, Vd, s);
#pragma unroll
            for (int j = 0; j < 3; j++) ld_pair<R>(p + (int64_t)j * Vd * 2, u[2 * j], u[2 * j + 1]);
        } else {
            const typename S::T2 *p = U.p + ((int64_t)d * 24 + mu * 6) * Vd + s;
#pragma unroll
            for (int k = 0; k < 6; k++) u[k] = ld_c<R>(p + (int64_t)k * Vd);
        }
        u[6] = conj(u[1] * u[5] - u[2] * u[4]);
        u[7] = conj(u[2] * u[3] - u[0] * u[5]);
        u[8] = conj(u[0] * u[4] - u[1] * u[3]);
    } else {
        ld_link<R, S, true>(U.p + (int64_t)d * 36 * Vd, mu, s, Vd, u);
    }
}

// one hop of a neighbour spinor x stored with per-site scale sc: the hop is
// linear, so the scale multiplies its 6-component result, not the 12 inputs
template <int MU, int SGN, bool SCALED, bool PAIRED, typename R>
__device__ __forceinline__ void hop_scaled(const cpx<R> *U, const cpx<R> *x, R sc, cpx<R> *acc)
{
    cpx<R> h[6], w[6];
    project<MU, SGN>(x, h);
    su3_mul_half<(SGN < 0), R, PAIRED>(U, h, w);
    if (SCALED) {
#pragma unroll
        for (int k = 0; k < 6; k++) w[k] = sc * w[k];
    }
    reconstruct_add<MU, SGN>(w, acc);
}

// the unscaled components of a spinor and, for a 16-bit field, its scale;
// fields in planes: the site's first component at gi_plane_base; FP16 fields
// (quad planes): site s of the domain block at blk_base
template <typename R, typename S>
__device__ __forceinline__ R load_spinor_raw_quad(const Field<S> &f, int64_t blk_base, int s, int64_t sidx, int Vd,
                                                  cpx<R> *x)
{
    ld_sp_site<R, S>(f.p + blk_base, s, Vd, x);
    return (R)__ldg(f.scale + sidx);
}

template <typename R, typename S>
__device__ __forceinline__ R load_spinor_raw(const Field<S> &f, int64_t gi_plane_base, int64_t sidx, int Vd,
                                             cpx<R> *x)
{
    const typename S::T2 *p = f.p + gi_plane_base;
#pragma unroll
    for (int k = 0; k < 12; k++) x[k] = ld_c<R>(p + (int64_t)k * Vd);
    return S::kScaled ? (R)__ldg(f.scale + sidx) : (R)1;
}

template <int MU, typename R, typename SL, typename SI, bool L12>
__device__ __forceinline__ void dslash_dir(const Geom &g, const Field<SL> &U, const Field<SI> &in, int64_t rbase,
                                           int64_t sbase, int d, int s, cpx<R> *acc)
{
    // paired FMAs in the colour products, except with FP16 links and FP32
    // spinors, where they measured slower (192.7 against 200.7 us on 32^3x64)
    constexpr bool kPaired = !(std::is_same<SL, StF16>::value && std::is_same<SI, StF32>::value);
    cpx<R> u[9], x[12];
    {
        uint16_t e = __ldg(g.nbl + s * 8 + 2 * MU);
        int nd = (e & kCross) ? __ldg(g.nbd + d * 8 + 2 * MU) : d;
        int ns = e & kSlotMask;
        if (QDD_IN_RANGE(nd, 0, g.Nd) && QDD_IN_RANGE(ns, 0, g.Vd)) {
            R sc;
            if constexpr (SI::kQuad)
                sc = load_spinor_raw_quad<R, SI>(in, rbase + (int64_t)nd * 12 * g.Vd, ns,
                                                 sbase + (int64_t)nd * g.Vd + ns, g.Vd, x);
            else
                sc = load_spinor_raw<R, SI>(in, rbase + (int64_t)nd * 12 * g.Vd + ns, sbase + (int64_t)nd * g.Vd + ns,
                                            g.Vd, x);
            load_link<R, SL, L12>(U, d, s, MU, g.Vd, u);
            hop_scaled<MU, +1, SI::kScaled, kPaired>(u, x, sc, acc);
        }
    }
    {
        uint16_t e = __ldg(g.nbl + s * 8 + 2 * MU + 1);
        int nd = (e & kCross) ? __ldg(g.nbd + d * 8 + 2 * MU + 1) : d;
        int ns = e & kSlotMask;
        if (QDD_IN_RANGE(nd, 0, g.Nd) && QDD_IN_RANGE(ns, 0, g.Vd)) {
            R sc;
            if constexpr (SI::kQuad)
                sc = load_spinor_raw_quad<R, SI>(in, rbase + (int64_t)nd * 12 * g.Vd, ns,
                                                 sbase + (int64_t)nd * g.Vd + ns, g.Vd, x);
            else
                sc = load_spinor_raw<R, SI>(in, rbase + (int64_t)nd * 12 * g.Vd + ns, sbase + (int64_t)nd * g.Vd + ns,
                                            g.Vd, x);
            load_link<R, SL, L12>(U, nd, ns, MU, g.Vd, u);
            hop_scaled<MU, -1, SI::kScaled, kPaired>(u, x, sc, acc);
        }
    }
}

// The geometry with the domain volume fixed at compile time when VD > 0 (a
// power of two): plane strides and site splits become immediates.
template <int VD>
__device__ __forceinline__ Geom fixed_geom(const Geom &g0)
{
    Geom g = g0;
    if (VD > 0) {
        static_assert(VD <= 0 || (VD & (VD - 1)) == 0, "a fixed domain volume is a power of two");
        g.Vd = VD;
        g.Vh = VD / 2;
        g.vd_shift = VD == 256 ? 8 : (VD == 512 ? 9 : (VD == 128 ? 7 : g0.vd_shift));
    }
    return g;
}

// Output in the host layout: FP64, a site's 12 components together (single
// precision results of the operator entry point, which a separate pass would
// read and widen again).
struct StHost {
    using T2 = double2;
    static constexpr bool kScaled = false;
    static constexpr int kBytes = 16;
    static constexpr bool kQuad = false;
};
struct HostOut {
    const int *site_of;  // host site index of an internal index
    bool a32;            // the buffer starts on a 32-byte boundary
};

// CTAs per SM the register allocation aims at.  FP16 links: 4 (the lower
// register cap of 5 costs more in the FP16 and H16 forms: on 32^3x64, FP16
// 181.5 -> 175.0 us and H16 193.6 -> 190.1 us at 4; FP32 and BF16 are
// faster at 5, BF16 176.6 against 188.0 us).
template <typename R, typename SL>
constexpr int dslash_min_blocks()
{
    return sizeof(R) == 4 ? (std::is_same<SL, StF16>::value ? 4 : 5) : 1;
}

template <typename R, typename SL, typename SC, typename SI, typename SO, bool RESID, bool L12, int VD = 0>
__global__ void __launch_bounds__(128, (dslash_min_blocks<R, SL>())) k_dslash(Geom g0, Field<SL> U, Field<SC> A, Field<SI> in, Field<SO> out,
                                                const double2 *b, R kappa, HostOut ho)
{
    const Geom g = fixed_geom<VD>(g0);
    int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= g.V) return;
    const int64_t r = blockIdx.y;
    const int64_t rbase = r * (int64_t)g.V * 12, sbase = r * (int64_t)g.V;
    int d, s;
    lex_site(g, gi, d, s);
    gi = d * g.Vd + s;
    cpx<R> acc[12];
#pragma unroll
    for (int k = 0; k < 12; k++) acc[k] = mk<R>(0, 0);
    dslash_dir<0, R, SL, SI, L12>(g, U, in, rbase, sbase, d, s, acc);
    dslash_dir<1, R, SL, SI, L12>(g, U, in, rbase, sbase, d, s, acc);
    dslash_dir<2, R, SL, SI, L12>(g, U, in, rbase, sbase, d, s, acc);
    dslash_dir<3, R, SL, SI, L12>(g, U, in, rbase, sbase, d, s, acc);

    cpx<R> x[12];
    if constexpr (SI::kQuad)
        load_spinor_quad<R, SI>(in, rbase + (int64_t)d * 12 * g.Vd, s, sbase + gi, g.Vd, x);
    else
        load_spinor<R, SI>(in, rbase + (int64_t)d * 12 * g.Vd + s, sbase + gi, g.Vd, x);
    cpx<R> y[12];
    {
        const typename SC::T2 *p = A.p + (int64_t)d * 36 * g.Vd + s;
        R sc = SC::kScaled ? (R)__ldg(A.scale + gi) : (R)1;
        cpx<R> m[2][18];
#pragma unroll
        for (int blk = 0; blk < 2; blk++) {
            if constexpr (SC::kBytes == 4) {  // 16-bit: paired planes
                const typename SC::T2 *pp = A.p + pair_index(d, 36, blk * 18, g.Vd, s);
#pragma unroll
                for (int j = 0; j < 9; j++) ld_pair<R>(pp + (int64_t)j * g.Vd * 2, m[blk][2 * j], m[blk][2 * j + 1]);
            } else {
#pragma unroll
                for (int k = 0; k < 18; k++) m[blk][k] = ld_c<R>(p + (int64_t)(blk * 18 + k) * g.Vd);
            }
        }
        // The two blocks as paired FMAs (the same bits) only with FP16 clover and
        // spinors: 175.0 -> 171.9 us on 32^3x64.  Measured slower in the other
        // forms: FP32 256.7 -> 344.0 us at 96 registers, H16 190.1 -> 198.2 us.
        if constexpr (std::is_same<SC, StF16>::value && std::is_same<SI, StF16>::value) {
            herm6_mul_x2(m[0], m[1], x, y);
        } else {
            herm6_mul(m[0], x, y);
            herm6_mul(m[1], x + 6, y + 6);
        }
        if (SC::kScaled) {  // the clover's per-site scale on the 12 products
#pragma unroll
            for (int k = 0; k < 12; k++) y[k] = sc * y[k];
        }
    }
#pragma unroll
    for (int k = 0; k < 12; k++) {
        y[k].re = fma(-kappa, acc[k].re, y[k].re);
        y[k].im = fma(-kappa, acc[k].im, y[k].im);
    }
    if (RESID) {
        const double2 *bp = b + rbase + (int64_t)d * 12 * g.Vd + s;
#pragma unroll
        for (int k = 0; k < 12; k++) {
            double2 v = __ldg(bp + (int64_t)k * g.Vd);
            // (FP32 arithmetic: the difference is FP64's, rounded once)
            if constexpr (sizeof(R) == 4) y[k] = mk<R>(d2f(v.x - f2d(y[k].re)), d2f(v.y - f2d(y[k].im)));
            else y[k] = mk<R>((R)v.x - y[k].re, (R)v.y - y[k].im);
        }
    }
    if constexpr (std::is_same<SO, StHost>::value) {
        double2 *o = out.p + (r * g.V + __ldg(ho.site_of + gi)) * 12;
        double2 v[12];
#pragma unroll
        for (int k = 0; k < 12; k++) v[k] = make_double2(f2d(y[k].re), f2d(y[k].im));
        if (ho.a32) {
#pragma unroll
            for (int k = 0; k < 12; k += 2) st_global_x4(o + k, v[k], v[k + 1]);
        } else {
#pragma unroll
            for (int k = 0; k < 12; k++) o[k] = v[k];
        }
        return;
    }
    typename SO::T2 *op = out.p + rbase + (int64_t)d * 12 * g.Vd + s;
    if (SO::kScaled) {
        R m = 0;
#pragma unroll
        for (int k = 0; k < 12; k++) m = fmax(m, fmax(fabs(y[k].re), fabs(y[k].im)));
        float scf = (float)m;
        out.scale[sbase + gi] = scf;
        R inv = m > 0 ? (R)1 / (R)scf : (R)0;
        if constexpr (SO::kQuad) {
#pragma unroll
            for (int k = 0; k < 12; k++) y[k] = inv * y[k];
            st_sp_site<R, SO>(out.p + rbase + (int64_t)d * 12 * g.Vd, s, g.Vd, y);
        } else {
#pragma unroll
            for (int k = 0; k < 12; k++) st_c<R>(op + (int64_t)k * g.Vd, inv * y[k]);
        }
    } else {
#pragma unroll
        for (int k = 0; k < 12; k++) st_c<R>(op + (int64_t)k * g.Vd, y[k]);
    }
}

// ------------------------------------------------------------------------
// The operator of the precisions F64 and DF64 in 64-bit fixed point (fixed.cuh):
// y = D x, or b - D x, in FP64.  One thread per site; a hop's
// colour products are three integer multiply-adds per real product, summed
// exactly at the neighbour site's scale, rounded, and shifted to the largest
// scale of the nine sites before the hops are added; the clover product keeps
// the site's own scale; both are converted once and combined in FP64.  Beside
// them run sums of the products' magnitudes from the factors' leading bits, two
// spins in one 32-bit word (72 multiply-adds per site): where one of the twelve is
// small against the scales, the site goes on a list and k_dslash_list computes it
// in FP64.
//
// Bound: integer multiply-adds 2520 per site (39 clocks of an SM at 64 lanes)
// and about as many other integer operations, against 69 clocks for the
// 1536 bytes per site at the measured HBM rate, where FP64 arithmetic takes 570
// clocks (1140 instructions at 2 lanes).  Measured, with the launch over an empty
// list: 32^4 sites in 4^4 domains 556 us, 157 clocks per site, against 2113 us in FP64
// arithmetic; 24x16x12x32 101 against 312 us.  The sums of magnitudes and that launch
// are 20 and 12 us of it.
// What is left is latency: 12 to 16 warps per SM at 168 or 128 registers.
// The four directions are compiled once each, for both signs (a runtime flag
// picks the transposed link and the signs): eight bodies would not fit the
// instruction cache.

__device__ __forceinline__ cfx ld_cfx(const int4 *p)
{
    const int4 v = __ldg(p);
    return {{v.x, v.y}, {v.z, v.w}};
}

// Fields of the fixed-point operator.
struct FxArgs {
    const int4 *U, *A, *x;    // links and clover in planes of 36, spinors in planes of 12
    const int *ae, *xe;       // exponents: clover per site, spinors per right-hand side and site
    int *list;                // list[0] sites left to FP64 (r V + index) from list[1] on
    int u;                    // exponent of the links
    int ush;                  // a link entry's leading bits are its upper limb >> ush
    float hop, clov;          // the test of the sums of magnitudes, in their units
    const double2 *b;         // residual form: b - D x
    double2 *out;             // internal planes, or (site_of) the host layout
    const int *site_of;
    bool a32;                 // host layout: out on a 32-byte boundary
    FxInput src;              // what x was made from
    const double2 *U64, *A64; // FP64 links and clover
};

struct cfxsum {
    int64_t re, im;
};

// t += a_mu^+ w, the part of the product w of spin sp, with project()'s a_mu
template <int MU>
__device__ __forceinline__ void fx_lower(int sp, int64_t wr, int64_t wi, cfxsum &t)
{
    // a^+ w: x: (i w1, i w0); y: (w1, -w0); z: (i w0, -i w1); t: (w0, w1)
    const bool neg = (MU == 1 && sp == 0) || (MU == 2 && sp == 1);
    if (MU == 0 || MU == 2) {
        if (neg) { t.re += wi; t.im -= wr; }
        else { t.re -= wi; t.im += wr; }
    } else {
        if (neg) { t.re -= wr; t.im -= wi; }
        else { t.re += wr; t.im += wi; }
    }
}

template <int MU>
__device__ __forceinline__ void fx_hop_dir(const Geom &g, const FxArgs &f, int64_t rbase, int d, int s, int E,
                                           const int *xe, cfxsum *acc, uint32_t *mag)
{
#pragma unroll 1
    for (int back = 0; back < 2; back++) {
        const int dir = 2 * MU + back;
        const uint16_t en = __ldg(g.nbl + s * 8 + dir);
        const int nd = (en & kCross) ? __ldg(g.nbd + d * 8 + dir) : d, ns = en & kSlotMask;
        if (!(QDD_IN_RANGE(nd, 0, g.Nd) && QDD_IN_RANGE(ns, 0, g.Vd))) continue;
        const int sft = min(E - __ldg(xe + (int64_t)nd * g.Vd + ns), 63);
        const int4 *xp = f.x + rbase + (int64_t)nd * 12 * g.Vd + ns;
        // projection h = u + q (a_mu l), limb by limb (the limbs grow by one bit)
        const int q = back ? 1 : -1;
        // forward: U h; backward: U^+ h (transposed link, conjugated)
        const int4 *up = f.U + ((int64_t)(back ? nd : d) * 36 + MU * 9) * g.Vd + (back ? ns : s);
        const int64_t sa = (back ? 1 : 3) * (int64_t)g.Vd, sb = (back ? 3 : 1) * (int64_t)g.Vd;
        cfx h[6];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const cfx u0 = ld_cfx(xp + (int64_t)c * g.Vd), u1 = ld_cfx(xp + (int64_t)(3 + c) * g.Vd);
            const cfx l0 = ld_cfx(xp + (int64_t)(6 + c) * g.Vd), l1 = ld_cfx(xp + (int64_t)(9 + c) * g.Vd);
            auto add = [](fx a, int qq, fx b) -> fx { return {a.hi + qq * b.hi, a.lo + qq * b.lo}; };
            auto tmi_ = [&](cfx u, cfx l, int qq) -> cfx { return {add(u.re, qq, l.im), add(u.im, -qq, l.re)}; };
            if (MU == 0) { h[c] = tmi_(u0, l1, q); h[3 + c] = tmi_(u1, l0, q); }
            else if (MU == 1) {
                h[c] = {add(u0.re, -q, l1.re), add(u0.im, -q, l1.im)};
                h[3 + c] = {add(u1.re, q, l0.re), add(u1.im, q, l0.im)};
            } else if (MU == 2) { h[c] = tmi_(u0, l0, q); h[3 + c] = tmi_(u1, l1, -q); }
            else {
                h[c] = {add(u0.re, q, l0.re), add(u0.im, q, l0.im)};
                h[3 + c] = {add(u1.re, q, l1.re), add(u1.im, q, l1.im)};
            }
        }
        // Leading bits of the half spinor, 2^5 at the common scale (a component is
        // below 2^6 of them), the two spins side by side; with a link's, 2^6 for 1 (5 for
        // links that are not SU(3)), the sums of a row and of eight hops stay below
        // 2^16: 2^6 sqrt(3) 2^6 8 (2^5 2.45 2^6 8).
        uint32_t hp[3];
        const int hsh = min(kFxSpinorBits - kFxLimb - 5 + sft, 31);
#pragma unroll
        for (int c = 0; c < 3; c++)
            hp[c] = (uint32_t)max(abs(h[c].re.hi), abs(h[c].im.hi)) >> hsh |
                    (uint32_t)max(abs(h[3 + c].re.hi), abs(h[3 + c].im.hi)) >> hsh << 16;
        // the lower spins get -a^+ w forward and +a^+ w backward: their sums
        // change sign before each of the two
#pragma unroll
        for (int k = 6; k < 12; k++) acc[k] = {-acc[k].re, -acc[k].im};
        // Per row of the link: both spins' real and imaginary sums at once, so
        // that a multiply-add's accumulator is needed again only four
        // instructions later.
#pragma unroll
        for (int a = 0; a < 3; a++) {
            fxacc t[4] = {fx_zero(), fx_zero(), fx_zero(), fx_zero()};  // spin 0 re, im, spin 1 re, im
            uint32_t sum = 0;
#pragma unroll
            for (int b = 0; b < 3; b++) {
                const cfx v = ld_cfx(up + a * sa + b * sb);
                const fx vp = {v.im.hi * q, v.im.lo * q}, vn = {-vp.hi, -vp.lo};
                sum += ((uint32_t)max(abs(v.re.hi), abs(v.im.hi)) >> f.ush) * hp[b];
                fx_mac4(t, v.re, h[b].re, h[b].im, h[3 + b].re, h[3 + b].im);
                fx_mac2(t[0], t[2], vp, h[b].im, h[3 + b].im);
                fx_mac2(t[1], t[3], vn, h[b].re, h[3 + b].re);
            }
#pragma unroll
            for (int sp = 0; sp < 2; sp++) {
                const int64_t wr = fx_value(t[2 * sp]) >> sft, wi = fx_value(t[2 * sp + 1]) >> sft;
                acc[sp * 3 + a].re += wr;
                acc[sp * 3 + a].im += wi;
                // the lower spin fed by this one: the other for x, y; the same for z, t
                const int lo = 6 + 3 * (MU < 2 ? 1 - sp : sp) + a;
                fx_lower<MU>(sp, wr, wi, acc[lo]);
            }
            mag[a] += sum;
            mag[3 + a] += MU < 2 ? sum << 16 | sum >> 16 : sum;
        }
    }
}

// CTAs per SM the register allocation aims at: 3 with the volume fixed at
// compile time (540 against 561 us on 32^4), 4 without (16^3x32 in 8x4^3 domains 88.7
// against 80.2, 24x16x12x32 in 6x4x2x4 91.0 against 89.5)
template <bool RESID, bool HOST, int VD = 0>
__global__ void __launch_bounds__(128, VD ? 3 : 4) k_dslash_fx(Geom g0, FxArgs f, double kappa)
{
    const Geom g = fixed_geom<VD>(g0);
    const int gt = blockIdx.x * blockDim.x + threadIdx.x;
    if (gt >= g.V) return;
    const int64_t r = blockIdx.y, rbase = r * (int64_t)g.V * 12, sbase = r * (int64_t)g.V;
    int d, s;
    lex_site(g, gt, d, s);
    const int gi = d * g.Vd + s;
    const int *xe = f.xe + sbase;
    // the common scale: the largest exponent of the site and its neighbours
    const int e0 = __ldg(xe + gi);
    int E = e0;
#pragma unroll
    for (int dir = 0; dir < 8; dir++) {
        const uint16_t en = __ldg(g.nbl + s * 8 + dir);
        const int nd = (en & kCross) ? __ldg(g.nbd + d * 8 + dir) : d, ns = en & kSlotMask;
        if (QDD_IN_RANGE(nd, 0, g.Nd) && QDD_IN_RANGE(ns, 0, g.Vd)) E = max(E, __ldg(xe + (int64_t)nd * g.Vd + ns));
    }
    const double2 *bp = RESID ? f.b + rbase + (int64_t)d * 12 * g.Vd + s : nullptr;
    double2 *op = HOST ? f.out + (r * g.V + __ldg(f.site_of + gi)) * 12 : f.out + rbase + (int64_t)d * 12 * g.Vd + s;
    auto store6 = [&](int blk, double2 *y) {
        if (RESID) {
#pragma unroll
            for (int k = 0; k < 6; k++) {
                const double2 v = __ldg(bp + (int64_t)(6 * blk + k) * g.Vd);
                y[k] = make_double2(v.x - y[k].x, v.y - y[k].y);
            }
        }
        if (HOST && f.a32) {
#pragma unroll
            for (int k = 0; k < 6; k += 2) st_global_x4(op + 6 * blk + k, y[k], y[k + 1]);
        } else {
#pragma unroll
            for (int k = 0; k < 6; k++) op[(int64_t)(6 * blk + k) * (HOST ? 1 : g.Vd)] = y[k];
        }
    };
    bool fp64 = E >= kFxRaw;
    const int ae = __ldg(f.ae + gi);
    cfxsum acc[12];
    if (!fp64) {
#pragma unroll
        for (int k = 0; k < 12; k++) acc[k] = {0, 0};
        uint32_t mag[6] = {0, 0, 0, 0, 0, 0};
        fx_hop_dir<0>(g, f, rbase, d, s, E, xe, acc, mag);
        fx_hop_dir<1>(g, f, rbase, d, s, E, xe, acc, mag);
        fx_hop_dir<2>(g, f, rbase, d, s, E, xe, acc, mag);
        fx_hop_dir<3>(g, f, rbase, d, s, E, xe, acc, mag);
        uint32_t low = mag[0];
#pragma unroll
        for (int k = 0; k < 6; k++) low = min(low & 0xffffu, min(mag[k] & 0xffffu, mag[k] >> 16));
        const int n = min(max(e0 + ae - E - f.u, -126), 127);
        fp64 = E != kFxZero && !((float)low >= fmaf(f.clov, __int_as_float((n + 127) << 23), f.hop));
    }
    if (fp64) {
        f.list[1 + atomicAdd(f.list, 1)] = (int)(r * g.V) + gi;
        return;
    }

    const int ca = e0 + ae + 2 * kFxLimb - kFxSpinorBits - kFxCloverBits;    // scale of the clover sums
    const int ch = E + f.u + 2 * kFxLimb - kFxSpinorBits - kFxLinkBits;      // scale of the hop sums
    const int4 *xp = f.x + rbase + (int64_t)d * 12 * g.Vd + s;
    const int4 *ap = f.A + (int64_t)d * 36 * g.Vd + s;
    // one chirality block per iteration; the hop sums wait in shared memory, so
    // that the clover sums have their registers (2 % on 4^4 domains, 6 % on others)
    __shared__ int64_t hop_sum[24][128];
#pragma unroll
    for (int k = 0; k < 12; k++) {
        hop_sum[2 * k][threadIdx.x] = acc[k].re;
        hop_sum[2 * k + 1][threadIdx.x] = acc[k].im;
    }
#pragma unroll 1
    for (int blk = 0; blk < 2; blk++) {
        cfx x[6];
#pragma unroll
        for (int k = 0; k < 6; k++) x[k] = ld_cfx(xp + (int64_t)(6 * blk + k) * g.Vd);
        // all six rows at once: every entry is read once, b for row i and
        // conj(b) for row j, and the sums it feeds are independent
        fxacc t[12];  // rows' real parts, then imaginary parts
#pragma unroll
        for (int i = 0; i < 12; i++) t[i] = fx_zero();
#pragma unroll
        for (int i = 0; i < 6; i += 2) {
            const cfx dd = ld_cfx(ap + (int64_t)(blk * 18 + (i >> 1)) * g.Vd);
            fx_mac(t[i], dd.re, x[i].re);
            fx_mac(t[6 + i], dd.re, x[i].im);
            fx_mac(t[i + 1], dd.im, x[i + 1].re);
            fx_mac(t[7 + i], dd.im, x[i + 1].im);
        }
        int k = 3;
#pragma unroll
        for (int i = 0; i < 6; i++)
#pragma unroll
            for (int j = i + 1; j < 6; j++) {
                const cfx m = ld_cfx(ap + (int64_t)(blk * 18 + k) * g.Vd);
                fxacc w[4] = {t[i], t[6 + i], t[j], t[6 + j]};
                fx_mac4(w, m.re, x[j].re, x[j].im, x[i].re, x[i].im);
                fx_mac4(w, m.im, fx{-x[j].im.hi, -x[j].im.lo}, x[j].re, x[i].im, fx{-x[i].re.hi, -x[i].re.lo});
                t[i] = w[0];
                t[6 + i] = w[1];
                t[j] = w[2];
                t[6 + j] = w[3];
                k++;
            }
        double2 y[6];
#pragma unroll
        for (int i = 0; i < 6; i++)
            y[i] = make_double2(fma(-kappa, fx_to_double(hop_sum[12 * blk + 2 * i][threadIdx.x], ch),
                                    fx_to_double(fx_value(t[i]), ca)),
                                fma(-kappa, fx_to_double(hop_sum[12 * blk + 2 * i + 1][threadIdx.x], ch),
                                    fx_to_double(fx_value(t[6 + i]), ca)));
        store6(blk, y);
    }
}

// component k of site ss of domain dd as the caller has it
__device__ __forceinline__ cpx<double> fx_source(const Geom &g, const FxArgs &f, int64_t r, int dd, int ss, int k)
{
    if (f.src.kind == kFxPlanes32) {
        const float2 v = __ldg((const float2 *)f.src.p + (r * g.V + (int64_t)dd * g.Vd) * 12 + (int64_t)k * g.Vd + ss);
        return mk(f2d(v.x), f2d(v.y));
    }
    const double2 *p = (const double2 *)f.src.p;
    const double2 v = f.src.kind == kFxHost64 ? __ldg(p + (r * g.V + __ldg(f.site_of + dd * g.Vd + ss)) * 12 + k)
                                              : __ldg(p + (r * g.V + (int64_t)dd * g.Vd) * 12 + (int64_t)k * g.Vd + ss);
    return mk(v.x, v.y);
}

template <bool RESID, bool HOST>
__device__ __forceinline__ void fx_store64(const Geom &g, const FxArgs &f, int64_t r, int d, int s, int k, double2 y)
{
    const int64_t plane = (r * g.V + (int64_t)d * g.Vd) * 12 + (int64_t)k * g.Vd + s;
    if (RESID) {
        const double2 v = __ldg(f.b + plane);
        y = make_double2(v.x - y.x, v.y - y.y);
    }
    if (HOST) f.out[(r * g.V + __ldg(f.site_of + d * g.Vd + s)) * 12 + k] = y;
    else f.out[plane] = y;
}

// one site by one thread
template <bool RESID, bool HOST>
__device__ __noinline__ void dslash_site64(const Geom &g, const FxArgs &f, int64_t r, int d, int s, double kappa)
{
    cpx<double> acc[12], x[12], u[9];
#pragma unroll
    for (int k = 0; k < 12; k++) acc[k] = mk(0.0, 0.0);
    auto load = [&](int dir) {
        const int back = dir & 1;
        const uint16_t e = __ldg(g.nbl + s * 8 + dir);
        const int nd = (e & kCross) ? __ldg(g.nbd + d * 8 + dir) : d, ns = e & kSlotMask;
        if (!(QDD_IN_RANGE(nd, 0, g.Nd) && QDD_IN_RANGE(ns, 0, g.Vd))) return false;
#pragma unroll
        for (int k = 0; k < 12; k++) x[k] = fx_source(g, f, r, nd, ns, k);
        const double2 *U = f.U64 + ((int64_t)(back ? nd : d) * 36 + (dir >> 1) * 9) * g.Vd + (back ? ns : s);
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const double2 v = __ldg(U + (int64_t)k * g.Vd);
            u[k] = mk(v.x, v.y);
        }
        return true;
    };
    if (load(0)) hop<0, +1>(u, x, acc);
    if (load(1)) hop<0, -1>(u, x, acc);
    if (load(2)) hop<1, +1>(u, x, acc);
    if (load(3)) hop<1, -1>(u, x, acc);
    if (load(4)) hop<2, +1>(u, x, acc);
    if (load(5)) hop<2, -1>(u, x, acc);
    if (load(6)) hop<3, +1>(u, x, acc);
    if (load(7)) hop<3, -1>(u, x, acc);
#pragma unroll
    for (int blk = 0; blk < 2; blk++) {
        cpx<double> m[18], z[6];
#pragma unroll
        for (int k = 0; k < 18; k++) {
            const double2 v = __ldg(f.A64 + ((int64_t)d * 36 + blk * 18 + k) * g.Vd + s);
            m[k] = mk(v.x, v.y);
        }
#pragma unroll
        for (int k = 0; k < 6; k++) x[k] = fx_source(g, f, r, d, s, 6 * blk + k);
        herm6_mul(m, x, z);
#pragma unroll
        for (int k = 0; k < 6; k++)
            fx_store64<RESID, HOST>(g, f, r, d, s, 6 * blk + k,
                                    make_double2(fma(-kappa, acc[6 * blk + k].re, z[k].re),
                                                 fma(-kappa, acc[6 * blk + k].im, z[k].im)));
    }
}

// The listed sites in FP64, from the FP64 links and clover and the spinors as they
// were before their conversion.  A short list by a warp per site: lane 6 mu + 3 sp + a
// takes direction mu, both signs, spin sp of the half spinor, colour a of its product
// (36 FP64 operations); lane k then adds component k of the hop sum, and lanes k
// and 12 + k take three columns each of its clover row.  With one thread per site
// the FP64 pipe (a warp's instruction takes 64 clocks of a quarter SM) would make
// a list of one site 38 us long; about 70 instructions make it 3.  But 70 are also
// twice a site's share of 1140 (5.2 against 2.7 ns per site), so a list of more than 16
// sites per warp of the grid, where both take about 200 us (one thread per site waits
// on its scattered loads that long), goes by one thread per site.  Few sites are
// listed on ordinary fields, and an empty list takes 2.4 us.
// Measured, 24x16x12x32 with the fixed-point kernel (no site listed 101 us, FP64
// arithmetic 316): a point source 107, a time slice 111, one colour 171 (a tenth of the
// sites), even sites only 317 (half of them; 502 by warps), one colour on a nearly unit
// field 507 (all; 874 by warps).
template <bool RESID, bool HOST>
__global__ void __launch_bounds__(128) k_dslash_list(Geom g, FxArgs f, double kappa)
{
    const int lane = threadIdx.x & 31, n = f.list[0];
    if (n > 16 * (int)(gridDim.x * (blockDim.x / 32))) {
        for (int i = ((threadIdx.x / 32) * gridDim.x + blockIdx.x) * 32 + lane; i < n; i += gridDim.x * blockDim.x) {
            const int at = f.list[1 + i];
            int d, s;
            split_index(g, at % g.V, d, s);
            dslash_site64<RESID, HOST>(g, f, at / g.V, d, s, kappa);
        }
        return;
    }
    const int mu = min(lane / 6, 3), k6 = lane % 6, sp = k6 / 3, a = k6 % 3;
    const int ls = mu < 2 ? 1 - sp : sp;  // the lower spin that meets upper spin sp
    for (int i = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; i < n; i += gridDim.x * (blockDim.x / 32)) {
        const int at = f.list[1 + i], gi = at % g.V;
        const int64_t r = at / g.V;
        int d, s;
        split_index(g, gi, d, s);
        cpx<double> up = mk(0.0, 0.0), lo = mk(0.0, 0.0);
#pragma unroll
        for (int back = 0; back < 2; back++) {
            const uint16_t e = __ldg(g.nbl + s * 8 + 2 * mu + back);
            const int nd = (e & kCross) ? __ldg(g.nbd + d * 8 + 2 * mu + back) : d, ns = e & kSlotMask;
            if (!(QDD_IN_RANGE(nd, 0, g.Nd) && QDD_IN_RANGE(ns, 0, g.Vd))) continue;
            const double2 *U = f.U64 + ((int64_t)(back ? nd : d) * 36 + mu * 9) * g.Vd + (back ? ns : s);
            // h = u + q A l, q = -1 forward and 1 backward; A: x (-i, -i), y (-1, 1), z (-i, i), t (1, 1)
            const double q = ((mu == 1 && sp == 0) || (mu == 2 && sp == 1)) == (back == 1) ? -1.0 : 1.0;
            cpx<double> w = mk(0.0, 0.0);
#pragma unroll
            for (int b = 0; b < 3; b++) {
                const cpx<double> u = fx_source(g, f, r, nd, ns, sp * 3 + b), l = fx_source(g, f, r, nd, ns, 6 + ls * 3 + b);
                const cpx<double> h = (mu & 1) == 0 ? mk(fma(q, l.im, u.re), fma(-q, l.re, u.im))
                                                    : mk(fma(q, l.re, u.re), fma(q, l.im, u.im));
                const double2 v = __ldg(U + (int64_t)(back ? b * 3 + a : a * 3 + b) * g.Vd);
                cfma(w, mk(v.x, back ? -v.y : v.y), h);
            }
            up = up + w;
            // q A^+ w: the conjugate phase
            lo = lo + ((mu & 1) == 0 ? mk(-q * w.im, q * w.re) : mk(q * w.re, q * w.im));
        }
        const int k = lane % 12, blk = k / 6, row = k % 6;
        cpx<double> hop = mk(0.0, 0.0);
#pragma unroll
        for (int m = 0; m < 4; m++) {
            // lower spin row / 3 comes from upper spin 1 - row / 3 in x and y
            const int from = m * 6 + (blk && m < 2 ? (row + 3) % 6 : row);
            const cpx<double> ua = mk(__shfl_sync(0xffffffffu, up.re, from), __shfl_sync(0xffffffffu, up.im, from));
            const cpx<double> la = mk(__shfl_sync(0xffffffffu, lo.re, from), __shfl_sync(0xffffffffu, lo.im, from));
            hop = hop + (blk ? la : ua);
        }
        cpx<double> y = mk(0.0, 0.0);
        const double2 *A = f.A64 + ((int64_t)d * 36 + blk * 18) * g.Vd + s;
        const int col0 = lane >= 12 && lane < 24 ? 3 : 0;
#pragma unroll
        for (int c = col0, m = 0; m < 3; m++, c++) {
            const cpx<double> x = fx_source(g, f, r, d, s, blk * 6 + c);
            if (c == row) {
                const double2 v = __ldg(A + (int64_t)(c >> 1) * g.Vd);
                const double dg = c & 1 ? v.y : v.x;
                y.re = fma(dg, x.re, y.re);
                y.im = fma(dg, x.im, y.im);
            } else {
                const int p = min(row, c), t = max(row, c);
                const double2 v = __ldg(A + (int64_t)(3 + p * 5 - p * (p - 1) / 2 + t - p - 1) * g.Vd);
                cfma(y, mk(v.x, row < c ? v.y : -v.y), x);
            }
        }
        y.re += __shfl_down_sync(0xffffffffu, y.re, 12);
        y.im += __shfl_down_sync(0xffffffffu, y.im, 12);
        if (lane < 12)
            fx_store64<RESID, HOST>(g, f, r, d, s, k, make_double2(fma(-kappa, hop.re, y.re), fma(-kappa, hop.im, y.im)));
    }
}

// A spinor field in internal planes (FP64 or FP32) into fixed point.
template <typename SI>
__global__ void __launch_bounds__(128) k_spinor_fx(Geom g, const typename SI::T2 *src, int4 *x, int *xe)
{
    const int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= g.V) return;
    const int64_t r = blockIdx.y, rbase = r * (int64_t)g.V * 12;
    if (gi == 0 && r == 0) xe[(int64_t)g.V * gridDim.y] = 0;  // the operator's list is empty
    int d, s;
    split_index(g, gi, d, s);
    cpx<double> v[12];
#pragma unroll
    for (int k = 0; k < 12; k++) {
        const typename SI::T2 a = __ldg(src + rbase + ((int64_t)d * 12 + k) * g.Vd + s);
        if constexpr (SI::kBytes == 16) v[k] = mk((double)a.x, (double)a.y);
        else v[k] = mk(f2d(a.x), f2d(a.y));
    }
    fx_store_site(x + rbase + (int64_t)d * 12 * g.Vd, s, g.Vd, xe + r * g.V + gi, v);
}

// Links (one scale) and clover (a scale per site) into fixed point.
__global__ void k_links_fx(int64_t n, const double2 *src, int4 *dst, int lsh)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double2 a = __ldg(src + i);
    // |U| <= 2^(60 - lsh) here; rounded at 2^-lsh
    auto conv = [&](double v) {
        const int ex = fx_exponent(v);
        const uint32_t hi = (uint32_t)__double2hiint(v);
        const uint64_t m = ex ? ((uint64_t)((hi & 0x000fffffu) | 0x00100000u) << 32 | (uint32_t)__double2loint(v)) : 0;
        const int sh = ex - 1075 + lsh;  // v 2^lsh = m 2^sh
        const uint64_t x = sh >= 0 ? m << sh : (sh > -63 ? (m + (1ull << (-sh - 1))) >> -sh : 0);
        return fx_split((int32_t)hi < 0 ? -(int64_t)x : (int64_t)x);
    };
    const fx re = conv(a.x), im = conv(a.y);
    dst[i] = make_int4(re.hi, re.lo, im.hi, im.lo);
}

// ae[g.V] (zero at the launch) takes the largest exponent in magnitude.
__global__ void __launch_bounds__(128) k_clover_fx(Geom g, const double2 *src, int4 *dst, int *ae)
{
    const int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= g.V) return;
    int d, s;
    split_index(g, gi, d, s);
    const double2 *p = src + (int64_t)d * 36 * g.Vd + s;
    int emax = 1;
    float big = 0.f;  // |Re| + |Im| summed over the rows of a block
#pragma unroll 1
    for (int blk = 0; blk < 2; blk++) {
        float row[6];
        auto entry = [&](int k) {
            const double2 a = __ldg(p + (int64_t)(blk * 18 + k) * g.Vd);
            emax = max(emax, max(fx_exponent(a.x), fx_exponent(a.y)));
            return make_float2(fabsf(d2f(a.x)), fabsf(d2f(a.y)));
        };
#pragma unroll
        for (int i = 0; i < 6; i += 2) {
            const float2 v = entry(i / 2);
            row[i] = v.x;
            row[i + 1] = v.y;
        }
        int k = 3;
#pragma unroll
        for (int i = 0; i < 6; i++)
#pragma unroll
            for (int j = i + 1; j < 6; j++) {
                const float2 v = entry(k++);
                row[i] += v.x + v.y;
                row[j] += v.x + v.y;
            }
#pragma unroll
        for (int i = 0; i < 6; i++) big = fmaxf(big, row[i]);
    }
    // (1 + 1e-6 for the FP32 sums; sites out of FP32's range have no copy)
    if (big > 0x1p-80f && emax < 0x7ff) emax = max(emax, 1022 + fx_ceil_exponent(big * (1.000001f / kFxCloverRow)));
    ae[gi] = emax - 1022;
    const int far = abs(emax - 1022);
    if (far > *(volatile int *)(ae + g.V)) atomicMax(ae + g.V, far);
    int4 *q = dst + (int64_t)d * 36 * g.Vd + s;
    for (int k = 0; k < 36; k++) {
        const double2 a = __ldg(p + (int64_t)k * g.Vd);
        const fx re = fx_from_double(a.x, emax, kFxCloverBits), im = fx_from_double(a.y, emax, kFxCloverBits);
        q[(int64_t)k * g.Vd] = make_int4(re.hi, re.lo, im.hi, im.lo);
    }
}

qdd_status launch_links_fx(Gauge *g, cudaStream_t s)
{
    const int64_t n = (int64_t)g->hg.V * 36;
    LaunchScope ls(g->ctx->timer, K_OTHER, s);
    k_links_fx<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, g->links64.as<double2>(), g->fx.links.as<int4>(),
                                                           kFxLinkBits - g->link_exp);
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

qdd_status launch_clover_fx(Gauge *g, cudaStream_t s)
{
    LaunchScope ls(g->ctx->timer, K_OTHER, s);
    QDD_CUDA(cudaMemsetAsync(g->fx.clov_e.as<int>() + g->hg.V, 0, sizeof(int), s));
    k_clover_fx<<<(g->hg.V + 127) / 128, 128, 0, s>>>(g->geom, g->clov64.as<double2>(), g->fx.clov.as<int4>(),
                                                      g->fx.clov_e.as<int>());
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

qdd_status launch_spinor_fx(Gauge *g, const void *src, qdd_prec ip, const FxField &x, int nrhs, cudaStream_t s)
{
    const dim3 grid((g->hg.V + 127) / 128, nrhs);
    LaunchScope ls(g->ctx->timer, K_DSLASH, s);
    if (ip == QDD_PREC_F64) k_spinor_fx<StF64><<<grid, 128, 0, s>>>(g->geom, (const double2 *)src, (int4 *)x.x, x.e);
    else if (ip == QDD_PREC_F32) k_spinor_fx<StF32><<<grid, 128, 0, s>>>(g->geom, (const float2 *)src, (int4 *)x.x, x.e);
    else {
        set_error("the fixed-point operator takes FP32 or FP64 spinors");
        return QDD_EINVAL;
    }
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

qdd_status launch_dslash_fx(Gauge *g, const FxField &x, const FxInput &src, double2 *out, bool host_layout,
                            const double2 *b, int nrhs, cudaStream_t s)
{
    const FxCopy &c = g->fx;
    const int ush = kFxLinkBits - kFxLimb - (g->su3 ? 6 : 5);
    const float unit = (float)(1 << (kFxLinkBits - kFxLimb - ush + 5));  // of the sums of magnitudes, for 2^(E + u)
    const FxArgs f{c.links.as<int4>(), c.clov.as<int4>(), (const int4 *)x.x, c.clov_e.as<int>(), x.e,
                   x.e + (int64_t)g->hg.V * nrhs, g->link_exp, ush, unit * kFxHop,
                   (float)(unit * kFxClover / std::fabs(g->kappa)), b, out, g->d_site_of.as<int>(),
                   ((uintptr_t)out & 31) == 0, src, g->links64.as<double2>(), g->clov64.as<double2>()};
    const int bt = site_block(g, nrhs);
    const dim3 grid((g->hg.V + bt - 1) / bt, nrhs);
    const bool v256 = g->hg.Vd == 256;  // 4^4 domains: the volume fixed at compile time
    {
        LaunchScope ls(g->ctx->timer, K_DSLASH, s);
        if (b) {
            if (v256) k_dslash_fx<true, false, 256><<<grid, bt, 0, s>>>(g->geom, f, g->kappa);
            else k_dslash_fx<true, false><<<grid, bt, 0, s>>>(g->geom, f, g->kappa);
        } else if (host_layout) {
            if (v256) k_dslash_fx<false, true, 256><<<grid, bt, 0, s>>>(g->geom, f, g->kappa);
            else k_dslash_fx<false, true><<<grid, bt, 0, s>>>(g->geom, f, g->kappa);
        } else {
            if (v256) k_dslash_fx<false, false, 256><<<grid, bt, 0, s>>>(g->geom, f, g->kappa);
            else k_dslash_fx<false, false><<<grid, bt, 0, s>>>(g->geom, f, g->kappa);
        }
    }
    LaunchScope ls(g->ctx->timer, K_DSLASH, s);
    const int nsm = g->ctx->nsm > 0 ? g->ctx->nsm : 148;
    const int64_t blocks = std::min<int64_t>(4 * nsm, ((int64_t)g->hg.V * nrhs + 3) / 4);
    if (b) k_dslash_list<true, false><<<(unsigned)blocks, 128, 0, s>>>(g->geom, f, g->kappa);
    else if (host_layout) k_dslash_list<false, true><<<(unsigned)blocks, 128, 0, s>>>(g->geom, f, g->kappa);
    else k_dslash_list<false, false><<<(unsigned)blocks, 128, 0, s>>>(g->geom, f, g->kappa);
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

// out-of-range indices the kernels of this file have skipped (QDD_CHECK builds)
unsigned long long check_hits_dslash()
{
#ifdef QDD_CHECK
    unsigned long long h = 0;
    if (cudaMemcpyFromSymbol(&h, g_check_hits, sizeof(h)) != cudaSuccess) return ~0ull;
    return h;
#else
    return 0;
#endif
}

template <typename R, typename SL, typename SC, typename SI, typename SO, bool RESID, bool L12 = false>
static qdd_status run_dslash(Gauge *g, Field<SL> U, Field<SC> A, const void *in, const float *in_s, void *out,
                             float *out_s, const double2 *b, int nrhs, cudaStream_t s)
{
    Field<SI> fi{(typename SI::T2 *)in, (float *)in_s};
    Field<SO> fo{(typename SO::T2 *)out, out_s};
    const int bt = site_block(g, nrhs);
    dim3 grid((g->hg.V + bt - 1) / bt, nrhs);
    const HostOut ho{g->d_site_of.as<int>(), ((uintptr_t)out & 31) == 0};
    LaunchScope ls(g->ctx->timer, K_DSLASH, s);
    if (g->hg.Vd == 256)  // 4^4 domains: the volume fixed at compile time
        k_dslash<R, SL, SC, SI, SO, RESID, L12, 256><<<grid, bt, 0, s>>>(g->geom, U, A, fi, fo, b, (R)g->kappa, ho);
    else
        k_dslash<R, SL, SC, SI, SO, RESID, L12><<<grid, bt, 0, s>>>(g->geom, U, A, fi, fo, b, (R)g->kappa, ho);
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

// FP32 arithmetic on links of storage SL: the two-row copy when the gauge
// field allows it, else whole links
template <typename SL, typename SC, typename SI, typename SO, bool RESID = false>
static qdd_status run_dslash_lowp(Gauge *g, qdd_prec fp, Field<SC> A, const void *in, const float *in_s, void *out,
                                  float *out_s, int nrhs, cudaStream_t s, const double2 *b = nullptr)
{
    if (g->two_rows) {
        QDD_TRY(ensure_links12(g, fp, s));
        Field<SL> U{(typename SL::T2 *)g->copies[fp].links12.p, nullptr};
        return run_dslash<float, SL, SC, SI, SO, RESID, true>(g, U, A, in, in_s, out, out_s, b, nrhs, s);
    }
    Field<SL> U{(typename SL::T2 *)g->copies[fp].links.p, nullptr};
    return run_dslash<float, SL, SC, SI, SO, RESID, false>(g, U, A, in, in_s, out, out_s, b, nrhs, s);
}

qdd_status launch_dslash_host(Gauge *g, qdd_prec fp, const void *in, double2 *out, int nrhs, cudaStream_t s)
{
    QDD_TRY(ensure_copy(g, fp, s));
    PrecCopy &c = g->copies[fp];
    if (fp == QDD_PREC_F32)
        return run_dslash_lowp<StF32, StF32, StF32, StHost>(g, fp, Field<StF32>{c.clov.as<float2>(), nullptr}, in,
                                                            nullptr, out, nullptr, nrhs, s);
    if (fp == QDD_PREC_F16S)
        return run_dslash_lowp<StF16, StF16, StF32, StHost>(
            g, fp, Field<StF16>{c.clov.as<__half2>(), c.clov_s.as<float>()}, in, nullptr, out, nullptr, nrhs, s);
    set_error("the operator writes the host layout for FP32 spinors only");
    return QDD_EINVAL;
}

qdd_status launch_dslash_residual32(Gauge *g, const void *in, const double2 *b, float2 *out, cudaStream_t s)
{
    QDD_TRY(ensure_copy(g, QDD_PREC_F32, s));
    const Field<StF32> A{g->copies[QDD_PREC_F32].clov.as<float2>(), nullptr};
    return run_dslash_lowp<StF32, StF32, StF32, StF32, true>(g, QDD_PREC_F32, A, in, nullptr, out, nullptr, 1, s, b);
}

qdd_status launch_dslash(Gauge *g, qdd_prec arith, qdd_prec fp, const void *in, const float *in_s, qdd_prec ip,
                         void *out, float *out_s, qdd_prec op, const double2 *b, int nrhs, cudaStream_t s,
                         const FxField *fxb)
{
    if (!g->have_clover) {
        set_error("set_clover has not been called");
        return QDD_EINVAL;
    }
    // FP64-class arithmetic: in fixed point when the caller has a fixed-point
    // buffer and the fields have their fixed-point copy, else in FP64
    if (arith == QDD_PREC_F64 || arith == QDD_PREC_DF64) {
        if (fp == QDD_PREC_DF64) fp = QDD_PREC_F64;
        if (fxb && op == QDD_PREC_F64 && (ip == QDD_PREC_F64 || ip == QDD_PREC_F32)) {
            FxLock lk;
            QDD_TRY(fx_acquire(g, arith == QDD_PREC_DF64, true, s, lk));
            if (lk.owns_lock()) {
                QDD_TRY(launch_spinor_fx(g, in, ip, *fxb, nrhs, s));
                return launch_dslash_fx(g, *fxb, {in, ip == QDD_PREC_F64 ? kFxPlanes64 : kFxPlanes32}, (double2 *)out,
                                        false, b, nrhs, s);
            }
        }
        if (fp != QDD_PREC_F64 || op != QDD_PREC_F64) {
            set_error("FP64 operator needs FP64 fields and output");
            return QDD_EINVAL;
        }
        Field<StF64> U{g->links64.as<double2>(), nullptr}, A{g->clov64.as<double2>(), nullptr};
        switch (ip) {
        case QDD_PREC_F64:
            return b ? run_dslash<double, StF64, StF64, StF64, StF64, true>(g, U, A, in, in_s, out, out_s, b, nrhs, s)
                     : run_dslash<double, StF64, StF64, StF64, StF64, false>(g, U, A, in, in_s, out, out_s, b, nrhs,
                                                                             s);
        case QDD_PREC_F32:
            return run_dslash<double, StF64, StF64, StF32, StF64, false>(g, U, A, in, in_s, out, out_s, b, nrhs, s);
        default: break;
        }
    } else if (arith == QDD_PREC_F32 && !b) {
        QDD_TRY(ensure_copy(g, fp, s));
        PrecCopy &c = g->copies[fp];
        switch (fp) {
        case QDD_PREC_F32: {
            Field<StF32> A{c.clov.as<float2>(), nullptr};
            if (ip == QDD_PREC_F32 && op == QDD_PREC_F32)
                return run_dslash_lowp<StF32, StF32, StF32, StF32>(g, fp, A, in, in_s, out, out_s, nrhs, s);
            if (ip == QDD_PREC_F32 && op == QDD_PREC_F64)
                return run_dslash_lowp<StF32, StF32, StF32, StF64>(g, fp, A, in, in_s, out, out_s, nrhs, s);
            break;
        }
        case QDD_PREC_F16S: {
            Field<StF16> A{c.clov.as<__half2>(), c.clov_s.as<float>()};
            if (ip == QDD_PREC_F16S && op == QDD_PREC_F16S)
                return run_dslash_lowp<StF16, StF16, StF16, StF16>(g, fp, A, in, in_s, out, out_s, nrhs, s);
            if (ip == QDD_PREC_F32 && op == QDD_PREC_F32)  // half links/clover, single spinors
                return run_dslash_lowp<StF16, StF16, StF32, StF32>(g, fp, A, in, in_s, out, out_s, nrhs, s);
            break;
        }
        case QDD_PREC_BF16S: {
            Field<StBF16> A{c.clov.as<__nv_bfloat162>(), c.clov_s.as<float>()};
            if (ip == QDD_PREC_BF16S && op == QDD_PREC_BF16S)
                return run_dslash_lowp<StBF16, StBF16, StBF16, StBF16>(g, fp, A, in, in_s, out, out_s, nrhs, s);
            break;
        }
        default: break;
        }
    }
    set_error("unsupported operator precision combination (arith %d, fields %d, in %d, out %d)", (int)arith, (int)fp,
              (int)ip, (int)op);
    return QDD_EINVAL;
}

}  // namespace qdd
