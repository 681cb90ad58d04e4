// Domain decomposition geometry and field layout conversions.
//
// The lattice is split into domains of dom[0..3] sites (arXiv:1502.04025,
// Sec. 3.1 and Sec. 3.3: 4^4 and 8x4^3 domains), coloured like a
// checkerboard so that the domains of one colour are independent (Sec. 3.5,
// footnote: n_d = N_d/2 domains can be processed at once).  Each domain's
// data is one contiguous, plane-major block in device memory (Sec. 3.2
// motivates choosing the layout for the algorithm; here it serves coalesced
// warps and single bulk copies into shared memory).
#include <cstdarg>
#include <cstdio>
#include <cstring>

#include "fixed.cuh"
#include "internal.h"

namespace qdd {

// ----------------------------------------------------------------- geometry

static void local_coords(const int dom[4], int Vh, int s, int c[4])
{
    int p = s >= Vh;
    int h = s - p * Vh;
    int l = 2 * h;
    c[0] = l % dom[0];
    l /= dom[0];
    c[1] = l % dom[1];
    l /= dom[1];
    c[2] = l % dom[2];
    c[3] = l / dom[2];
    c[0] += (p + c[1] + c[2] + c[3]) & 1;
}

static int local_slot(const int dom[4], int Vh, const int c[4])
{
    int p = (c[0] + c[1] + c[2] + c[3]) & 1;
    int l = c[0] + dom[0] * (c[1] + dom[1] * (c[2] + dom[2] * c[3]));
    return p * Vh + (l >> 1);
}

qdd_status make_geometry(const int L[4], const int dom[4], HostGeom &hg)
{
    long long V = 1;
    hg.Vd = 1;
    hg.Nd = 1;
    for (int mu = 0; mu < 4; mu++) {
        if (L[mu] <= 0 || dom[mu] < 2 || dom[mu] % 2 || L[mu] % dom[mu]) {
            set_error("invalid geometry: L[%d]=%d dom[%d]=%d (dom must be even and divide L)", mu, L[mu], mu,
                      dom[mu]);
            return QDD_EINVAL;
        }
        int nb = L[mu] / dom[mu];
        if (nb < 2 || nb % 2) {
            set_error("invalid geometry: L[%d]/dom[%d] = %d blocks; need an even number >= 2", mu, mu, nb);
            return QDD_EINVAL;
        }
        hg.L[mu] = L[mu];
        hg.dom[mu] = dom[mu];
        hg.nb[mu] = nb;
        V *= L[mu];
        hg.Vd *= dom[mu];
        hg.Nd *= nb;
    }
    if (hg.Vd > 512) {
        set_error("domain volume %d exceeds 512 sites", hg.Vd);
        return QDD_EINVAL;
    }
    if (V > (1LL << 30)) {
        set_error("lattice volume %lld too large", V);
        return QDD_EINVAL;
    }
    hg.V = (int)V;
    hg.Vh = hg.Vd / 2;
    hg.Nd2 = hg.Nd / 2;

    // slot <-> block: slot = colour*Nd/2 + (block >> 1)
    hg.slot_block.assign(hg.Nd, -1);
    hg.block_slot.assign(hg.Nd, -1);
    std::vector<int> &block_slot = hg.block_slot;
    for (int b = 0; b < hg.Nd; b++) {
        int bc[4], t = b;
        for (int mu = 0; mu < 4; mu++) {
            bc[mu] = t % hg.nb[mu];
            t /= hg.nb[mu];
        }
        int colour = (bc[0] + bc[1] + bc[2] + bc[3]) & 1;
        int slot = colour * hg.Nd2 + (b >> 1);
        hg.slot_block[slot] = b;
        block_slot[b] = slot;
    }
    for (int d = 0; d < hg.Nd; d++)
        if (hg.slot_block[d] < 0) {
            set_error("internal error: domain slot map is not a bijection");
            return QDD_EINVAL;
        }

    // local neighbour table
    hg.nbl.assign((size_t)hg.Vd * 8, 0);
    for (int s = 0; s < hg.Vd; s++) {
        int c[4];
        local_coords(hg.dom, hg.Vh, s, c);
        if (local_slot(hg.dom, hg.Vh, c) != s) {
            set_error("internal error: site slot map is not a bijection");
            return QDD_EINVAL;
        }
        for (int mu = 0; mu < 4; mu++)
            for (int b = 0; b < 2; b++) {
                int cc[4] = {c[0], c[1], c[2], c[3]};
                cc[mu] += b ? -1 : 1;
                uint16_t cross = 0;
                if (cc[mu] < 0 || cc[mu] >= hg.dom[mu]) {
                    cc[mu] = (cc[mu] + hg.dom[mu]) % hg.dom[mu];
                    cross = kCross;
                }
                hg.nbl[(size_t)s * 8 + 2 * mu + b] = (uint16_t)(local_slot(hg.dom, hg.Vh, cc) | cross);
            }
    }
    // face slots: the hops that leave a domain, direction by direction; within
    // direction mu (either sign) a site's slot is the lexicographic index of
    // its coordinates transverse to mu, shared by the site across the face
    hg.nf = 0;
    for (int dir = 0; dir < 8; dir++) {
        hg.foff[dir] = hg.nf;
        hg.nf += hg.Vd / hg.dom[dir >> 1];
    }
    hg.fcoord.assign(hg.Vd, 0);
    for (int s = 0; s < hg.Vd; s++) {
        int c[4];
        local_coords(hg.dom, hg.Vh, s, c);
        uint32_t packed = 0;
        for (int mu = 0; mu < 4; mu++) {
            int t = 0, stride = 1;
            for (int nu = 0; nu < 4; nu++)
                if (nu != mu) {
                    t += c[nu] * stride;
                    stride *= hg.dom[nu];
                }
            packed |= (uint32_t)t << (8 * mu);  // t < Vd / dom[mu] <= 256
        }
        hg.fcoord[s] = packed;
    }
    // domain neighbour table
    hg.nbd.assign((size_t)hg.Nd * 8, 0);
    for (int d = 0; d < hg.Nd; d++) {
        int b = hg.slot_block[d], bc[4], t = b;
        for (int mu = 0; mu < 4; mu++) {
            bc[mu] = t % hg.nb[mu];
            t /= hg.nb[mu];
        }
        for (int mu = 0; mu < 4; mu++)
            for (int st = 0; st < 2; st++) {
                int cc[4] = {bc[0], bc[1], bc[2], bc[3]};
                cc[mu] = (cc[mu] + (st ? -1 : 1) + hg.nb[mu]) % hg.nb[mu];
                int nbk = cc[0] + hg.nb[0] * (cc[1] + hg.nb[1] * (cc[2] + hg.nb[2] * cc[3]));
                hg.nbd[(size_t)d * 8 + 2 * mu + st] = block_slot[nbk];
            }
    }
    // internal index -> host site index: the domain's origin plus the site's
    // offset, the same in every domain (per site coordinates of 131072 sites
    // took 0.7 ms of a gauge field's creation)
    auto lex = [&](const int x[4]) { return x[0] + hg.L[0] * (x[1] + hg.L[1] * (x[2] + hg.L[2] * x[3])); };
    std::vector<int> off(hg.Vd);
    for (int s = 0; s < hg.Vd; s++) {
        int c[4];
        local_coords(hg.dom, hg.Vh, s, c);
        off[s] = lex(c);
    }
    hg.site_of.resize(hg.V);
    for (int d = 0; d < hg.Nd; d++) {
        int t = hg.slot_block[d], x[4];
        for (int mu = 0; mu < 4; mu++) {
            x[mu] = t % hg.nb[mu] * hg.dom[mu];
            t /= hg.nb[mu];
        }
        const int base = lex(x);
        int *out = hg.site_of.data() + (size_t)d * hg.Vd;
        for (int s = 0; s < hg.Vd; s++) out[s] = base + off[s];
    }
    return QDD_OK;
}

// ------------------------------------------------------------------ kernels

// threads of a block of the one-thread-per-site conversions (at most)
constexpr int kSiteThreads = 128;

// Spinor conversions between the host layout (FP64, one site's 12 components
// contiguous) and the internal storages.  Bound by memory: the conversions
// themselves are integer operations (d2f, f2d, mul_f2d), and a site's 192
// bytes move as six 32-byte accesses, whole sectors (aligned host buffers;
// `a32` false: 16 bytes at a time).  Measured on 32^3x64, per right-hand side,
// against the conversion instructions and 16-byte accesses (89 us at the
// measured HBM rate for FP32): in, FP32 95 -> 92 us, BF16 316 -> 94 us; out,
// FP32 250 -> 92 us, FP64 336 -> 116 us; FP16 in, 12 x 16^3x32, 240 -> 69 us.

// one component of an unscaled storage
__device__ __forceinline__ void st_d(double2 *p, cpx<double> v) { *p = make_double2(v.re, v.im); }
__device__ __forceinline__ void st_d(float2 *p, cpx<double> v) { *p = make_float2(d2f(v.re), d2f(v.im)); }
__device__ __forceinline__ void st_d(__half2 *p, cpx<double> v) { *p = __floats2half2_rn(d2f(v.re), d2f(v.im)); }
__device__ __forceinline__ void st_d(__nv_bfloat162 *p, cpx<double> v)
{
    *p = __floats2bfloat162_rn(d2f(v.re), d2f(v.im));
}

// The 12 components y of a site in a 16-bit storage with its scale (largest
// component), in FP32 arithmetic.
template <typename S>
__device__ __forceinline__ void store_scaled(Field<S> f, int64_t base, int64_t sbase, int Vd, int d, int s,
                                             const cpx<float> *y)
{
    float m = 0.f;
#pragma unroll
    for (int k = 0; k < 12; k++) m = fmaxf(m, fmaxf(fabsf(y[k].re), fabsf(y[k].im)));
    f.scale[sbase + (int64_t)d * Vd + s] = m;
    const float inv = m > 0.f ? 1.f / m : 0.f;
    cpx<float> v[12];
#pragma unroll
    for (int k = 0; k < 12; k++) v[k] = inv * y[k];
    st_sp_site<float, S>(f.p + base + (int64_t)d * 12 * Vd, s, Vd, v);
}

// FP64 (re, im) divided by the site's scale m, rounded through FP32 to 16 bits.
// y: the same in FP32; inv = 1 / m in FP32 (0 and small = true where m is near
// the end of its range).
template <typename T2>
__device__ __forceinline__ uint32_t scaled_word(double re, double im, cpx<float> y, float m, float inv, bool small)
{
    const T2 *tag = nullptr;
    const float a = inv * y.re, b = inv * y.im;
    const float lo = 1.f - 0x1p-21f, hi = 1.f + 0x1p-21f;
    const uint32_t w = f2_word(a * lo, b * lo, tag);
    if (!small && w == f2_word(a * hi, b * hi, tag)) return w;
    asm volatile("" : "+f"(m));  // the FP64 division stays on this path (hoisted, it would run for every site)
    const double inv64 = m > 0.f ? 1.0 / (double)m : 0.0;
    return f2_word((float)(re * inv64), (float)(im * inv64), tag);
}

// The 12 FP64 components v of a site in a 16-bit storage: each is the FP64
// quotient by the site's scale, rounded (through FP32) to 16 bits.  FP64
// multiplications would bind the pass (24 per site at 2 per clock and SM), so
// the quotient is taken in FP32, where it is within 2^-22 of the FP64 one, and
// the two 16-bit roundings of the interval of 2^-21 around it are compared:
// where they agree, that is the result; where a rounding boundary lies between
// them (one value in 2^11 for FP16, 2^14 for BF16) the FP64 product decides.
// Sites whose scale is near the end of FP32's range take FP64 throughout.
template <typename S>
__device__ __forceinline__ void store_scaled_d(Field<S> f, int64_t base, int64_t sbase, int Vd, int d, int s,
                                               const cpx<double> *v)
{
    cpx<float> y[12];
    float m = 0.f;
#pragma unroll
    for (int k = 0; k < 12; k++) {
        y[k] = mk(d2f(v[k].re), d2f(v[k].im));
        m = fmaxf(m, fmaxf(fabsf(y[k].re), fabsf(y[k].im)));
    }
    f.scale[sbase + (int64_t)d * Vd + s] = m;
    const bool small = m < 0x1p-100f;
    const float inv = small ? 0.f : 1.f / m;
    uint32_t w[12];
#pragma unroll
    for (int k = 0; k < 12; k++) w[k] = scaled_word<typename S::T2>(v[k].re, v[k].im, y[k], m, inv, small);
    typename S::T2 *p = f.p + base + (int64_t)d * 12 * Vd;
    if constexpr (S::kQuad) {
        uint4 *q = reinterpret_cast<uint4 *>(p) + s;
#pragma unroll
        for (int j = 0; j < 3; j++) q[(int64_t)j * Vd] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
    } else {
        uint32_t *q = reinterpret_cast<uint32_t *>(p) + s;
#pragma unroll
        for (int k = 0; k < 12; k++) q[(int64_t)k * Vd] = w[k];
    }
}

template <typename S>
__device__ __forceinline__ void store_spinor(Field<S> f, int64_t base, int64_t sbase, int Vd, int d, int s,
                                             const cpx<double> *v)
{
    if constexpr (S::kScaled) {
        store_scaled_d<S>(f, base, sbase, Vd, d, s, v);
    } else {
        typename S::T2 *p = f.p + base + (int64_t)d * 12 * Vd + s;
#pragma unroll
        for (int k = 0; k < 12; k++) st_d(p + (int64_t)k * Vd, v[k]);
    }
}

template <typename S>
__device__ __forceinline__ void load_spinor_d(Field<S> f, int64_t base, int64_t sbase, int Vd, int d, int s,
                                              cpx<double> *v)
{
    if constexpr (S::kBytes == 16) {
        const double2 *p = f.p + base + (int64_t)d * 12 * Vd + s;
#pragma unroll
        for (int k = 0; k < 12; k++) v[k] = ld_c<double>(p + (int64_t)k * Vd);
    } else {
        cpx<float> y[12];
        ld_sp_site<float, S>(f.p + base + (int64_t)d * 12 * Vd, s, Vd, y);
        if constexpr (S::kScaled) {
            const float sc = f.scale[sbase + (int64_t)d * Vd + s];
#pragma unroll
            for (int k = 0; k < 12; k++) v[k] = mk(mul_f2d(sc, y[k].re), mul_f2d(sc, y[k].im));
        } else {
#pragma unroll
            for (int k = 0; k < 12; k++) v[k] = mk(f2d(y[k].re), f2d(y[k].im));
        }
    }
}

__global__ void k_links_in(Geom g, const int *site_of, const double2 *src, double2 *dst)
{
    int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= g.V) return;
    int d, s;
    split_index(g, gi, d, s);
    const double2 *p = src + (int64_t)__ldg(site_of + gi) * 36;
    for (int k = 0; k < 36; k++) dst[((int64_t)d * 36 + k) * g.Vd + s] = __ldg(p + k);
}

// the 12 components of a site in the host layout
__device__ __forceinline__ void ld_host_site(const double2 *p, bool a32, cpx<double> *v)
{
    double2 a[12];
    if (a32) {
#pragma unroll
        for (int k = 0; k < 12; k += 2) ld_global_x4(p + k, a[k], a[k + 1]);
    } else {
#pragma unroll
        for (int k = 0; k < 12; k++) a[k] = __ldg(p + k);
    }
#pragma unroll
    for (int k = 0; k < 12; k++) v[k] = mk(a[k].x, a[k].y);
}

template <typename S>
__global__ void __launch_bounds__(kSiteThreads) k_spinor_in(Geom g, const int *site_of, const double2 *src,
                                                            Field<S> dst, int64_t rstride, int64_t sstride, bool a32)
{
    int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= g.V) return;
    int r = blockIdx.y;
    int d, s;
    split_index(g, gi, d, s);
    cpx<double> v[12];
    ld_host_site(src + ((int64_t)r * g.V + __ldg(site_of + gi)) * 12, a32, v);
    store_spinor<S>(dst, r * rstride, r * sstride, g.Vd, d, s, v);
}

// the same into fixed point
__global__ void __launch_bounds__(kSiteThreads) k_spinor_in_fx(Geom g, const int *site_of, const double2 *src, int4 *x,
                                                               int *xe, bool a32)
{
    int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= g.V) return;
    const int64_t r = blockIdx.y;
    if (gi == 0 && r == 0) xe[(int64_t)g.V * gridDim.y] = 0;  // the operator's list is empty
    int d, s;
    split_index(g, gi, d, s);
    cpx<double> v[12];
    ld_host_site(src + (r * g.V + __ldg(site_of + gi)) * 12, a32, v);
    fx_store_site(x + (r * g.V + (int64_t)d * g.Vd) * 12, s, g.Vd, xe + r * g.V + gi, v);
}

template <typename S>
__global__ void __launch_bounds__(kSiteThreads) k_spinor_out(Geom g, const int *site_of, Field<S> src, int64_t rstride,
                                                             int64_t sstride, double2 *dst, bool a32)
{
    int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= g.V) return;
    int r = blockIdx.y;
    int d, s;
    split_index(g, gi, d, s);
    cpx<double> v[12];
    load_spinor_d<S>(src, r * rstride, r * sstride, g.Vd, d, s, v);
    double2 *p = dst + ((int64_t)r * g.V + __ldg(site_of + gi)) * 12;
    if (a32) {
#pragma unroll
        for (int k = 0; k < 12; k += 2)
            st_global_x4(p + k, make_double2(v[k].re, v[k].im), make_double2(v[k + 1].re, v[k + 1].im));
    } else {
#pragma unroll
        for (int k = 0; k < 12; k++) p[k] = make_double2(v[k].re, v[k].im);
    }
}

template <typename SI, typename SO>
__global__ void __launch_bounds__(kSiteThreads) k_spinor_convert(Geom g, Field<SI> src, Field<SO> dst, int64_t rstride, int64_t sstride)
{
    int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= g.V) return;
    int r = blockIdx.y;
    int d, s;
    split_index(g, gi, d, s);
    cpx<double> v[12];
    load_spinor_d<SI>(src, r * rstride, r * sstride, g.Vd, d, s, v);
    store_spinor<SO>(dst, r * rstride, r * sstride, g.Vd, d, s, v);
}

// v = w / |w| in FP64 (out64, may alias w; |w|^2 from the device) and the
// same vector in a 16-bit storage with its per-site scale, in one pass: the
// Arnoldi step's new basis vector and the Schwarz input made from it.  The
// scaling is the FP64 arithmetic of the plain scaling kernel; the 16-bit copy
// is rounded from the FP32 value.  One thread per site.
template <typename SO>
__global__ void k_scale_convert(Geom g, const double2 *w, const double2 *norm2, double2 *out64, Field<SO> dst)
{
    __shared__ double fs;  // once per block: FP64 square root and division are long on the FP64 pipe
    if (threadIdx.x == 0) {
        double nn = norm2[0].x;
        fs = nn > 0.0 ? 1.0 / sqrt(nn) : 0.0;
    }
    __syncthreads();
    const int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= g.V) return;
    int d, s;
    split_index(g, gi, d, s);
    const double f = fs;
    const int64_t base = (int64_t)d * 12 * g.Vd + s;
    cpx<float> v[12];
#pragma unroll
    for (int k = 0; k < 12; k++) {
        double2 a = w[base + (int64_t)k * g.Vd];
        a = make_double2(a.x * f, a.y * f);
        out64[base + (int64_t)k * g.Vd] = a;
        v[k] = mk(d2f(a.x), d2f(a.y));
    }
    store_scaled<SO>(dst, 0, 0, g.Vd, d, s, v);
}

// whole links in the order the Schwarz kernel stages (ld_link); i runs over the
// destination, so that a warp writes consecutive elements
template <typename S>
__global__ void k_links_convert(int64_t n, int Vd, const double2 *src, typename S::T2 *dst)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    constexpr int W = 16 / S::kBytes;  // entries side by side
    const int64_t link = i / (9 * Vd);  // nine planes of one domain and direction
    const int e = (int)(i - link * 9 * Vd);
    const int k = e < 8 * Vd ? (e / (W * Vd)) * W + e % W : 8, s = e < 8 * Vd ? e % (W * Vd) / W : e - 8 * Vd;
    const int64_t j = link * 9 * Vd + (int64_t)k * Vd + s;
    const double2 a = __ldg(src + j);
    st_d(dst + i, mk(a.x, a.y));
}

// Sets out[0] when a link is not SU(3) to tol: max |(U U^+ - 1)_ij| or
// |det U - 1|; out[1] = 1022 + the largest of the links' exponents u (fixed.cuh; 0x7ff
// and more with a non-finite entry); out[2] = 0x7ff less the smallest such value of a
// link that is not zero.
// One thread per link (domain d, direction mu, site s).
__global__ void k_su3_check(Geom g, const double2 *U, double tol, int *out)
{
    const int64_t li = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (li >= (int64_t)g.V * 4) return;
    const int64_t d = li / (4 * g.Vd);
    const int mu = (int)((li / g.Vd) % 4), s = (int)(li % g.Vd);
    const double2 *p = U + (d * 36 + mu * 9) * g.Vd + s;
    cpx<double> u[9];
    for (int k = 0; k < 9; k++) {
        double2 a = __ldg(p + (int64_t)k * g.Vd);
        u[k] = mk(a.x, a.y);
    }
    int ex = 0;
#pragma unroll
    for (int k = 0; k < 9; k++) ex = max(ex, max(fx_exponent(u[k].re), fx_exponent(u[k].im)));
    // Rows 0 and 1 orthonormal and row 2 the conjugate of their cross product to
    // a tenth of the tolerance imply both conditions; otherwise they are taken
    // as they stand.  (54 FP64 multiply-adds for 170; 16^3x32: 200 -> 60 us)
    double near = 0;
    {
        double n0 = -1.0, n1 = -1.0;
        cpx<double> x01 = mk(0.0, 0.0);
#pragma unroll
        for (int k = 0; k < 3; k++) {
            n0 = fma(u[k].re, u[k].re, fma(u[k].im, u[k].im, n0));
            n1 = fma(u[3 + k].re, u[3 + k].re, fma(u[3 + k].im, u[3 + k].im, n1));
            cfmac(x01, u[k], u[3 + k]);
        }
        near = fmax(fmax(fabs(n0), fabs(n1)), fmax(fabs(x01.re), fabs(x01.im)));
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const int a = (k + 1) % 3, b = (k + 2) % 3;
            cpx<double> t = conj(u[6 + k]);
            cfma(t, -u[a], u[3 + b]);
            cfma(t, u[b], u[3 + a]);
            near = fmax(near, fmax(fabs(t.re), fabs(t.im)));
        }
    }
    const bool su3 = near <= 0.1 * tol && ex < 0x7ff;  // (fmax passes NaN over)
    double dev = 0;
    if (!su3) {
        for (int i = 0; i < 3; i++)
            for (int j = 0; j < 3; j++) {
                cpx<double> t = mk(i == j ? -1.0 : 0.0, 0.0);
                for (int k = 0; k < 3; k++) t = t + u[i * 3 + k] * conj(u[j * 3 + k]);
                dev = fmax(dev, fmax(fabs(t.re), fabs(t.im)));
            }
        cpx<double> det = u[0] * (u[4] * u[8] - u[5] * u[7]) - u[1] * (u[3] * u[8] - u[5] * u[6]) +
                          u[2] * (u[3] * u[7] - u[4] * u[6]);
        dev = fmax(dev, fmax(fabs(det.re - 1.0), fabs(det.im)));
    }
    if (!(dev <= tol) || ex == 0x7ff) atomicOr(out, 1);
    if (su3) {  // u = 0
        if (*(volatile int *)(out + 1) < 1022) atomicMax(out + 1, 1022);
        if (*(volatile int *)(out + 2) < 0x7ff - 1022) atomicMax(out + 2, 0x7ff - 1022);
        return;
    }
    bool zero = true;
    float row[3] = {0.f, 0.f, 0.f}, col[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 9; k++) {
        zero = zero && u[k].re == 0 && u[k].im == 0;
        const float m = fabsf(d2f(u[k].re)) + fabsf(d2f(u[k].im));
        row[k / 3] += m;
        col[k % 3] += m;
    }
    const float l1 = fmaxf(fmaxf(fmaxf(row[0], row[1]), fmaxf(row[2], col[0])), fmaxf(col[1], col[2]));
    // (within 2^60 only: other fields keep FP64 arithmetic; 1 + 1e-6 for the FP32 sums)
    if (l1 > 0x1p-80f && ex < 0x7ff) ex = max(ex, 1022 + fx_ceil_exponent(l1 * (1.000001f / kFxLinkRow)));
    if (ex > *(volatile int *)(out + 1)) atomicMax(out + 1, ex);
    if (!zero && 0x7ff - ex > *(volatile int *)(out + 2)) atomicMax(out + 2, 0x7ff - ex);
}

// The first two rows of every link: 24 planes per site, plane mu*6 + 3*row + col
// (an SU(3) link's third row is the conjugated cross product of the two).
// 16-bit formats are stored with planes paired (pair_index below), so that
// the operator reads two planes with one 8-byte load.
template <typename S>
__global__ void k_links12_convert(Geom g, const double2 *src, typename S::T2 *dst)
{
    int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= g.V) return;
    int d, s;
    split_index(g, gi, d, s);
    for (int mu = 0; mu < 4; mu++)
        for (int k = 0; k < 6; k++) {
            double2 a = __ldg(src + ((int64_t)d * 36 + mu * 9 + k) * g.Vd + s);
            const int p = mu * 6 + k;
            st_d(dst + (S::kBytes == 4 ? pair_index(d, 24, p, g.Vd, s) : ((int64_t)d * 24 + p) * g.Vd + s),
                         mk(a.x, a.y));
        }
}

// clover blocks: 36 planes per site; 16-bit formats get one scale per site (32^3x64
// BF16: FP64 maxima and products 868 us, this form 450)
// (paired: the full-lattice operator's copy, 16-bit planes in pairs; else the
// order the Schwarz kernel stages, ld_clover_blk)
template <typename S>
__global__ void k_clover_convert(Geom g, const double2 *src, Field<S> dst, int paired)
{
    int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= g.V) return;
    int d, s;
    split_index(g, gi, d, s);
    const double2 *p = src + (int64_t)d * 36 * g.Vd + s;
    typename S::T2 *q = dst.p + (int64_t)d * 36 * g.Vd + s;
    float m = 0.f;
    if (S::kScaled) {
        for (int k = 0; k < 36; k++) {
            double2 a = __ldg(p + (int64_t)k * g.Vd);
            m = fmaxf(m, fmaxf(fabsf(d2f(a.x)), fabsf(d2f(a.y))));
        }
        dst.scale[gi] = m;
    }
    const bool small = m < 0x1p-100f;
    const float inv = small ? 0.f : 1.f / m;
    for (int k = 0; k < 36; k++) {
        double2 a = __ldg(p + (int64_t)k * g.Vd);
        typename S::T2 *o = q + (int64_t)k * g.Vd;
        if (paired && S::kBytes == 4) o = dst.p + pair_index(d, 36, k, g.Vd, s);
        else if (!paired) o = dst.p + ((int64_t)d * 36 + k / 18 * 18) * g.Vd + clover_elem<S>(k % 18, g.Vd, s);
        if constexpr (S::kScaled)
            *reinterpret_cast<uint32_t *>(o) =
                scaled_word<typename S::T2>(a.x, a.y, mk(d2f(a.x), d2f(a.y)), m, inv, small);
        else
            st_d(o, mk(a.x, a.y));
    }
}

// -------------------------------------------------------------- launchers

static inline dim3 grid_sites(int V, int nrhs, int bs) { return dim3((V + bs - 1) / bs, nrhs); }

qdd_status launch_links_to_internal(Gauge *g, const double *src, cudaStream_t s)
{
    LaunchScope ls(g->ctx->timer, K_OTHER, s);
    k_links_in<<<grid_sites(g->hg.V, 1, 256), 256, 0, s>>>(g->geom, g->d_site_of.as<int>(), (const double2 *)src,
                                                           g->links64.as<double2>());
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

#define QDD_DISPATCH_PREC(prec, S, ...)                   \
    switch (prec) {                                       \
    case QDD_PREC_F64: { using S = StF64; __VA_ARGS__; break; } \
    case QDD_PREC_F32: { using S = StF32; __VA_ARGS__; break; } \
    case QDD_PREC_F16S: { using S = StF16; __VA_ARGS__; break; } \
    case QDD_PREC_BF16S: { using S = StBF16; __VA_ARGS__; break; } \
    default: set_error("invalid precision %d", (int)prec); return QDD_EINVAL; \
    }

qdd_status launch_spinor_in(Gauge *g, const double *src, void *dst, float *dst_scale, qdd_prec prec, int nrhs,
                            cudaStream_t s)
{
    const HostGeom &hg = g->hg;
    int64_t rs = (int64_t)hg.V * 12, ss = hg.V;
    const int bt = site_block(g, nrhs);
    LaunchScope ls(g->ctx->timer, K_OTHER, s);
    QDD_DISPATCH_PREC(prec, S, {
        Field<S> f{(typename S::T2 *)dst, dst_scale};
        k_spinor_in<S><<<grid_sites(hg.V, nrhs, bt), bt, 0, s>>>(
            g->geom, g->d_site_of.as<int>(), (const double2 *)src, f, rs, ss, ((uintptr_t)src & 31) == 0);
    });
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

qdd_status launch_spinor_in_fx(Gauge *g, const double *src, const FxField &x, int nrhs, cudaStream_t s)
{
    const HostGeom &hg = g->hg;
    const int bt = site_block(g, nrhs);
    LaunchScope ls(g->ctx->timer, K_OTHER, s);
    k_spinor_in_fx<<<grid_sites(hg.V, nrhs, bt), bt, 0, s>>>(
        g->geom, g->d_site_of.as<int>(), (const double2 *)src, (int4 *)x.x, x.e, ((uintptr_t)src & 31) == 0);
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

qdd_status launch_spinor_out(Gauge *g, const void *src, const float *src_scale, double *dst, qdd_prec prec, int nrhs,
                             cudaStream_t s)
{
    const HostGeom &hg = g->hg;
    int64_t rs = (int64_t)hg.V * 12, ss = hg.V;
    const int bt = site_block(g, nrhs);
    LaunchScope ls(g->ctx->timer, K_OTHER, s);
    QDD_DISPATCH_PREC(prec, S, {
        Field<S> f{(typename S::T2 *)src, (float *)src_scale};
        k_spinor_out<S><<<grid_sites(hg.V, nrhs, bt), bt, 0, s>>>(
            g->geom, g->d_site_of.as<int>(), f, rs, ss, (double2 *)dst, ((uintptr_t)dst & 31) == 0);
    });
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

qdd_status launch_spinor_convert(Gauge *g, const void *src, const float *src_scale, qdd_prec sp, void *dst,
                                 float *dst_scale, qdd_prec dp, int nrhs, cudaStream_t s)
{
    const HostGeom &hg = g->hg;
    int64_t rs = (int64_t)hg.V * 12, ss = hg.V;
    dim3 grid = grid_sites(hg.V, nrhs, kSiteThreads);
    LaunchScope ls(g->ctx->timer, K_OTHER, s);
    QDD_DISPATCH_PREC(sp, SI, {
        Field<SI> fi{(typename SI::T2 *)src, (float *)src_scale};
        QDD_DISPATCH_PREC(dp, SO, {
            Field<SO> fo{(typename SO::T2 *)dst, dst_scale};
            k_spinor_convert<SI, SO><<<grid, kSiteThreads, 0, s>>>(g->geom, fi, fo, rs, ss);
        });
    });
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

qdd_status launch_scale_convert(Gauge *g, const double2 *w, const double2 *norm2, double2 *out64, void *dst,
                                float *dst_scale, qdd_prec dp, cudaStream_t s)
{
    const int64_t n = (int64_t)g->hg.V * 12;
    g->ctx->timer.work(K_BLAS, 2.0 * n, (32.0 + 4.0) * n + 4.0 * g->hg.V);
    LaunchScope ls(g->ctx->timer, K_BLAS, s);
    const unsigned grid = (unsigned)((g->hg.V + 127) / 128);
    if (dp == QDD_PREC_F16S)
        k_scale_convert<StF16><<<grid, 128, 0, s>>>(g->geom, w, norm2, out64, Field<StF16>{(__half2 *)dst, dst_scale});
    else if (dp == QDD_PREC_BF16S)
        k_scale_convert<StBF16><<<grid, 128, 0, s>>>(g->geom, w, norm2, out64,
                                                     Field<StBF16>{(__nv_bfloat162 *)dst, dst_scale});
    else {
        set_error("scale-and-convert takes a 16-bit storage");
        return QDD_EINVAL;
    }
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

qdd_status launch_links_convert(Gauge *g, qdd_prec dp, void *dst, cudaStream_t s)
{
    int64_t n = (int64_t)g->hg.V * 36;
    LaunchScope ls(g->ctx->timer, K_OTHER, s);
    QDD_DISPATCH_PREC(dp, S, {
        k_links_convert<S><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, g->hg.Vd, g->links64.as<double2>(),
                                                                        (typename S::T2 *)dst);
    });
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

qdd_status launch_su3_check(Gauge *g, double tol, int *d_out, cudaStream_t s)
{
    const int64_t n = (int64_t)g->hg.V * 4;
    LaunchScope ls(g->ctx->timer, K_OTHER, s);
    QDD_CUDA(cudaMemsetAsync(d_out, 0, 3 * sizeof(int), s));
    k_su3_check<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(g->geom, g->links64.as<double2>(), tol, d_out);
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

qdd_status launch_links12_convert(Gauge *g, qdd_prec dp, void *dst, cudaStream_t s)
{
    LaunchScope ls(g->ctx->timer, K_OTHER, s);
    QDD_DISPATCH_PREC(dp, S, {
        k_links12_convert<S><<<grid_sites(g->hg.V, 1, 256), 256, 0, s>>>(g->geom, g->links64.as<double2>(),
                                                                          (typename S::T2 *)dst);
    });
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

qdd_status launch_clover_convert(Gauge *g, const double2 *src, qdd_prec dp, void *dst, float *dst_scale,
                                 cudaStream_t s, bool paired)
{
    LaunchScope ls(g->ctx->timer, K_OTHER, s);
    QDD_DISPATCH_PREC(dp, S, {
        Field<S> f{(typename S::T2 *)dst, dst_scale};
        k_clover_convert<S><<<grid_sites(g->hg.V, 1, 256), 256, 0, s>>>(g->geom, src, f, paired ? 1 : 0);
    });
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

}  // namespace qdd
