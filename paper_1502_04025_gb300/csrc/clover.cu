// Clover term of the Wilson-clover operator (arXiv:1502.04025, Sec. 3.1
// names the operator; Sec. 3.6 counts 1848 flop per site for it).
//
//   A(n) = 1 + i kappa c_sw sum_{mu<nu} sigma_{mu nu} F_{mu nu}(n),
//   F_{mu nu} = traceless part of (Q_{mu nu} - Q_{mu nu}^+)/8, Q the four-leaf
//   clover of plaquettes at n in the (mu, nu) plane.
// In the chiral basis sigma_{mu nu} is block diagonal: A is two Hermitian 6x6
// blocks (spins {0,1} and {2,3}), each  1 + i kappa c_sw sum_k sigma_k (x) G_k,
// with G_k = B_k +- E_k, B = (-F_yz, F_xz, -F_xy), E_k = F_kt (+ for the
// upper block, - for the lower).  The even-odd domain solver also needs the
// inverse blocks on odd sites (the Schwarz form keeps A on even sites and
// A^{-1} on odd sites).  Built in FP64 once per (gauge, c_sw, kappa).
#include "fixed.cuh"
#include "internal.h"

namespace qdd {

typedef cpx<double> zd;

struct M3 {
    zd m[9];
};

__device__ __forceinline__ M3 load_link(const Geom &g, const double2 *U, int gi, int mu)
{
    M3 r;
    int d, s;
    split_index(g, gi, d, s);
    const double2 *p = U + ((int64_t)d * 36 + mu * 9) * g.Vd + s;
    for (int k = 0; k < 9; k++) {
        double2 v = __ldg(p + (int64_t)k * g.Vd);
        r.m[k] = mk(v.x, v.y);
    }
    return r;
}

__device__ __forceinline__ M3 mul(const M3 &a, const M3 &b)
{
    M3 r;
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) {
            zd acc = mk(0.0, 0.0);
            for (int k = 0; k < 3; k++) cfma(acc, a.m[i * 3 + k], b.m[k * 3 + j]);
            r.m[i * 3 + j] = acc;
        }
    return r;
}

__device__ __forceinline__ M3 dag(const M3 &a)
{
    M3 r;
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) r.m[i * 3 + j] = conj(a.m[j * 3 + i]);
    return r;
}

__device__ __forceinline__ int nbr(const Geom &g, int gi, int k)
{
    int d, s;
    split_index(g, gi, d, s);
    return neighbour(g, d, s, k);
}

// F_{mu nu} at gi
__device__ M3 field_strength(const Geom &g, const double2 *U, int gi, int mu, int nu)
{
    int n_pm = nbr(g, gi, 2 * mu), n_mm = nbr(g, gi, 2 * mu + 1);
    int n_pn = nbr(g, gi, 2 * nu), n_mn = nbr(g, gi, 2 * nu + 1);
    int n_mm_pn = nbr(g, n_mm, 2 * nu), n_mm_mn = nbr(g, n_mm, 2 * nu + 1);
    int n_pm_mn = nbr(g, n_pm, 2 * nu + 1);
    M3 Umu = load_link(g, U, gi, mu), Unu = load_link(g, U, gi, nu);
    // leaf 1: n -> n+mu -> n+mu+nu -> n+nu -> n
    M3 q = mul(mul(Umu, load_link(g, U, n_pm, nu)), mul(dag(load_link(g, U, n_pn, mu)), dag(Unu)));
    // leaf 2: n -> n+nu -> n+nu-mu -> n-mu -> n
    M3 l = mul(mul(Unu, dag(load_link(g, U, n_mm_pn, mu))),
               mul(dag(load_link(g, U, n_mm, nu)), load_link(g, U, n_mm, mu)));
    for (int k = 0; k < 9; k++) q.m[k] = q.m[k] + l.m[k];
    // leaf 3: n -> n-mu -> n-mu-nu -> n-nu -> n
    l = mul(mul(dag(load_link(g, U, n_mm, mu)), dag(load_link(g, U, n_mm_mn, nu))),
            mul(load_link(g, U, n_mm_mn, mu), load_link(g, U, n_mn, nu)));
    for (int k = 0; k < 9; k++) q.m[k] = q.m[k] + l.m[k];
    // leaf 4: n -> n-nu -> n-nu+mu -> n+mu -> n
    l = mul(mul(dag(load_link(g, U, n_mn, nu)), load_link(g, U, n_mn, mu)),
            mul(load_link(g, U, n_pm_mn, nu), dag(Umu)));
    for (int k = 0; k < 9; k++) q.m[k] = q.m[k] + l.m[k];
    M3 F;
    for (int a = 0; a < 3; a++)
        for (int b = 0; b < 3; b++) F.m[a * 3 + b] = 0.125 * (q.m[a * 3 + b] - conj(q.m[b * 3 + a]));
    zd tr = (1.0 / 3.0) * (F.m[0] + F.m[4] + F.m[8]);
    F.m[0] = F.m[0] - tr;
    F.m[4] = F.m[4] - tr;
    F.m[8] = F.m[8] - tr;
    return F;
}

// Gauss-Jordan inverse of a 6x6 complex matrix with partial pivoting
__device__ bool invert6(zd *M /* 36, overwritten */, zd *inv /* 36 */)
{
    for (int i = 0; i < 36; i++) inv[i] = mk(0.0, 0.0);
    for (int i = 0; i < 6; i++) inv[i * 6 + i] = mk(1.0, 0.0);
    for (int c = 0; c < 6; c++) {
        int piv = c;
        double best = M[c * 6 + c].re * M[c * 6 + c].re + M[c * 6 + c].im * M[c * 6 + c].im;
        for (int r = c + 1; r < 6; r++) {
            double v = M[r * 6 + c].re * M[r * 6 + c].re + M[r * 6 + c].im * M[r * 6 + c].im;
            if (v > best) { best = v; piv = r; }
        }
        if (!(best > 0.0)) return false;
        if (piv != c)
            for (int j = 0; j < 6; j++) {
                zd t = M[c * 6 + j]; M[c * 6 + j] = M[piv * 6 + j]; M[piv * 6 + j] = t;
                t = inv[c * 6 + j]; inv[c * 6 + j] = inv[piv * 6 + j]; inv[piv * 6 + j] = t;
            }
        zd p = M[c * 6 + c];
        zd pinv = (1.0 / best) * conj(p);
        for (int j = 0; j < 6; j++) {
            M[c * 6 + j] = M[c * 6 + j] * pinv;
            inv[c * 6 + j] = inv[c * 6 + j] * pinv;
        }
        for (int r = 0; r < 6; r++) {
            if (r == c) continue;
            zd f = M[r * 6 + c];
            for (int j = 0; j < 6; j++) {
                M[r * 6 + j] = M[r * 6 + j] - f * M[c * 6 + j];
                inv[r * 6 + j] = inv[r * 6 + j] - f * inv[c * 6 + j];
            }
        }
    }
    return true;
}

__device__ __forceinline__ void pack_herm6(const zd *M, double2 *dst, int64_t stride)
{
    dst[0] = make_double2(M[0].re, M[7].re);
    dst[stride] = make_double2(M[14].re, M[21].re);
    dst[2 * stride] = make_double2(M[28].re, M[35].re);
    int k = 3;
    for (int i = 0; i < 6; i++)
        for (int j = i + 1; j < 6; j++) {
            // symmetrise the rounding of the two triangles
            zd v = 0.5 * (M[i * 6 + j] + conj(M[j * 6 + i]));
            dst[k * stride] = make_double2(v.re, v.im);
            k++;
        }
}

// the term of site gi in FP64
__device__ __noinline__ void clover_site(const Geom &g, const double2 *U, int gi, double kc, double2 *A, double2 *S,
                                         int *singular)
{
    int d, s;
    split_index(g, gi, d, s);
    // F in the order (xy, xz, xt, yz, yt, zt)
    M3 Fxy = field_strength(g, U, gi, 0, 1), Fxz = field_strength(g, U, gi, 0, 2);
    M3 Fxt = field_strength(g, U, gi, 0, 3), Fyz = field_strength(g, U, gi, 1, 2);
    M3 Fyt = field_strength(g, U, gi, 1, 3), Fzt = field_strength(g, U, gi, 2, 3);
    bool odd = s >= g.Vh;
    for (int ch = 0; ch < 2; ch++) {
        double se = ch == 0 ? 1.0 : -1.0;
        zd G1[9], G2[9], G3[9];
        for (int k = 0; k < 9; k++) {
            G1[k] = (-1.0) * Fyz.m[k] + se * Fxt.m[k];
            G2[k] = Fxz.m[k] + se * Fyt.m[k];
            G3[k] = (-1.0) * Fxy.m[k] + se * Fzt.m[k];
        }
        zd M[36];
        for (int a = 0; a < 3; a++)
            for (int b = 0; b < 3; b++) {
                zd g3 = G3[a * 3 + b];
                zd c01 = G1[a * 3 + b] - ti(G2[a * 3 + b]);  // (sigma_1 G1 + sigma_2 G2)_{01}
                zd c10 = G1[a * 3 + b] + ti(G2[a * 3 + b]);  // (...)_{10}
                // M = 1 + i kappa c_sw (...)
                M[(0 * 3 + a) * 6 + 0 * 3 + b] = kc * ti(g3);
                M[(1 * 3 + a) * 6 + 1 * 3 + b] = kc * ti(-g3);
                M[(0 * 3 + a) * 6 + 1 * 3 + b] = kc * ti(c01);
                M[(1 * 3 + a) * 6 + 0 * 3 + b] = kc * ti(c10);
            }
        for (int i = 0; i < 6; i++) M[i * 6 + i].re += 1.0;
        const int64_t base = ((int64_t)d * 36 + ch * 18) * g.Vd + s;
        pack_herm6(M, A + base, g.Vd);
        if (!odd) {
            pack_herm6(M, S + base, g.Vd);
        } else {
            zd inv[36];
            if (!invert6(M, inv)) {
                atomicAdd(singular, 1);
                for (int i = 0; i < 36; i++) inv[i] = mk(0.0, 0.0);
            }
            pack_herm6(inv, S + base, g.Vd);
        }
    }
}

__global__ void k_clover_build(Geom g, const double2 *U, double kc, double2 *A, double2 *S, int *singular)
{
    const int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi < g.V) clover_site(g, U, gi, kc, A, S, singular);
}

// ------------------------------------------------------------------------
// The same for SU(3) links, in 64-bit fixed point (fixed.cuh): the 72 matrix
// products of a site's 24 leaves are integer multiply-adds on the links'
// fixed-point copy (entries of SU(3) matrices stay below 1, so every product
// keeps the links' scale 2^-60), the leaf sums, the anti-Hermitian and traceless
// parts and the sums over planes are integers, and FP64 starts at the entries
// of A.  In FP64 arithmetic the 7776 multiply-adds of the leaves take 3900 of
// an SM's clocks per site (2 lanes per clock); as integer multiply-adds they take
// about 360.  Measured on 16^3x32: 2945 -> 741 us, of which the FP64 inverses of
// the odd sites' blocks keep the FP64 pipe busy 17 % (symmetric sweeps: 420 FP64
// operations per block for 1730 of Gauss-Jordan with pivoting); the rest waits
// on integer latencies (2.6 warps per scheduler at 168-255 registers; 128
// registers spill and are no faster).
//
// An entry of a leaf is off by at most 10 2^-60: the links' rounding, each product's
// left-out lower limbs (six of at most 1/4) and rounding, through three products.
// FP64 arithmetic rounds it by up to 18 2^-53 S, S the sum of the magnitudes of the
// last product's terms, and by about 2^-53 S on average.  So a plane's four leaves are
// as good as FP64's where S, added over them, is at least 4 2^-6 for each of the nine
// entries, which the factors' leading six bits show; a site with a smaller one in
// any plane (a field that is nearly the unit field, whose field strength lies that
// far below the leaves' entries) is computed in FP64.

struct M3x {
    cfx m[9];
};

__device__ __forceinline__ M3x load_link_fx(const Geom &g, const int4 *U, int gi, int mu)
{
    M3x r;
    int d, s;
    split_index(g, gi, d, s);
    const int4 *p = U + ((int64_t)d * 36 + mu * 9) * g.Vd + s;
#pragma unroll
    for (int k = 0; k < 9; k++) {
        const int4 v = __ldg(p + (int64_t)k * g.Vd);
        r.m[k] = {{v.x, v.y}, {v.z, v.w}};
    }
    return r;
}

__device__ __forceinline__ M3x fx_mul(const M3x &a, const M3x &b)
{
    M3x r;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            fxacc re = fx_zero(), im = fx_zero();
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const cfx x = a.m[i * 3 + k], y = b.m[k * 3 + j];
                fx_mac2(re, im, x.re, y.re, y.im);
                fx_mac2(im, re, x.im, y.re, fx{-y.im.hi, -y.im.lo});
            }
            r.m[i * 3 + j] = {fx_split(fx_value(re)), fx_split(fx_value(im))};
        }
    return r;
}

__device__ __forceinline__ M3x fx_adjoint(const M3x &u)
{
    M3x r;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const cfx x = u.m[j * 3 + i];
            r.m[i * 3 + j] = {x.re, {-x.im.hi, -x.im.lo}};
        }
    return r;
}

// Q = sum of leaves / 8 (three bits dropped, so that the sums below keep their
// headroom): scale 2^-57 per leaf
struct M3q {
    int64_t re[9], im[9];
};

// the link of the step from n to m = n +- da: U_da(n) forward, U_da(m)^+ backward
__device__ __forceinline__ M3x step_link_fx(const Geom &g, const int4 *U, int n, int m, int da, bool back)
{
    const M3x u = load_link_fx(g, U, back ? m : n, da), v = fx_adjoint(u);
    M3x r;
#pragma unroll
    for (int k = 0; k < 9; k++) {
        r.m[k].re = {back ? v.m[k].re.hi : u.m[k].re.hi, back ? v.m[k].re.lo : u.m[k].re.lo};
        r.m[k].im = {back ? v.m[k].im.hi : u.m[k].im.hi, back ? v.m[k].im.lo : u.m[k].im.lo};
    }
    return r;
}

// 8 F_{mu nu} = traceless part of Q - Q^+ at gi, scale 2^-57, as nine integers:
// the imaginary diagonal, then re and im of the entries (0,1), (0,2), (1,2)
constexpr int kLeafBits = 57;
constexpr uint32_t kLeafLow = 4 * 64 * 64 >> 6;
__device__ __forceinline__ uint32_t lead6(const cfx &x)
{
    return (uint32_t)max(abs(x.re.hi), abs(x.im.hi)) >> (kFxLinkBits - kFxLimb - 6);
}
// low: lowered to the plane's smallest sum of magnitudes, 64^2 for 1
__device__ __forceinline__ void field_strength_fx(const Geom &g, const int4 *U, int gi, int mu, int nu, int64_t *F,
                                                  uint32_t &low)
{
    const int n_pm = nbr(g, gi, 2 * mu), n_mm = nbr(g, gi, 2 * mu + 1);
    const int n_pn = nbr(g, gi, 2 * nu), n_mn = nbr(g, gi, 2 * nu + 1);
    M3q q;
#pragma unroll
    for (int k = 0; k < 9; k++) q.re[k] = q.im[k] = 0;
    uint32_t mag[5] = {0, 0, 0, 0, 0};  // two entries a word: at most 4 3 64^2 < 2^16
    // A leaf runs from n over the steps a, b and back over a, b: X Y^+ with X =
    // link(n, a) link(n + a, b) and Y = link(n, b) link(n + b, a), for (a, b) =
    // (+mu, +nu), (+nu, -mu), (-mu, -nu), (-nu, +mu).  X, Y and X Y^+ run through
    // one copy of the product (three copies: 826 us for 741, instruction fetch).
#pragma unroll 1
    for (int leaf = 0; leaf < 4; leaf++) {
        const bool swap = leaf & 1;
        const int da = swap ? nu : mu, db = swap ? mu : nu;
        const bool ba = leaf >= 2, bb = leaf == 1 || leaf == 2;         // a, b backward
        const int na = swap ? (ba ? n_mn : n_pn) : (ba ? n_mm : n_pm);  // n + a
        const int nb = swap ? (bb ? n_mm : n_pm) : (bb ? n_mn : n_pn);  // n + b
        const int nab = nbr(g, na, 2 * db + (bb ? 1 : 0));
        M3x X, Yd;
#pragma unroll 1
        for (int h = 0; h < 3; h++) {
            M3x l, r;
            if (h < 2) {
                const int m = h ? nb : na;
                l = step_link_fx(g, U, gi, m, h ? db : da, h ? bb : ba);
                r = step_link_fx(g, U, m, nab, h ? da : db, h ? ba : bb);
            } else {
                l = X;
                r = Yd;
            }
            const M3x p = fx_mul(l, r);
            if (h == 0) {
                X = p;
            } else if (h == 1) {
                Yd = fx_adjoint(p);
            } else {
#pragma unroll
                for (int k = 0; k < 9; k++) {
                    q.re[k] += fx_join(p.m[k].re) >> 3;
                    q.im[k] += fx_join(p.m[k].im) >> 3;
                }
#pragma unroll
                for (int i = 0; i < 3; i++)
#pragma unroll
                    for (int j = 0; j < 3; j++)
                        mag[(i * 3 + j) / 2] +=
                            (lead6(l.m[i * 3]) * lead6(r.m[j]) + lead6(l.m[i * 3 + 1]) * lead6(r.m[3 + j]) +
                             lead6(l.m[i * 3 + 2]) * lead6(r.m[6 + j]))
                            << ((i * 3 + j) % 2 * 16);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 9; k++) low = min(low, k % 2 ? mag[k / 2] >> 16 : mag[k / 2] & 0xffffu);
    const int64_t d0 = q.im[0], d1 = q.im[4], d2 = q.im[8], mean = (d0 + d1 + d2) / 3;
    F[0] = 2 * (d0 - mean);
    F[1] = 2 * (d1 - mean);
    F[2] = 2 * (d2 - mean);
    F[3] = q.re[1] - q.re[3];
    F[4] = q.im[1] + q.im[3];
    F[5] = q.re[2] - q.re[6];
    F[6] = q.im[2] + q.im[6];
    F[7] = q.re[5] - q.re[7];
    F[8] = q.im[5] + q.im[7];
}

// Minus the inverse of a Hermitian 6x6 matrix by six symmetric sweeps without
// pivoting, in place: dg the diagonal, u the upper triangle row by row (i < j).
// False (the caller pivots instead) unless every pivot is as large as either part of
// the entries below it when its turn comes, so that a sweep at most doubles the
// rest as partial pivoting does, and no smaller than the largest entry of the
// matrix by 2^6 or more (and not NaN or infinite).  Ordinary terms pass: all blocks at
// kappa c_sw up to 0.4 on links of eps = 0.7, 96 % at 0.6, 22 % at 1, with the
// errors of partial pivoting.  The comparisons are of the numbers' high words: in
// FP64 they would take the FP64 pipe.
__device__ __forceinline__ bool sweep6(double *dg, zd *u)
{
    auto word = [](double v) { return (uint32_t)__double2hiint(v) & 0x7fffffffu; };
    uint32_t big = 0;
#pragma unroll
    for (int i = 0; i < 6; i++) big = max(big, word(dg[i]));
#pragma unroll
    for (int i = 0; i < 15; i++) big = max(big, max(word(u[i].re), word(u[i].im)));
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 6; k++) {
        auto at = [](int i, int j) { return i * 5 - i * (i - 1) / 2 + (j - i - 1); };  // i < j
        uint32_t below = 0;
#pragma unroll
        for (int i = k + 1; i < 6; i++) below = max(below, max(word(u[at(k, i)].re), word(u[at(k, i)].im)));
        const uint32_t piv = word(dg[k]);
        ok = ok && piv >= below && piv + (6u << 20) >= big && piv < 0x7ff00000u;
        const double p = 1.0 / dg[k];
        zd col[6], row[6];  // a_ik, and a_ik / d
#pragma unroll
        for (int i = 0; i < 6; i++) {
            if (i == k) continue;
            col[i] = i < k ? u[at(i, k)] : conj(u[at(k, i)]);
            row[i] = p * col[i];
        }
#pragma unroll
        for (int i = 0; i < 6; i++) {
            if (i == k) continue;
            dg[i] = fma(-row[i].re, col[i].re, dg[i]);
            dg[i] = fma(-row[i].im, col[i].im, dg[i]);
#pragma unroll
            for (int j = i + 1; j < 6; j++) {
                if (j == k) continue;
                zd &t = u[at(i, j)];  // a_ij -= a_ik conj(a_jk) / d
                t.re = fma(-row[i].re, col[j].re, t.re);
                t.re = fma(-row[i].im, col[j].im, t.re);
                t.im = fma(-row[i].im, col[j].re, t.im);
                t.im = fma(row[i].re, col[j].im, t.im);
            }
        }
#pragma unroll
        for (int i = 0; i < 6; i++) {
            if (i < k) u[at(i, k)] = row[i];
            else if (i > k) u[at(k, i)] = conj(row[i]);
        }
        dg[k] = -p;
    }
    return ok;
}

// the inverse with pivoting, for blocks that sweep6 refuses
__device__ __noinline__ bool invert6_packed(const double *dg, const zd *u, double *dgo, zd *uo)
{
    zd M[36], inv[36];
    int k = 0;
    for (int i = 0; i < 6; i++) {
        M[i * 6 + i] = mk(dg[i], 0.0);
        for (int j = i + 1; j < 6; j++) {
            M[i * 6 + j] = u[k];
            M[j * 6 + i] = conj(u[k]);
            k++;
        }
    }
    if (!invert6(M, inv)) return false;
    k = 0;
    for (int i = 0; i < 6; i++) {
        dgo[i] = inv[i * 6 + i].re;
        for (int j = i + 1; j < 6; j++) uo[k++] = 0.5 * (inv[i * 6 + j] + conj(inv[j * 6 + i]));
    }
    return true;
}

__device__ __forceinline__ void store_herm6(double2 *dst, int64_t stride, const double *dg, const zd *u)
{
#pragma unroll
    for (int k = 0; k < 3; k++) dst[k * stride] = make_double2(dg[2 * k], dg[2 * k + 1]);
#pragma unroll
    for (int k = 0; k < 15; k++) dst[(3 + k) * stride] = make_double2(u[k].re, u[k].im);
}

constexpr int kCloverThreads = 64;

__global__ void __launch_bounds__(kCloverThreads, 4) k_clover_build_fx(Geom g, const int4 *U, const double2 *U64,
                                                                    double kc, double2 *A, double2 *S, int *singular)
{
    __shared__ int64_t F[6][9][kCloverThreads];
    const int gi = blockIdx.x * kCloverThreads + threadIdx.x, t = threadIdx.x;
    if (gi >= g.V) return;
    int d, s;
    split_index(g, gi, d, s);
    uint32_t low = ~0u;
#pragma unroll 1
    for (int plane = 0; plane < 6; plane++) {  // xy, xz, xt, yz, yt, zt
        const int mu = plane < 3 ? 0 : (plane < 5 ? 1 : 2), nu = plane < 3 ? plane + 1 : (plane < 5 ? plane - 1 : 3);
        int64_t f[9];
        field_strength_fx(g, U, gi, mu, nu, f, low);
#pragma unroll
        for (int k = 0; k < 9; k++) F[plane][k][t] = f[k];
    }
    if (low < kLeafLow) {
        clover_site(g, U64, gi, kc, A, S, singular);
        return;
    }
    const bool odd = s >= g.Vh;
    constexpr int ex = -kLeafBits - 3;  // F is an eighth of its integers
#pragma unroll 1
    for (int ch = 0; ch < 2; ch++) {
        const int se = ch == 0 ? 1 : -1;
        // G_1 = -F_yz +- F_xt, G_2 = F_xz +- F_yt, G_3 = -F_xy +- F_zt
        int64_t g1[9], g2[9], g3[9];
#pragma unroll
        for (int k = 0; k < 9; k++) {
            g1[k] = se * F[2][k][t] - F[3][k][t];
            g2[k] = F[1][k][t] + se * F[4][k][t];
            g3[k] = se * F[5][k][t] - F[0][k][t];
        }
        // i G is Hermitian: diagonal -im, upper entry (a,b) (-im, re), lower its conjugate
        auto her = [](const int64_t *gk, int a, int b, int64_t &re, int64_t &im) {
            if (a == b) { re = -gk[a]; im = 0; return; }
            const int lo = a < b ? a : b, k = lo == 0 ? (a + b == 1 ? 3 : 5) : 7;
            re = -gk[k + 1];
            im = a < b ? gk[k] : -gk[k];
        };
        double dg[6];
        zd u[15];
        int k = 0;
#pragma unroll
        for (int i = 0; i < 6; i++) {
            const int a = i % 3;
            int64_t re, im;
            her(g3, a, a, re, im);
            dg[i] = fma(i < 3 ? kc : -kc, fx_to_double(re, ex), 1.0);
#pragma unroll
            for (int j = i + 1; j < 6; j++) {
                const int b = j % 3;
                if ((i < 3) == (j < 3)) {  // +-kc i G_3
                    her(g3, a, b, re, im);
                    if (i >= 3) { re = -re; im = -im; }
                } else {  // kc (i G_1 - i (i G_2))
                    int64_t r2, i2;
                    her(g1, a, b, re, im);
                    her(g2, a, b, r2, i2);
                    re += i2;
                    im -= r2;
                }
                u[k++] = mk(kc * fx_to_double(re, ex), kc * fx_to_double(im, ex));
            }
        }
        const int64_t base = ((int64_t)d * 36 + ch * 18) * g.Vd + s;
        store_herm6(A + base, g.Vd, dg, u);
        if (odd) {
            double d0[6];
            zd u0[15];
#pragma unroll
            for (int i = 0; i < 6; i++) d0[i] = dg[i];
#pragma unroll
            for (int i = 0; i < 15; i++) u0[i] = u[i];
            if (sweep6(dg, u)) {
#pragma unroll
                for (int i = 0; i < 6; i++) dg[i] = -dg[i];
#pragma unroll
                for (int i = 0; i < 15; i++) u[i] = -u[i];
            } else if (!invert6_packed(d0, u0, dg, u)) {
                atomicAdd(singular, 1);
                for (int i = 0; i < 6; i++) dg[i] = 0.0;
                for (int i = 0; i < 15; i++) u[i] = mk(0.0, 0.0);
            }
        }
        store_herm6(S + base, g.Vd, dg, u);
    }
}

qdd_status launch_clover_build(Gauge *g, double csw, double kappa, int *d_singular, bool fixed, cudaStream_t s)
{
    LaunchScope ls(g->ctx->timer, K_OTHER, s);
    if (fixed)
        k_clover_build_fx<<<(g->hg.V + kCloverThreads - 1) / kCloverThreads, kCloverThreads, 0, s>>>(
            g->geom, g->fx.links.as<int4>(), g->links64.as<double2>(), kappa * csw, g->clov64.as<double2>(),
            g->sclov64.as<double2>(), d_singular);
    else
        k_clover_build<<<(g->hg.V + 127) / 128, 128, 0, s>>>(g->geom, g->links64.as<double2>(), kappa * csw,
                                                            g->clov64.as<double2>(), g->sclov64.as<double2>(),
                                                            d_singular);
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

}  // namespace qdd
