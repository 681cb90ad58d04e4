// FP64 complex vector algebra of the outer flexible GMRES (arXiv:1502.04025,
// Sec. 3.1: the outer solver is flexible GMRES).  Gram-Schmidt, norms,
// basis updates and the solution update run in FP64 on the device.
//
// Vectors are flat arrays of complex FP64 (double2); the lattice layout does
// not matter here.  All reductions are two-level and deterministic: a fixed
// number of blocks (a multiple of the SM count) writes per-block partials,
// and the last block to finish (a counter in the scratch buffer) sums them in
// block order; the allocation-free entry point sums them in a separate
// launch instead.  Fused forms read each vector once: the multi-dot reads w
// once for all basis vectors, the multi-axpy writes w once and returns its
// new norm.
#include <mutex>
#include <type_traits>

#include "fixed.cuh"
#include "internal.h"

namespace qdd {

constexpr int kBT = 256;       // threads per block
constexpr int kNV = 16;        // vectors per pass of k_combine and places of a block's partials
// Vectors per launch of the multi-dot and the updates, at most: more spill
// registers (dots at 8: 372 bytes, 16 vectors of 6.3 M elements 538 us against 457;
// updates at 8 and 16: 200 and 1200).
constexpr int kPassNV = 6;
// vectors of the next launch when `left` remain: as even as whole numbers allow
static int pass_share(int left)
{
    if (left <= 0) return 0;
    const int launches = (left + kPassNV - 1) / kPassNV;
    return (left + launches - 1) / launches;
}

int blas_blocks(const Ctx *ctx, int64_t n)
{
    int64_t want = (n + kBT - 1) / kBT;
    int64_t cap = 2LL * (ctx->nsm > 0 ? ctx->nsm : 148);
    if (want > cap) want = cap;
    return (int)(want < 1 ? 1 : want);
}

// per-block partials of up to 2 blocks per SM, then one slot whose first
// word counts the blocks that have finished (zero between launches)
size_t blas_scratch_elems(const Ctx *ctx) { return (size_t)2 * (ctx->nsm > 0 ? ctx->nsm : 148) * kNV + 1; }

static unsigned *scratch_counter(const Ctx *ctx, double2 *scratch)
{
    return (unsigned *)(scratch + blas_scratch_elems(ctx) - 1);
}

qdd_status blas_scratch_ensure(Ctx *ctx, DevMem &m)
{
    const size_t bytes = blas_scratch_elems(ctx) * sizeof(double2);
    if (m.p && m.bytes >= bytes) return QDD_OK;
    QDD_TRY(m.alloc(ctx, bytes));
    QDD_CUDA(cudaMemset(scratch_counter(ctx, m.as<double2>()), 0, sizeof(unsigned)));
    QDD_CUDA(cudaDeviceSynchronize());
    return QDD_OK;
}

__device__ __forceinline__ double2 dsum2(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }

// One step of warp_transpose_sum: pairs of values (a[2i], a[2i+1]) become one
// value per lane, a[2i] on the lanes with bit O clear and a[2i+1] on the
// others, each summed with the lane across bit O; an odd last value is summed
// on both.
template <int M, int O>
__device__ __forceinline__ void warp_transpose_sum(double *a, int lane, int &idx)
{
    constexpr int H = (M + 1) / 2;
    const bool up = (lane & O) != 0;
#pragma unroll
    for (int i = 0; i < M / 2; i++) {
        const double keep = up ? a[2 * i + 1] : a[2 * i], send = up ? a[2 * i] : a[2 * i + 1];
        a[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
    }
    if (M % 2) a[H - 1] = a[M - 1] + __shfl_xor_sync(0xffffffffu, a[M - 1], O);
    if constexpr (O > 1) warp_transpose_sum<H, O / 2>(a, lane, idx);
    // idx names a value of this step's result: its place among the M before it
    idx = 2 * idx + 1 < M ? 2 * idx + (up ? 1 : 0) : M - 1;
}

// Sums of NV double2 (NV <= 16) over the block's warps: sm[w * NV + j] holds
// warp w's sum of value j after the call.  An FP64 addition takes the FP64 pipe
// 16 clocks per warp, so each lane adds a share of the values: 2 NV (1 - 1/32)
// additions per lane instead of five per value (5 vectors of 49152 elements,
// almost all of it latency: 23.7 -> 20.5 us).
template <int NV>
__device__ __forceinline__ void block_reduce(double2 *acc, double2 *sm /* [kBT/32][NV] */)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double a[2 * NV];
#pragma unroll
    for (int j = 0; j < NV; j++) {
        a[2 * j] = acc[j].x;
        a[2 * j + 1] = acc[j].y;
    }
    int idx = 0;
    warp_transpose_sum<2 * NV, 16>(a, lane, idx);
    // lanes that hold the same value hold the same bits
    reinterpret_cast<double *>(sm)[w * 2 * NV + idx] = a[0];
    __syncthreads();
}

// The last block to finish sums every block's partials (stride `stride`,
// nv values each) in block order, with the same arithmetic as
// k_reduce_final, writes out[0..nv) and resets the counter.  Called by all
// threads after the block's own partials are written.
template <int NV>
__device__ __forceinline__ void last_block_final(const double2 *part, int stride, int nv, unsigned *count,
                                                 double2 *out, double2 *sm /* [kBT/32][NV] */)
{
    __shared__ bool last;
    __threadfence();  // this block's partials before its count
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(count, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    double2 acc[NV];
#pragma unroll
    for (int j = 0; j < NV; j++) acc[j] = make_double2(0, 0);
    for (int b = threadIdx.x; b < (int)gridDim.x; b += kBT)
#pragma unroll
        for (int j = 0; j < NV; j++)
            if (j < nv) acc[j] = dsum2(acc[j], __ldcg(part + (int64_t)b * stride + j));
    block_reduce<NV>(acc, sm);
    if (threadIdx.x < nv) {
        double2 t = make_double2(0, 0);
        for (int ww = 0; ww < kBT / 32; ww++) t = dsum2(t, sm[ww * NV + threadIdx.x]);
        out[threadIdx.x] = t;
    }
    if (threadIdx.x == 0) *count = 0;
}

// Multi-dot.  In FP64 arithmetic it is bound by the FP64 pipe (4 multiply-adds
// per element and vector at 2 lanes per clock and SM: 2 clocks, against 0.72
// for the 16 bytes at the measured HBM rate), so the products run in 64-bit
// fixed point (fixed.cuh) for four elements of seven: a thread gives kDotTile
// elements of w and of each vector a common scale (their largest exponent),
// sums the products exactly with integer multiply-adds and adds one FP64 number
// per tile, vector and component to its running sum; the kDotFma elements next
// to them run on the FP64 pipe meanwhile.
//
// The error of a tile's sum belongs to the scales A of v and B of w, not to its
// products: 59 bits of each factor, truncated, give 8 products an error below
// 8 2^-58 A B, the dropped products of the lower limbs (each at most 2^29) 8 2^-60,
// and the last bit kept 2^-58: together below 2^-54.7 A B.  Eight FP64
// multiply-adds round the tile's sum by up to 8 2^-53 S, S the sum of the products'
// magnitudes.  So a tile is taken in fixed point where both components have
// S >= A B / 16, which six leading bits of every factor show (four integer
// multiply-adds for both sums of an element), and its error is then below 2^-50.7 S;
// any other tile (elements of very different sizes, a part that is nearly zero
// throughout, a non-finite element, an extreme exponent) takes FP64 arithmetic.
// Of Gaussian tiles 1 in 8000 does.
// Measured, us (event-timed), FP64 arithmetic against this: 5 vectors of 25.2 M
// elements 914 -> 513 (4712 GB/s), 3 vectors 540 -> 333 (4838 GB/s), 16 vectors of
// 6.3 M 706 -> 457, 5 vectors of 1.57 M 81 -> 53.  The magnitudes' check costs 0 to 6 %.
constexpr int kDotTile = 4, kDotFma = 3;
constexpr int kDotBits = 59;  // of both factors: 8 products per sum, |cross| <= 8 * 2 * 2^29 2^29 = 2^62
constexpr uint32_t kDotLow = 64 * 64 / 16;

__device__ __forceinline__ void fma_dot(double2 &s, double2 a, double2 x)
{
    s.x = fma(a.x, x.x, s.x);
    s.x = fma(a.y, x.y, s.x);
    s.y = fma(a.x, x.y, s.y);
    s.y = fma(-a.y, x.x, s.y);
}

// acc[j] += <v_j, w> over kDotTile elements k, k + step, ... in fixed point and
// the F after them in FP64
template <int NV, int F>
__device__ __forceinline__ void dot_tile(const double2 *__restrict__ v, int64_t ld, const double2 *__restrict__ w,
                                         int64_t k, int64_t step, double2 *acc)
{
    constexpr int K = kDotTile;
    double2 b[K + F];
    fxgroup gw = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < K + F; i++) b[i] = __ldg(w + k + i * step);
#pragma unroll
    for (int i = 0; i < K; i++) fx_group_add(gw, b[i]);
    const bool okw = fx_group_done(gw), zerow = fx_group_zero(gw);
    cfx fw[K];
    uint32_t pw[K];  // leading bits of both parts
#pragma unroll
    for (int i = 0; i < K; i++) {
        uint32_t x, y;
        fw[i] = {fx_centred<kDotBits>(b[i].x, gw.emax, x), fx_centred<kDotBits>(b[i].y, gw.emax, y)};
        pw[i] = x | y << 16;
    }
#pragma unroll
    for (int j = 0; j < NV; j++) {
        const double2 *vj = v + j * ld + k;
        double2 a[K + F];
        fxgroup gv = {0, 0, 0};
#pragma unroll
        for (int i = 0; i < K + F; i++) a[i] = __ldg(vj + i * step);
#pragma unroll
        for (int i = 0; i < K; i++) fx_group_add(gv, a[i]);
#pragma unroll
        for (int i = K; i < K + F; i++) fma_dot(acc[j], a[i], b[i]);
        const bool okv = fx_group_done(gv);
        cfx fa[K];
        uint32_t px = 0, py = 0;  // sums of |Re v| (|Re w|, |Im w|) and |Im v| (|Re w|, |Im w|)
#pragma unroll
        for (int i = 0; i < K; i++) {
            uint32_t x, y;
            fa[i] = {fx_centred<kDotBits>(a[i].x, gv.emax, x), fx_centred<kDotBits>(a[i].y, gv.emax, y)};
            px += x * pw[i];
            py += y * pw[i];
        }
        const uint32_t low = min((px & 0xffffu) + (py >> 16), (px >> 16) + (py & 0xffffu));
        if (okv && okw && (low >= kDotLow || zerow || fx_group_zero(gv))) {
            fxacc re = fx_zero(), im = fx_zero();
#pragma unroll
            for (int i = 0; i < K; i++) {
                fx_mac2(re, im, fa[i].re, fw[i].re, fw[i].im);
                fx_mac2(re, im, fa[i].im, fw[i].im, fx{-fw[i].re.hi, -fw[i].re.lo});
            }
            const int ex = gv.emax + gw.emax - 2 * 1022 + 2 * kFxLimb - 2 * kDotBits;
            acc[j].x += fx_to_double(fx_value(re), ex);
            acc[j].y += fx_to_double(fx_value(im), ex);
        } else {
#pragma unroll
            for (int i = 0; i < K; i++) fma_dot(acc[j], a[i], __ldg(w + k + i * step));
        }
    }
}

// count != NULL: the last block also writes the final sums to out
template <int NV>
__global__ void __launch_bounds__(kBT, 2) k_cdot_partial(const double2 *__restrict__ v, int64_t ld,
                                                      const double2 *__restrict__ w, int64_t n, double2 *part,
                                                      unsigned *count = nullptr, double2 *out = nullptr)
{
    __shared__ double2 sm[(kBT / 32) * NV];
    double2 acc[NV];
#pragma unroll
    for (int j = 0; j < NV; j++) acc[j] = make_double2(0, 0);
    const int64_t step = (int64_t)gridDim.x * kBT;
    int64_t k = (int64_t)blockIdx.x * kBT + threadIdx.x;
    constexpr int kT = kDotTile + kDotFma;
    for (; k + (kT - 1) * step < n; k += kT * step) dot_tile<NV, kDotFma>(v, ld, w, k, step, acc);
    for (; k < n; k += step) {  // fewer than kT elements
        const double2 b = __ldg(w + k);
#pragma unroll
        for (int j = 0; j < NV; j++) fma_dot(acc[j], __ldg(v + j * ld + k), b);
    }
    block_reduce<NV>(acc, sm);
    if (threadIdx.x < NV) {
        double2 s = make_double2(0, 0);
        for (int ww = 0; ww < kBT / 32; ww++) s = dsum2(s, sm[ww * NV + threadIdx.x]);
        part[(int64_t)blockIdx.x * kNV + threadIdx.x] = s;
    }
    if (count) {
        __syncthreads();  // sm is reused
        last_block_final<NV>(part, kNV, NV, count, out, sm);
    }
}

// out[j] = sum over blocks of part[b*stride + j], j < nvec; one block per j
__global__ void __launch_bounds__(kBT) k_reduce_final(const double2 *part, int nblk, int stride, double2 *out,
                                                      int sqrt_x)
{
    __shared__ double2 sm[kBT / 32];
    const int j = blockIdx.x;
    double2 s = make_double2(0, 0);
    for (int b = threadIdx.x; b < nblk; b += kBT) s = dsum2(s, part[(int64_t)b * stride + j]);
    double2 acc[1] = {s};
    block_reduce<1>(acc, sm);
    if (threadIdx.x == 0) {
        double2 t = make_double2(0, 0);
        for (int ww = 0; ww < kBT / 32; ww++) t = dsum2(t, sm[ww]);
        out[j] = t;
    }
}

// w = w + sign * sum_j coef[j] v_j, v in FP64 or FP32, with an optional
// per-block partial of |w|^2.  As the multi-dot, most elements run in 64-bit
// fixed point next to the FP64 pipe (4 multiply-adds per element and vector, 2
// lanes per clock and SM): of every kAxpyFx + kAxpyFma elements of a thread the
// first run in integers.  Every real product is formed from the two 53-bit
// mantissas (64 bits of it, below 2^-61 off) with its own exponent, shifted to the
// largest exponent of the products and the old value that make up its sum, real and
// imaginary parts apart, and added there; the sum keeps at least 55 bits below the
// largest of its terms' scales (2 NV + 1 terms, 62 bits less their carry) and is
// rounded once.  So the error is a fraction of the largest term, as FP64's is,
// whatever the other part or the other elements are.  Elements with a non-finite
// term or a sum near the ends of the range take FP64 arithmetic.  Measured, us, 25.2 M
// elements, FP64 arithmetic against this: 5 vectors with the norm 906 -> 596, 3
// vectors 682 -> 456, 5 FP32 vectors (16 bytes of x and 8 per vector) 1354 -> 1029.
// All vector kernels of the 32^3x64 BF16 solve at shares 1:1, 3:2, 2:1, 3:1 and all in
// integers: 6.26, 6.36, 6.46, 6.58, 7.00 ms.
constexpr int kAxpyFx = 1, kAxpyFma = 1;

// |x| = (t:r) 2^(e - 1086), t with its leading bit set (t = r = 0, e = kFxNone for
// zeros and subnormal numbers); s the sign in its leading bit
constexpr int kFxNone = -8192;
struct FxReal {
    uint32_t t, r;
    int e;
    uint32_t s;
};
__device__ __forceinline__ FxReal fx_real(double v)
{
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const int e = (int)((hi >> 20) & 0x7ffu);
    FxReal x;
    x.t = e ? __funnelshift_l(lo, hi, 11) | 0x80000000u : 0u;
    x.r = e ? lo << 11 : 0u;
    x.e = e ? e : kFxNone;
    x.s = hi;
    return x;
}

__device__ __forceinline__ double2 as_d2(double2 v) { return v; }
__device__ __forceinline__ double2 as_d2(float2 v) { return make_double2(f2d(v.x), f2d(v.y)); }

// a coefficient's parts; those of the fixed-point path are below 2^300, so that
// nothing is lost with subnormal numbers (below 2^-722 in sums above 2^-646)
struct FxCoef {
    FxReal x, y;
};
__device__ __forceinline__ bool fx_coef_ok(double v)
{
    const int e = fx_exponent(v);
    return e < 1323 && (e > 0 || v == 0);
}

// bits above a sum of n terms below 2^64 so that it stays below 2^63
template <int N>
__host__ __device__ constexpr int fx_carry()
{
    int g = 1;
    while ((1 << (g - 1)) < N) g++;
    return g;
}

// acc += +-(the 64-bit magnitude m >> sh), the sign in the leading bit of s; one
// unit short for a negative term (the sums start with that made up for, and with the
// half unit that truncation takes on average)
__device__ __forceinline__ void fx_add(int64_t &acc, uint64_t m, int sh, uint32_t s)
{
    const int64_t x = (int64_t)(m >> min(sh, 63)), sg = (int64_t)((int32_t)s >> 31);
    acc += x ^ sg;
}
// acc += +-|a||c|, at 2^(top - 2108 + G) per unit
template <int G>
__device__ __forceinline__ void fx_add_product(int64_t &acc, const FxReal &a, const FxReal &c, int top, uint32_t flip)
{
    const uint64_t m = (uint64_t)a.t * c.t + __umulhi(a.t, c.r) + __umulhi(a.r, c.t);
    fx_add(acc, m, top - (a.e + c.e) + G, a.s ^ c.s ^ flip);
}

template <int NV, int SIGN, typename T2>
__device__ __forceinline__ double2 axpy_fma(const T2 *__restrict__ v, int64_t ld, const double2 *c, double2 b)
{
#pragma unroll
    for (int j = 0; j < NV; j++) {
        const double2 a = as_d2(__ldg(v + j * ld)), cj = c[j];
        b.x = fma(SIGN * cj.x, a.x, b.x);
        b.x = fma(-SIGN * cj.y, a.y, b.x);
        b.y = fma(SIGN * cj.x, a.y, b.y);
        b.y = fma(SIGN * cj.y, a.x, b.y);
    }
    return b;
}

template <int NV, int SIGN, typename T2>
__device__ __forceinline__ double2 axpy_fx(const T2 *__restrict__ v, int64_t ld, const double2 *c, const FxCoef *fc,
                                           bool coefs, double2 b)
{
    constexpr int G = fx_carry<2 * NV + 1>();
    double2 a[NV];
    const FxReal bx = fx_real(b.x), by = fx_real(b.y);
    // exponents of the products, e_a + e_c; the old value's as a product with 1
    int tx = bx.e + 1023, ty = by.e + 1023, any = max(bx.e, by.e);
#pragma unroll
    for (int j = 0; j < NV; j++) {
        a[j] = as_d2(__ldg(v + j * ld));
        const int ex = fx_real(a[j].x).e, ey = fx_real(a[j].y).e, cx = fc[j].x.e, cy = fc[j].y.e;
        any = max(any, max(ex, ey));
        tx = max(tx, max(ex + cx, ey + cy));
        ty = max(ty, max(ey + cx, ex + cy));
    }
    // sums between 2^-646 and 2^1000, no term infinite or NaN
    if (!(coefs && any < 0x7ff && min(tx, ty) >= 1400 && max(tx, ty) <= 3040)) return axpy_fma<NV, SIGN>(v, ld, c, b);
    int64_t sx = NV, sy = NV;
    fx_add(sx, ((uint64_t)bx.t << 32) | bx.r, tx - (bx.e + 1023) + G + 1, bx.s);
    fx_add(sy, ((uint64_t)by.t << 32) | by.r, ty - (by.e + 1023) + G + 1, by.s);
    constexpr uint32_t kNeg = SIGN < 0 ? 0x80000000u : 0u;
#pragma unroll
    for (int j = 0; j < NV; j++) {
        const FxReal x = fx_real(a[j].x), y = fx_real(a[j].y), cx = fc[j].x, cy = fc[j].y;
        fx_add_product<G>(sx, x, cx, tx, kNeg);
        fx_add_product<G>(sx, y, cy, tx, kNeg ^ 0x80000000u);
        fx_add_product<G>(sy, y, cx, ty, kNeg);
        fx_add_product<G>(sy, x, cy, ty, kNeg);
    }
    return make_double2(fx_to_double(sx, tx - 2108 + G), fx_to_double(sy, ty - 2108 + G));
}

template <int NV, int SIGN, typename T2>
__global__ void __launch_bounds__(kBT, 2) k_axpy(const T2 *__restrict__ v, int64_t ld,
                                                 const double2 *__restrict__ coef, double2 *w, int64_t n,
                                                 double2 *part, unsigned *count, double2 *norm2_out)
{
    __shared__ double2 sm[kBT / 32];
    __shared__ double2 c[NV];
    __shared__ FxCoef fc[NV];
    int mine = 1;
    if (threadIdx.x < NV) {
        const double2 x = coef[threadIdx.x];
        c[threadIdx.x] = x;
        fc[threadIdx.x] = {fx_real(x.x), fx_real(x.y)};
        mine = fx_coef_ok(x.x) && fx_coef_ok(x.y);
    }
    const bool coefs = __syncthreads_and(mine);
    double nrm = 0;
    const int64_t step = (int64_t)gridDim.x * kBT;
    auto put = [&](int64_t k, double2 b) {
        w[k] = b;
        if (part) {
            nrm = fma(b.x, b.x, nrm);
            nrm = fma(b.y, b.y, nrm);
        }
    };
    int64_t k = (int64_t)blockIdx.x * kBT + threadIdx.x;
    constexpr int kT = kAxpyFx + kAxpyFma;
    for (; k + (kT - 1) * step < n; k += kT * step) {
#pragma unroll
        for (int i = 0; i < kAxpyFma; i++) {
            const int64_t q = k + (kAxpyFx + i) * step;
            put(q, axpy_fma<NV, SIGN>(v + q, ld, c, w[q]));
        }
#pragma unroll
        for (int i = 0; i < kAxpyFx; i++) {
            const int64_t q = k + i * step;
            put(q, axpy_fx<NV, SIGN>(v + q, ld, c, fc, coefs, w[q]));
        }
    }
    for (; k < n; k += step) put(k, axpy_fx<NV, SIGN>(v + k, ld, c, fc, coefs, w[k]));
    if (part) {
        double2 acc[1] = {make_double2(nrm, 0)};
        block_reduce<1>(acc, sm);
        if (threadIdx.x == 0) {
            double2 t = make_double2(0, 0);
            for (int ww = 0; ww < kBT / 32; ww++) t = dsum2(t, sm[ww]);
            part[blockIdx.x] = t;
        }
        __syncthreads();  // sm is reused
        last_block_final<1>(part, 1, 1, count, norm2_out, sm);
    }
}

// per-block partials of |w|^2
__global__ void __launch_bounds__(kBT) k_norm2(const double2 *__restrict__ w, int64_t n, double2 *part,
                                               unsigned *count, double2 *norm2_out)
{
    __shared__ double2 sm[kBT / 32];
    double nrm = 0;
    for (int64_t k = (int64_t)blockIdx.x * kBT + threadIdx.x; k < n; k += (int64_t)gridDim.x * kBT) {
        const double2 b = __ldg(w + k);
        nrm = fma(b.x, b.x, nrm);
        nrm = fma(b.y, b.y, nrm);
    }
    double2 acc[1] = {make_double2(nrm, 0)};
    block_reduce<1>(acc, sm);
    if (threadIdx.x == 0) {
        double2 t = make_double2(0, 0);
        for (int ww = 0; ww < kBT / 32; ww++) t = dsum2(t, sm[ww]);
        part[blockIdx.x] = t;
    }
    __syncthreads();  // sm is reused
    last_block_final<1>(part, 1, 1, count, norm2_out, sm);
}

// out = w / sqrt(norm2[0]) (out may alias w); out32 (optional) gets the same
// vector rounded to FP32
__global__ void k_scale_by_norm(const double2 *w, int64_t n, const double2 *norm2, double2 *out, float2 *out32)
{
    // once per block: FP64 square root and division are long sequences on
    // the FP64 pipe
    __shared__ double fs;
    if (threadIdx.x == 0) {
        double nn = norm2[0].x;
        fs = nn > 0.0 ? 1.0 / sqrt(nn) : 0.0;
    }
    __syncthreads();
    const double f = fs;
    for (int64_t k = (int64_t)blockIdx.x * kBT + threadIdx.x; k < n; k += (int64_t)gridDim.x * kBT) {
        double2 a = w[k];
        a = make_double2(a.x * f, a.y * f);
        out[k] = a;
        if (out32) out32[k] = make_float2(d2f(a.x), d2f(a.y));
    }
}

// Basis recombination of a deflated restart: out_c (+)= sum_i src_i P[i][c]
// for the NC columns c0..c0+NC-1 of P (row-major, ldp columns), src in FP64
// or FP32, out in FP64.
template <typename T2, int NC>
__global__ void __launch_bounds__(kBT) k_combine(const T2 *__restrict__ src, int nsrc, int64_t ld,
                                                 const double2 *__restrict__ P, int ldp, int c0, double2 *out,
                                                 int64_t ldo, int64_t n, int accumulate)
{
    for (int64_t k = (int64_t)blockIdx.x * kBT + threadIdx.x; k < n; k += (int64_t)gridDim.x * kBT) {
        double2 acc[NC];
#pragma unroll
        for (int c = 0; c < NC; c++) acc[c] = accumulate ? out[(int64_t)c * ldo + k] : make_double2(0, 0);
        for (int i = 0; i < nsrc; i++) {
            T2 a = src[i * ld + k];
            double ax = (double)a.x, ay = (double)a.y;
#pragma unroll
            for (int c = 0; c < NC; c++) {
                double2 p = __ldg(P + (int64_t)i * ldp + c0 + c);
                acc[c].x = fma(p.x, ax, acc[c].x);
                acc[c].x = fma(-p.y, ay, acc[c].x);
                acc[c].y = fma(p.x, ay, acc[c].y);
                acc[c].y = fma(p.y, ax, acc[c].y);
            }
        }
#pragma unroll
        for (int c = 0; c < NC; c++) out[(int64_t)c * ldo + k] = acc[c];
    }
}

// ------------------------------------------------------------- launchers

// Call f with std::integral_constant<int, NV> for NV = nv (1..kNV): kernels
// are instantiated for exactly the number of vectors they handle, because
// predicated-off iterations of a wider unrolled loop would still occupy the
// FP64 pipe, the bottleneck of these kernels on this GPU.
template <typename F>
static void nv_dispatch(int nv, F &&f)
{
    switch (nv) {
    case 1: f(std::integral_constant<int, 1>{}); break;
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 3: f(std::integral_constant<int, 3>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    case 5: f(std::integral_constant<int, 5>{}); break;
    case 6: f(std::integral_constant<int, 6>{}); break;
    case 7: f(std::integral_constant<int, 7>{}); break;
    case 8: f(std::integral_constant<int, 8>{}); break;
    case 9: f(std::integral_constant<int, 9>{}); break;
    case 10: f(std::integral_constant<int, 10>{}); break;
    case 11: f(std::integral_constant<int, 11>{}); break;
    case 12: f(std::integral_constant<int, 12>{}); break;
    case 13: f(std::integral_constant<int, 13>{}); break;
    case 14: f(std::integral_constant<int, 14>{}); break;
    case 15: f(std::integral_constant<int, 15>{}); break;
    default: f(std::integral_constant<int, 16>{}); break;
    }
}

// the same for the multi-dot and the updates, nv = 1..kPassNV
template <typename F>
static void pass_dispatch(int nv, F &&f)
{
    switch (nv) {
    case 1: f(std::integral_constant<int, 1>{}); break;
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 3: f(std::integral_constant<int, 3>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    case 5: f(std::integral_constant<int, 5>{}); break;
    default: f(std::integral_constant<int, 6>{}); break;
    }
}

qdd_status blas_cdot_multi(Ctx *ctx, const double2 *v, int nvec, int64_t ld, const double2 *w, int64_t n,
                           double2 *out, double2 *scratch, cudaStream_t s)
{
    if (nvec <= 0) return QDD_OK;
    const int nb = blas_blocks(ctx, n);
    for (int j0 = 0, nv; j0 < nvec; j0 += nv) {
        nv = pass_share(nvec - j0);
        ctx->timer.work(K_BLAS, 8.0 * nv * n, 16.0 * (nv + 1) * n);
        LaunchScope ls(ctx->timer, K_BLAS, s);
        pass_dispatch(nv, [&](auto c) {
            k_cdot_partial<decltype(c)::value><<<nb, kBT, 0, s>>>(v + j0 * ld, ld, w, n, scratch,
                                                                  scratch_counter(ctx, scratch), out + j0);
        });
    }
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

qdd_status blas_caxpy_multi_norm(Ctx *ctx, const double2 *v, int nvec, int64_t ld, const double2 *coef, double2 *w,
                                 int64_t n, double2 *norm2_out, double2 *scratch, cudaStream_t s)
{
    const int nb = blas_blocks(ctx, n);
    int j0 = 0;
    do {
        const int nv = pass_share(nvec - j0);
        bool last = j0 + nv >= nvec;
        // v read, w read and (when updated) written; |w|^2 on the last pass
        ctx->timer.work(K_BLAS, 8.0 * nv * n + ((last && norm2_out) ? 4.0 * n : 0.0),
                        16.0 * (nv + 1 + (nv > 0 ? 1 : 0)) * n);
        {
            LaunchScope ls(ctx->timer, K_BLAS, s);
            double2 *part = (last && norm2_out) ? scratch : nullptr;
            unsigned *cnt = scratch_counter(ctx, scratch);
            if (nv == 0)
                k_norm2<<<nb, kBT, 0, s>>>(w, n, scratch, cnt, norm2_out);
            else
                pass_dispatch(nv, [&](auto c) {
                    k_axpy<decltype(c)::value, -1, double2><<<nb, kBT, 0, s>>>(v + j0 * ld, ld, coef + j0, w, n, part,
                                                                               cnt, norm2_out);
                });
        }
        j0 += nv;
    } while (j0 < nvec);
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

qdd_status blas_norm2(Ctx *ctx, const double2 *w, int64_t n, double2 *out, double2 *scratch, cudaStream_t s)
{
    return blas_caxpy_multi_norm(ctx, nullptr, 0, 0, nullptr, (double2 *)w, n, out, scratch, s);
}

qdd_status blas_scale_by_norm(Ctx *ctx, const double2 *w, int64_t n, const double2 *norm2, double2 *out,
                              cudaStream_t s, float2 *out32)
{
    // one element per thread: a memory-bound pass needs every load in flight
    // at once (the reduction kernels' two blocks per SM keep too few)
    const int64_t nb = (n + kBT - 1) / kBT;
    ctx->timer.work(K_BLAS, 2.0 * n, (32.0 + (out32 ? 8.0 : 0.0)) * n);
    LaunchScope ls(ctx->timer, K_BLAS, s);
    k_scale_by_norm<<<(unsigned)(nb < (1LL << 30) ? nb : (1LL << 30)), kBT, 0, s>>>(w, n, norm2, out, out32);
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

qdd_status blas_combine(Ctx *ctx, const void *src, bool src_f32, int nsrc, int64_t ld, const double2 *P, int ldp,
                        int ncols, double2 *out, int64_t ldo, int64_t n, int accumulate, cudaStream_t s)
{
    if (nsrc <= 0 || ncols <= 0) return QDD_OK;
    const int nb = blas_blocks(ctx, n);
    for (int c0 = 0; c0 < ncols; c0 += kNV) {
        int nc = ncols - c0 < kNV ? ncols - c0 : kNV;
        ctx->timer.work(K_BLAS, 8.0 * nsrc * nc * n,
                        ((src_f32 ? 8.0 : 16.0) * nsrc + 16.0 * nc * (accumulate ? 2 : 1)) * n);
        LaunchScope ls(ctx->timer, K_BLAS, s);
        nv_dispatch(nc, [&](auto c) {
            if (src_f32)
                k_combine<float2, decltype(c)::value><<<nb, kBT, 0, s>>>((const float2 *)src, nsrc, ld, P, ldp, c0,
                                                                         out + (int64_t)c0 * ldo, ldo, n, accumulate);
            else
                k_combine<double2, decltype(c)::value><<<nb, kBT, 0, s>>>((const double2 *)src, nsrc, ld, P, ldp, c0,
                                                                          out + (int64_t)c0 * ldo, ldo, n,
                                                                          accumulate);
        });
    }
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

qdd_status blas_axpy_multi(Ctx *ctx, const void *z, bool z_f32, int nvec, int64_t ld, const double2 *coef,
                           double2 *x, int64_t n, cudaStream_t s)
{
    if (nvec <= 0) return QDD_OK;
    for (int j0 = 0, nv; j0 < nvec; j0 += nv) {
        nv = pass_share(nvec - j0);
        ctx->timer.work(K_BLAS, 8.0 * nv * n, ((z_f32 ? 8.0 : 16.0) * nv + 32.0) * n);
        LaunchScope ls(ctx->timer, K_BLAS, s);
        pass_dispatch(nv, [&](auto c) {
            if (z_f32)
                k_axpy<decltype(c)::value, 1, float2><<<blas_blocks(ctx, n), kBT, 0, s>>>(
                    (const float2 *)z + j0 * ld, ld, coef + j0, x, n, nullptr, nullptr, nullptr);
            else
                k_axpy<decltype(c)::value, 1, double2><<<blas_blocks(ctx, n), kBT, 0, s>>>(
                    (const double2 *)z + j0 * ld, ld, coef + j0, x, n, nullptr, nullptr, nullptr);
        });
    }
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free multi-dot (qdd_cdot_multi_noalloc).
//
// The per-block partial sums live in a fixed device array that is part of the
// library image instead of in memory from cudaMalloc.  Host code may not use
// the array's name as a device pointer: it only stands in for the symbol, so
// the device address is looked up once per device with cudaGetSymbolAddress
// and passed to the kernels.  The array holds kNoAllocBlocks * kNV partials
// (128 KiB) on every GPU that loads the library, until the process exits.

constexpr int kNoAllocBlocks = 512;
static __device__ __align__(256) double2 g_noalloc_partials[kNoAllocBlocks * kNV];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
double2 *g_noalloc_ptr[kMaxDevices] = {};
int g_noalloc_nsm[kMaxDevices] = {};

// Device address of the partials array on the current device, resolved on
// the first call for that device.
qdd_status noalloc_setup(int dev, double2 **ptr, int *nsm)
{
    if (dev < 0 || dev >= kMaxDevices) {
        set_error("device %d out of range for the allocation-free entry points", dev);
        return QDD_EINVAL;
    }
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_partials);
        if (e != cudaSuccess || !p) {
            set_error("cudaGetSymbolAddress of the partial-sum array failed on device %d: %s", dev,
                      cudaGetErrorString(e));
            return QDD_ECUDA;
        }
        int sm = 0;
        e = cudaDeviceGetAttribute(&sm, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) {
            set_error("cudaDeviceGetAttribute failed on device %d: %s", dev, cudaGetErrorString(e));
            return QDD_ECUDA;
        }
        g_noalloc_nsm[dev] = sm;
        g_noalloc_ptr[dev] = (double2 *)p;
    }
    *ptr = g_noalloc_ptr[dev];
    *nsm = g_noalloc_nsm[dev];
    return QDD_OK;
}
}  // namespace

}  // namespace qdd

extern "C" qdd_status qdd_cdot_multi_noalloc(const double *v, int nvec, int64_t ld, const double *w, int64_t n,
                                             double *out, void *stream)
{
    using namespace qdd;
    clear_error();
    if (!v || !w || !out) {
        set_error("null pointer argument");
        return QDD_EINVAL;
    }
    if (nvec < 1 || nvec > 64) {
        set_error("nvec = %d outside 1..64", nvec);
        return QDD_EINVAL;
    }
    if (n < 1 || n > (int64_t(1) << 40) || ld < n) {
        set_error("vector length n = %lld (stride %lld) outside 1..2^40 or stride below n", (long long)n,
                  (long long)ld);
        return QDD_EINVAL;
    }
    int dev = 0;
    QDD_CUDA(cudaGetDevice(&dev));
    double2 *part = nullptr;
    int nsm = 0;
    QDD_TRY(noalloc_setup(dev, &part, &nsm));
    cudaStream_t s = (cudaStream_t)stream;
    int64_t nb64 = (n + kBT - 1) / kBT;
    int64_t cap = 2LL * nsm;
    if (cap > kNoAllocBlocks) cap = kNoAllocBlocks;
    if (nb64 > cap) nb64 = cap;
    const int nb = (int)(nb64 < 1 ? 1 : nb64);
    const double2 *V2 = (const double2 *)v, *W2 = (const double2 *)w;
    double2 *O2 = (double2 *)out;
    // every block overwrites its own partials before the final sum reads them,
    // so nothing in the shared array has to start at zero
    for (int j0 = 0, nv; j0 < nvec; j0 += nv) {
        nv = pass_share(nvec - j0);
        pass_dispatch(nv, [&](auto c) {
            k_cdot_partial<decltype(c)::value><<<nb, kBT, 0, s>>>(V2 + j0 * ld, ld, W2, n, part);
        });
        k_reduce_final<<<nv, kBT, 0, s>>>(part, nb, kNV, O2 + j0, 0);
    }
    // no synchronisation: out is ready in the order of `stream`
    QDD_CUDA(cudaGetLastError());
    return QDD_OK;
}
