// C ABI of libqdd: contexts, gauge fields, operator and preconditioner
// entry points, and host-side helpers (arXiv:1502.04025, Sec. 3).
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>

#include "internal.h"

namespace qdd {

// ------------------------------------------------------------------ errors

static thread_local char g_err[1024] = "";

void set_error(const char *fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
}

void clear_error() { g_err[0] = 0; }

// ------------------------------------------------------------------ timing

cudaEvent_t Timer::get_event()
{
    if (!pool.empty()) {
        cudaEvent_t e = pool.back();
        pool.pop_back();
        return e;
    }
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    return e;
}

void Timer::begin(int cls, cudaStream_t s, cudaEvent_t *a)
{
    std::lock_guard<std::mutex> lk(mu);
    launches[cls]++;
    if (mask & (1 << cls)) {
        *a = get_event();
        cudaEventRecord(*a, s);
    }
}

void Timer::begin_seq(int cls, cudaStream_t s, cudaEvent_t *a)
{
    std::lock_guard<std::mutex> lk(mu);
    if (mask & (1 << cls)) {
        *a = get_event();
        cudaEventRecord(*a, s);
    }
}

void Timer::count(int cls)
{
    std::lock_guard<std::mutex> lk(mu);
    launches[cls]++;
}

void Timer::work(int cls, double f, double b)
{
    std::lock_guard<std::mutex> lk(mu);
    flop[cls] += f;
    bytes[cls] += b;
}

void Timer::end(int cls, cudaStream_t s, cudaEvent_t a)
{
    if (!a) return;
    std::lock_guard<std::mutex> lk(mu);
    cudaEvent_t b = get_event();
    cudaEventRecord(b, s);
    pending.push_back({a, b, cls});
}

void Timer::resolve()
{
    std::lock_guard<std::mutex> lk(mu);
    std::vector<Pending> keep;
    for (auto &p : pending) {
        if (cudaEventQuery(p.b) != cudaSuccess) {
            keep.push_back(p);
            continue;
        }
        float t = 0;
        if (cudaEventElapsedTime(&t, p.a, p.b) == cudaSuccess) {
            ms[p.cls] += t;
            timed[p.cls]++;
        }
        pool.push_back(p.a);
        pool.push_back(p.b);
    }
    pending.swap(keep);
    cudaGetLastError();
}

Timer::~Timer()
{
    for (auto &p : pending) {
        cudaEventDestroy(p.a);
        cudaEventDestroy(p.b);
    }
    for (auto e : pool) cudaEventDestroy(e);
}

// ------------------------------------------------------------------ memory

// the gauge field whose fixed-point copy this thread is building (its lock is held)
static thread_local const Gauge *fx_building = nullptr;
// this thread asks for memory that it can do without: it takes no copies back for it
static thread_local bool fx_optional = false;

static void fx_release(Gauge *g)
{
    FxCopy &f = g->fx;
    if (!f.required) g->ctx->optional -= f.links.bytes + f.clov.bytes + f.clov_e.bytes;
    f.links.release();
    f.clov.release();
    f.clov_e.release();
    f.have_links = f.have_clov = f.required = f.wide = false;
}

// Gives up optional fixed-point copies, until at least `need` bytes have come
// back.  Another thread holds a copy while it launches the operator or builds the
// copy, so one that is held is tried again for up to a second (two threads that build
// copies may each want the other's).  This thread holds none but the one it builds:
// whoever acquires a copy has made its own allocations before.
static void fx_reclaim(Ctx *c, size_t need)
{
    size_t got = 0;
    for (int turn = 0; turn < 10000 && c->optional.load() != 0; turn++) {
        bool held = false;
        {
            std::lock_guard<std::mutex> lk(c->gauges_mu);
            for (Gauge *g : c->gauges) {
                if (got >= need) return;
                if (g == fx_building) continue;
                std::unique_lock<std::shared_mutex> ul(g->fx.mu, std::try_to_lock);
                if (!ul.owns_lock()) {
                    held = true;
                    continue;
                }
                if (g->fx.required) continue;
                got += g->fx.links.bytes + g->fx.clov.bytes + g->fx.clov_e.bytes;
                fx_release(g);
            }
        }
        if (!held || got >= need) return;
        std::this_thread::sleep_for(std::chrono::microseconds(100));
    }
}

// n bytes of the budget, if they are there (threads allocate side by side)
static bool reserve(Ctx *c, size_t n)
{
    size_t u = c->used.load();
    do {
        if (u + n > c->budget) return false;
    } while (!c->used.compare_exchange_weak(u, u + n));
    return true;
}

qdd_status DevMem::alloc(Ctx *c, size_t n)
{
    release();
    if (n == 0) return QDD_OK;
    // (another thread may build a copy anew between the two, so more than once)
    bool room = reserve(c, n);
    for (int turn = 0; !room && !fx_optional && turn < 8; turn++) {
        const size_t u = c->used.load();
        if (c->optional.load() == 0) break;
        if (u + n > c->budget) fx_reclaim(c, u + n - c->budget);
        room = reserve(c, n);
    }
    if (!room) {
        set_error("allocation of %zu bytes exceeds the HBM budget (%zu of %zu bytes in use)", n, c->used.load(),
                  c->budget);
        return QDD_EBUDGET;
    }
    cudaError_t e = cudaMalloc(&p, n);
    if (e == cudaErrorMemoryAllocation && !fx_optional && c->optional.load() != 0) {
        // the device is full below the budget (another library, another process)
        cudaGetLastError();
        fx_reclaim(c, n);
        e = cudaMalloc(&p, n);
    }
    if (e != cudaSuccess) {
        p = nullptr;
        c->used -= n;
        cudaGetLastError();
        set_error("cudaMalloc(%zu) failed: %s", n, cudaGetErrorString(e));
        return QDD_ENOMEM;
    }
    ctx = c;
    bytes = n;
    return QDD_OK;
}

qdd_status optional_room(DevMem &m, Ctx *c, size_t n)
{
    fx_optional = true;
    const qdd_status st = m.ensure(c, n);
    fx_optional = false;
    if (st != QDD_EBUDGET && st != QDD_ENOMEM) return st;
    clear_error();
    return QDD_EBUDGET;
}

void DevMem::release()
{
    if (p) {
        cudaFree(p);
        if (ctx) {
            ctx->used -= bytes;
            ctx->frees++;
        }
    }
    p = nullptr;
    bytes = 0;
}

// -------------------------------------------------------- precision copies

// Links have a fixed-point copy from 2^-60 to 2^64, and where their sizes differ
// by no more than 2^4: the field has one scale, 60 bits below its largest entry, so
// a link 2^4 smaller keeps the 53 bits of an FP64 number below its own largest.
// SU(3) links (largest entries between 0.57 and 1) and unitary ones always do.
constexpr int kMinFixedLinkExp = -60, kMaxFixedLinkExp = 64, kMaxFixedLinkSpread = 4;
// A clover term has one where every site's largest entry lies within 2^+-60 (an
// ordinary one's is near 1).  With spinors within 2^+-900 the scales of all
// products then stay inside FP64's normal range, -1016 to 965 and 62 bits more.
constexpr int kMaxFixedCloverExp = 60;
// The operator's fixed-point sums are as good as FP64's where the hops, times kappa, are
// not far below the clover sum (fixed.cuh): with kappa at 0.04 the test leaves two
// Gaussian sites of 65536 to FP64, below that soon many.
constexpr double kMinFixedKappa = 0.04;

static size_t elem_bytes(qdd_prec p)
{
    switch (p) {
    case QDD_PREC_F64: return 16;
    case QDD_PREC_DF64: return 16;
    case QDD_PREC_F32: return 8;
    default: return 4;
    }
}

qdd_status ensure_copy(Gauge *g, qdd_prec prec, cudaStream_t s)
{
    if (prec == QDD_PREC_F64) return QDD_OK;
    if (prec == QDD_PREC_H16) return ensure_copy(g, QDD_PREC_F16S, s);
    if (prec == QDD_PREC_DF64) {
        FxLock lk;
        return fx_acquire(g, true, true, s, lk);
    }
    if (prec < QDD_PREC_F64 || prec > QDD_PREC_DF64) {
        set_error("invalid precision %d", (int)prec);
        return QDD_EINVAL;
    }
    std::lock_guard<std::mutex> lk(g->copy_mu);
    PrecCopy &c = g->copies[prec];
    if (c.valid) return QDD_OK;
    if (!g->have_clover) {
        set_error("set_clover has not been called");
        return QDD_EINVAL;
    }
    const size_t V = g->hg.V, eb = elem_bytes(prec);
    const bool scaled = prec == QDD_PREC_F16S || prec == QDD_PREC_BF16S;
    QDD_TRY(c.links.ensure(g->ctx, V * 36 * eb));
    QDD_TRY(c.clov.ensure(g->ctx, V * 36 * eb));
    QDD_TRY(c.sclov.ensure(g->ctx, V * 36 * eb));
    if (scaled) {
        QDD_TRY(c.clov_s.ensure(g->ctx, V * 4));
        QDD_TRY(c.sclov_s.ensure(g->ctx, V * 4));
    }
    QDD_TRY(launch_links_convert(g, prec, c.links.p, s));
    QDD_TRY(launch_clover_convert(g, g->clov64.as<double2>(), prec, c.clov.p, c.clov_s.as<float>(), s, true));
    QDD_TRY(launch_clover_convert(g, g->sclov64.as<double2>(), prec, c.sclov.p, c.sclov_s.as<float>(), s));
    c.valid = true;
    return QDD_OK;
}

static qdd_status fx_build(Gauge *g, bool required, bool clover, cudaStream_t s)
{
    FxCopy &f = g->fx;
    Ctx *c = g->ctx;
    const size_t n = (size_t)g->hg.V * 36 * 16, ne = ((size_t)g->hg.V + 1) * sizeof(int);
    if (!required && !f.required) {
        const size_t more = (f.links.p ? 0 : n) + (clover && !f.clov.p ? n + ne : 0);
        if (c->used.load() + more > c->budget / 2 || f.no_room == c->frees.load()) return QDD_EBUDGET;
    }
    const size_t before = f.links.bytes + f.clov.bytes + f.clov_e.bytes;
    fx_optional = !required;
    qdd_status st = f.links.ensure(c, n);
    if (st == QDD_OK && clover) st = f.clov.ensure(c, n);
    if (st == QDD_OK && clover) st = f.clov_e.ensure(c, ne);
    fx_optional = false;
    f.no_room = st == QDD_ENOMEM ? c->frees.load() : ~0ull;
    if (!f.required) c->optional += f.links.bytes + f.clov.bytes + f.clov_e.bytes - before;
    QDD_TRY(st);
    if (!f.have_links) QDD_TRY(launch_links_fx(g, s));
    if (clover && !f.have_clov) QDD_TRY(launch_clover_fx(g, s));
    int far = 0;
    if (clover && !f.have_clov)
        QDD_CUDA(cudaMemcpyAsync(&far, f.clov_e.as<int>() + g->hg.V, sizeof(int), cudaMemcpyDeviceToHost, s));
    QDD_CUDA(cudaStreamSynchronize(s));  // other streams may read it from here on
    f.have_links = true;
    if (clover && !f.have_clov) {
        f.have_clov = true;
        f.wide = far > kMaxFixedCloverExp;
        if (f.wide) {  // FP64 arithmetic, until the next clover term: the room is not needed
            if (!f.required) c->optional -= f.clov.bytes + f.clov_e.bytes;
            f.clov.release();
            f.clov_e.release();
        }
    }
    if (f.wide) return QDD_OK;
    if (required && !f.required) {
        f.required = true;
        c->optional -= f.links.bytes + f.clov.bytes + f.clov_e.bytes;
    }
    return QDD_OK;
}

qdd_status fx_acquire(Gauge *g, bool required, bool clover, cudaStream_t s, FxLock &lk)
{
    if (clover && !g->have_clover) {
        set_error("set_clover has not been called");
        return QDD_EINVAL;
    }
    if (g->link_exp < kMinFixedLinkExp || g->link_exp > kMaxFixedLinkExp || g->link_spread > kMaxFixedLinkSpread ||
        (clover && !(std::fabs(g->kappa) >= kMinFixedKappa)))
        return QDD_OK;
    FxCopy &f = g->fx;
    for (int turn = 0; turn < 3; turn++) {  // an optional copy may be given up between the two locks
        lk = FxLock(f.mu);
        if (clover && f.have_clov && f.wide) {
            lk.unlock();
            return QDD_OK;
        }
        if (f.have_links && (!clover || f.have_clov) && (!required || f.required)) return QDD_OK;
        lk.unlock();
        std::unique_lock<std::shared_mutex> ul(f.mu);
        fx_building = g;
        qdd_status st = fx_build(g, required, clover, s);
        fx_building = nullptr;
        if (st != QDD_OK && !required && (st == QDD_EBUDGET || st == QDD_ENOMEM)) {
            clear_error();
            return QDD_OK;
        }
        QDD_TRY(st);
    }
    return QDD_OK;
}

qdd_status ensure_links12(Gauge *g, qdd_prec prec, cudaStream_t s)
{
    prec = field_store(prec);
    if (prec != QDD_PREC_F32 && prec != QDD_PREC_F16S && prec != QDD_PREC_BF16S) {
        set_error("two-row links exist for FP32, FP16 and BF16 storage only");
        return QDD_EINVAL;
    }
    std::lock_guard<std::mutex> lk(g->copy_mu);
    PrecCopy &c = g->copies[prec];
    if (c.valid12) return QDD_OK;
    QDD_TRY(c.links12.ensure(g->ctx, (size_t)g->hg.V * 24 * elem_bytes(prec)));
    QDD_TRY(launch_links12_convert(g, prec, c.links12.p, s));
    c.valid12 = true;
    return QDD_OK;
}

// per-gauge staging buffers for the entry points that are not the solver
struct Staging {
    DevMem io, a, a_s, b, b_s, c, c_s, err;
    int *host_err = nullptr;  // page-locked copy of err, read after the call's last synchronisation
    ~Staging()
    {
        if (host_err) cudaFreeHost(host_err);
    }
};

Gauge::~Gauge()
{
    if (!registered) return;
    {
        std::lock_guard<std::mutex> lk(ctx->gauges_mu);
        for (size_t k = 0; k < ctx->gauges.size(); k++)
            if (ctx->gauges[k] == this) {
                ctx->gauges.erase(ctx->gauges.begin() + k);
                break;
            }
    }
    fx_release(this);
}

static qdd_status stage_in(Gauge *g, DevMem &io, const double *src, int nrhs, int on_device, cudaStream_t s,
                           const double **dev)
{
    size_t bytes = (size_t)g->hg.V * 24 * sizeof(double) * nrhs;
    if (on_device) {
        *dev = src;
        return QDD_OK;
    }
    QDD_TRY(io.ensure(g->ctx, bytes));
    QDD_CUDA(cudaMemcpyAsync(io.p, src, bytes, cudaMemcpyHostToDevice, s));
    *dev = io.as<double>();
    return QDD_OK;
}

static qdd_status stage_out(Gauge *g, DevMem &io, double *dst, int nrhs, int on_device, cudaStream_t s,
                            double **dev)
{
    size_t bytes = (size_t)g->hg.V * 24 * sizeof(double) * nrhs;
    if (on_device) {
        *dev = dst;
        return QDD_OK;
    }
    QDD_TRY(io.ensure(g->ctx, bytes));
    *dev = io.as<double>();
    return QDD_OK;
}

static qdd_status finish_out(Gauge *g, DevMem &io, double *dst, int nrhs, int on_device, cudaStream_t s)
{
    size_t bytes = (size_t)g->hg.V * 24 * sizeof(double) * nrhs;
    if (!on_device) QDD_CUDA(cudaMemcpyAsync(dst, io.p, bytes, cudaMemcpyDeviceToHost, s));
    QDD_CUDA(cudaStreamSynchronize(s));
    g->ctx->timer.resolve();
    return QDD_OK;
}

}  // namespace qdd

using namespace qdd;

// ======================================================================= C ABI

extern "C" {

const char *qdd_last_error(void) { return g_err; }

qdd_status qdd_create(qdd_ctx **out, int device, size_t hbm_budget_bytes)
{
    clear_error();
    if (!out) {
        set_error("ctx is NULL");
        return QDD_EINVAL;
    }
    *out = nullptr;
    int ndev = 0;
    QDD_CUDA(cudaGetDeviceCount(&ndev));
    if (device < 0 || device >= ndev) {
        set_error("device %d out of range (%d devices)", device, ndev);
        return QDD_EINVAL;
    }
    QDD_CUDA(cudaSetDevice(device));
    size_t free_b = 0, total_b = 0;
    QDD_CUDA(cudaMemGetInfo(&free_b, &total_b));
    qdd_ctx *c = new qdd_ctx();
    c->device = device;
    QDD_CUDA(cudaDeviceGetAttribute(&c->nsm, cudaDevAttrMultiProcessorCount, device));
    c->budget = hbm_budget_bytes ? hbm_budget_bytes : (size_t)(0.8 * (double)total_b);
    *out = c;
    return QDD_OK;
}

qdd_status qdd_set_profiling(qdd_ctx *ctx, int classes)
{
    if (!ctx) return QDD_EINVAL;
    QDD_CUDA(cudaSetDevice(ctx->device));
    std::lock_guard<std::mutex> lk(ctx->timer.mu);
    ctx->timer.mask = classes & QDD_PROF_ALL;
    // create the events up front so that timed regions create none
    while (classes && ctx->timer.pool.size() < 4096) {
        cudaEvent_t e = nullptr;
        QDD_CUDA(cudaEventCreate(&e));
        ctx->timer.pool.push_back(e);
    }
    return QDD_OK;
}

qdd_status qdd_get_kernel_times(qdd_ctx *ctx, double out[6], int reset)
{
    if (!ctx || !out) return QDD_EINVAL;
    cudaSetDevice(ctx->device);
    ctx->timer.resolve();
    std::lock_guard<std::mutex> lk(ctx->timer.mu);
    for (int c = 0; c < 3; c++) {
        out[2 * c] = ctx->timer.ms[c];
        out[2 * c + 1] = (double)ctx->timer.launches[c];
    }
    if (reset)
        for (int c = 0; c < 4; c++) {
            ctx->timer.ms[c] = 0;
            ctx->timer.launches[c] = 0;
            ctx->timer.timed[c] = 0;
            ctx->timer.flop[c] = 0;
            ctx->timer.bytes[c] = 0;
        }
    return QDD_OK;
}

qdd_status qdd_get_kernel_work(qdd_ctx *ctx, double out[6])
{
    if (!ctx || !out) return QDD_EINVAL;
    std::lock_guard<std::mutex> lk(ctx->timer.mu);
    for (int c = 0; c < 3; c++) {
        out[2 * c] = ctx->timer.flop[c];
        out[2 * c + 1] = ctx->timer.bytes[c];
    }
    return QDD_OK;
}

qdd_status qdd_memory(qdd_ctx *ctx, size_t *used, size_t *budget)
{
    if (!ctx) return QDD_EINVAL;
    if (used) *used = ctx->used.load();
    if (budget) *budget = ctx->budget;
    return QDD_OK;
}

qdd_status qdd_create_gauge_field(qdd_ctx *ctx, const int L[4], const int dom[4], const double *links,
                                  int links_on_device, qdd_gauge **out)
{
    clear_error();
    if (!ctx || !L || !dom || !links || !out) {
        set_error("null argument");
        return QDD_EINVAL;
    }
    *out = nullptr;
    QDD_CUDA(cudaSetDevice(ctx->device));
    std::unique_ptr<qdd_gauge> g(new qdd_gauge());
    g->ctx = ctx;
    QDD_TRY(make_geometry(L, dom, g->hg));
    const HostGeom &hg = g->hg;
    QDD_TRY(g->d_nbl.alloc(ctx, hg.nbl.size() * sizeof(uint16_t)));
    QDD_TRY(g->d_nbd.alloc(ctx, hg.nbd.size() * sizeof(int)));
    QDD_TRY(g->d_site_of.alloc(ctx, hg.site_of.size() * sizeof(int)));
    QDD_TRY(g->d_block_slot.alloc(ctx, hg.block_slot.size() * sizeof(int)));
    QDD_TRY(g->d_fcoord.alloc(ctx, hg.fcoord.size() * sizeof(uint32_t)));
    QDD_CUDA(cudaMemcpy(g->d_fcoord.p, hg.fcoord.data(), hg.fcoord.size() * sizeof(uint32_t),
                        cudaMemcpyHostToDevice));
    QDD_CUDA(cudaMemcpy(g->d_block_slot.p, hg.block_slot.data(), hg.block_slot.size() * sizeof(int),
                        cudaMemcpyHostToDevice));
    QDD_CUDA(cudaMemcpy(g->d_nbl.p, hg.nbl.data(), hg.nbl.size() * sizeof(uint16_t), cudaMemcpyHostToDevice));
    QDD_CUDA(cudaMemcpy(g->d_nbd.p, hg.nbd.data(), hg.nbd.size() * sizeof(int), cudaMemcpyHostToDevice));
    QDD_CUDA(cudaMemcpy(g->d_site_of.p, hg.site_of.data(), hg.site_of.size() * sizeof(int),
                        cudaMemcpyHostToDevice));
    Geom &G = g->geom;
    for (int mu = 0; mu < 4; mu++) {
        G.L[mu] = hg.L[mu];
        G.dom[mu] = hg.dom[mu];
        G.nb[mu] = hg.nb[mu];
    }
    G.V = hg.V;
    G.Vd = hg.Vd;
    G.Vh = hg.Vh;
    G.Nd = hg.Nd;
    G.Nd2 = hg.Nd2;
    G.vd_shift = -1;
    for (int k = 0; k < 31; k++)
        if ((1 << k) == hg.Vd) G.vd_shift = k;
    G.nbl = g->d_nbl.as<uint16_t>();
    G.nbd = g->d_nbd.as<int>();
    G.block_slot = g->d_block_slot.as<int>();
    G.fcoord = g->d_fcoord.as<uint32_t>();
    for (int k = 0; k < 8; k++) G.foff[k] = hg.foff[k];
    G.nf = hg.nf;

    const size_t lbytes = (size_t)hg.V * 36 * sizeof(double2);
    QDD_TRY(g->links64.alloc(ctx, lbytes));
    const double *src = links;
    DevMem tmp;
    if (!links_on_device) {
        QDD_TRY(tmp.alloc(ctx, lbytes));
        QDD_CUDA(cudaMemcpy(tmp.p, links, lbytes, cudaMemcpyHostToDevice));
        src = tmp.as<double>();
    }
    QDD_TRY(launch_links_to_internal(g.get(), src, 0));
    // SU(3) links (to rounding) let the full-lattice operator read two rows per link
    DevMem bad;
    QDD_TRY(bad.alloc(ctx, 3 * sizeof(int)));
    QDD_TRY(launch_su3_check(g.get(), kSu3Tol, bad.as<int>(), 0));
    int h_bad[3] = {1, 0, 0};
    QDD_CUDA(cudaMemcpy(h_bad, bad.p, sizeof(h_bad), cudaMemcpyDeviceToHost));
    g->su3 = h_bad[0] == 0;
    g->link_exp = h_bad[1] == 0x7ff ? 1 << 20 : std::max(h_bad[1] - 1022, -800);
    g->link_spread = std::max(h_bad[1] - (0x7ff - h_bad[2]), 0);
    if (g->su3) g->link_exp = g->link_spread = 0;
    g->two_rows = g->su3;
    QDD_CUDA(cudaDeviceSynchronize());
    ctx->timer.resolve();
    {
        std::lock_guard<std::mutex> lk(ctx->gauges_mu);
        ctx->gauges.push_back(g.get());
        g->registered = true;
    }
    *out = g.release();
    return QDD_OK;
}

qdd_status qdd_create_gauge_field_slab(qdd_ctx *ctx, const int Lloc[4], const int dom[4], const double *links_ext,
                                       int links_on_device, const qdd_comm *comm, qdd_gauge **out)
{
    clear_error();
    if (!ctx || !Lloc || !dom || !links_ext || !comm || !out) {
        set_error("null argument");
        return QDD_EINVAL;
    }
    *out = nullptr;
    if (comm->size < 1 || comm->rank < 0 || comm->rank >= comm->size || !comm->allreduce_sum || !comm->shift) {
        set_error("invalid communication hooks (rank %d of %d)", comm->rank, comm->size);
        return QDD_EINVAL;
    }
    if (dom[3] < 2) {
        set_error("invalid domain extent in t");
        return QDD_EINVAL;
    }
    const int Le[4] = {Lloc[0], Lloc[1], Lloc[2], Lloc[3] + 2 * dom[3]};
    const size_t Ls = (size_t)Lloc[0] * Lloc[1] * Lloc[2];
    // the owned planes start dom[3] planes into the extended field (t is the slowest index)
    const double *own = links_ext + (size_t)dom[3] * Ls * 4 * 18;
    qdd_gauge *g = nullptr, *e = nullptr;
    QDD_TRY(qdd_create_gauge_field(ctx, Lloc, dom, own, links_on_device, &g));
    qdd_status st = qdd_create_gauge_field(ctx, Le, dom, links_ext, links_on_device, &e);
    if (st == QDD_OK) st = slab_setup(g, e, *comm);
    if (st != QDD_OK) {
        if (!g->slab) qdd_destroy_gauge(e);
        qdd_destroy_gauge(g);
        return st;
    }
    *out = g;
    return QDD_OK;
}

void qdd_destroy_gauge(qdd_gauge *g)
{
    if (!g) return;
    cudaSetDevice(g->ctx->device);
    cudaDeviceSynchronize();
    delete g;
}

qdd_status qdd_set_link_compression(qdd_gauge *g, int two_rows)
{
    clear_error();
    if (!g || (two_rows != 0 && two_rows != 1)) {
        set_error("invalid argument");
        return QDD_EINVAL;
    }
    std::lock_guard<std::mutex> lk(g->mu);
    if (two_rows && !g->su3) {
        set_error("links are not SU(3) to %g: the third row cannot be rebuilt from the first two", kSu3Tol);
        return QDD_EINVAL;
    }
    g->two_rows = two_rows != 0;
    return QDD_OK;
}

qdd_status qdd_check_hits(unsigned long long *hits)
{
    clear_error();
    if (!hits) {
        set_error("null argument");
        return QDD_EINVAL;
    }
#ifdef QDD_CHECK
    *hits = check_hits_sap() + check_hits_dslash() + check_hits_mg();
    return QDD_OK;
#else
    *hits = 0;
    set_error("this library was built without range checks (QDD_CHECK)");
    return QDD_EINVAL;
#endif
}

qdd_status qdd_set_schwarz_variant(qdd_gauge *g, int variant)
{
    clear_error();
    if (!g || variant < 0 || variant > 3) {
        set_error("invalid argument");
        return QDD_EINVAL;
    }
    std::lock_guard<std::mutex> lk(g->mu);
    g->sap_variant = variant;
    return QDD_OK;
}

qdd_status qdd_check_set_wait_limit(int device, unsigned spins)
{
    clear_error();
#ifdef QDD_CHECK
    QDD_CUDA(cudaSetDevice(device));
    return set_first_wait_spins_sap(spins);
#else
    (void)device;
    (void)spins;
    set_error("this library was built without range checks (QDD_CHECK)");
    return QDD_EINVAL;
#endif
}

qdd_status qdd_link_compression(qdd_gauge *g, int *two_rows, int *is_su3)
{
    clear_error();
    if (!g || !two_rows || !is_su3) {
        set_error("null argument");
        return QDD_EINVAL;
    }
    *two_rows = g->two_rows ? 1 : 0;
    *is_su3 = g->su3 ? 1 : 0;
    return QDD_OK;
}

qdd_status qdd_set_clover(qdd_gauge *g, double c_sw, double kappa)
{
    clear_error();
    if (!g) return QDD_EINVAL;
    if (!std::isfinite(c_sw) || !std::isfinite(kappa)) {
        set_error("c_sw and kappa must be finite");
        return QDD_EINVAL;
    }
    // a sharded field takes the clover of its owned sites from its extended
    // lattice, whose halo holds the links the boundary planes' leaves need
    qdd_status ext_st = g->slab ? qdd_set_clover(g->slab->ext, c_sw, kappa) : QDD_OK;
    std::lock_guard<std::mutex> lk(g->mu);
    QDD_CUDA(cudaSetDevice(g->ctx->device));
    const size_t cb = (size_t)g->hg.V * 36 * sizeof(double2);
    QDD_TRY(g->clov64.ensure(g->ctx, cb));
    QDD_TRY(g->sclov64.ensure(g->ctx, cb));
    int singular = 0;
    if (g->slab) {
        g->have_clover = false;
        if (ext_st != QDD_OK) return ext_st;
        QDD_TRY(slab_clover_remap(g, 0));
        QDD_CUDA(cudaDeviceSynchronize());
    } else {
        DevMem flag;
        QDD_TRY(flag.alloc(g->ctx, sizeof(int)));
        QDD_CUDA(cudaMemset(flag.p, 0, sizeof(int)));
        FxLock fl;
        if (g->su3) QDD_TRY(fx_acquire(g, false, false, 0, fl));
        QDD_TRY(launch_clover_build(g, c_sw, kappa, flag.as<int>(), fl.owns_lock(), 0));
        QDD_CUDA(cudaMemcpy(&singular, flag.p, sizeof(int), cudaMemcpyDeviceToHost));
    }
    g->ctx->timer.resolve();
    for (auto &c : g->copies) c.valid = false;
    {
        std::unique_lock<std::shared_mutex> ul(g->fx.mu);
        g->fx.have_clov = g->fx.wide = false;
    }
    g->have_clover = false;
    if (singular) {
        set_error("clover block singular on %d sites", singular);
        return QDD_EINVAL;
    }
    g->csw = c_sw;
    g->kappa = kappa;
    g->have_clover = true;
    return QDD_OK;
}

qdd_status qdd_get_clover(qdd_gauge *g, int which, double *out)
{
    clear_error();
    if (!g || !out || (which != 0 && which != 1)) return QDD_EINVAL;
    if (!g->have_clover) {
        set_error("set_clover has not been called");
        return QDD_EINVAL;
    }
    QDD_CUDA(cudaSetDevice(g->ctx->device));
    const HostGeom &hg = g->hg;
    std::vector<double2> buf((size_t)hg.V * 36);
    QDD_CUDA(cudaMemcpy(buf.data(), (which ? g->sclov64 : g->clov64).p, buf.size() * sizeof(double2),
                        cudaMemcpyDeviceToHost));
    for (int gi = 0; gi < hg.V; gi++) {
        int d = gi / hg.Vd, s = gi % hg.Vd;
        int n = hg.site_of[gi];
        for (int blk = 0; blk < 2; blk++) {
            const double2 *p = buf.data() + ((size_t)d * 36 + blk * 18) * hg.Vd + s;
            double *o = out + ((size_t)n * 2 + blk) * 72;  // 36 complex
            double diag[6] = {p[0].x, p[0].y, p[(size_t)hg.Vd].x, p[(size_t)hg.Vd].y, p[(size_t)2 * hg.Vd].x,
                              p[(size_t)2 * hg.Vd].y};
            for (int i = 0; i < 6; i++) {
                o[(i * 6 + i) * 2] = diag[i];
                o[(i * 6 + i) * 2 + 1] = 0;
            }
            int k = 3;
            for (int i = 0; i < 6; i++)
                for (int j = i + 1; j < 6; j++) {
                    double2 v = p[(size_t)k * hg.Vd];
                    o[(i * 6 + j) * 2] = v.x;
                    o[(i * 6 + j) * 2 + 1] = v.y;
                    o[(j * 6 + i) * 2] = v.x;
                    o[(j * 6 + i) * 2 + 1] = -v.y;
                    k++;
                }
        }
    }
    return QDD_OK;
}

qdd_status qdd_apply_D(qdd_gauge *g, const double *in, double *out, int nrhs, qdd_prec prec, int on_device,
                       void *stream)
{
    clear_error();
    if (!g || !in || !out || nrhs < 1 || prec < QDD_PREC_F64 || prec > QDD_PREC_H16) {
        set_error("invalid argument");
        return QDD_EINVAL;
    }
    std::lock_guard<std::mutex> lk(g->mu);
    QDD_CUDA(cudaSetDevice(g->ctx->device));
    cudaStream_t s = (cudaStream_t)stream;
    auto &st = g->stage;  // under g->mu
    if (!st) st.reset(new Staging());
    const size_t V = g->hg.V;
    const size_t eb = elem_bytes(spinor_store(prec));
    const bool scaled = prec == QDD_PREC_F16S || prec == QDD_PREC_BF16S;
    const qdd_prec arith = prec == QDD_PREC_F64 || prec == QDD_PREC_DF64 ? prec : QDD_PREC_F32;
    const qdd_prec fp = field_store(prec);                                // link / clover copy
    if (prec == QDD_PREC_DF64) prec = QDD_PREC_F64;                       // spinor storage
    prec = spinor_store(prec);
    const double *din = nullptr;
    double *dout = nullptr;
    QDD_TRY(stage_in(g, st->io, in, nrhs, on_device, s, &din));
    QDD_TRY(st->a.ensure(g->ctx, V * 12 * eb * nrhs));
    if (g->slab && on_device && out == in) {
        set_error("a sharded field needs separate input and output buffers");
        return QDD_EINVAL;
    }
    if (scaled) {
        QDD_TRY(st->a_s.ensure(g->ctx, V * 4 * nrhs));
        QDD_TRY(st->b_s.ensure(g->ctx, V * 4 * nrhs));
    }
    // a sharded field: its boundary planes (FP64, host layout) move while the operator runs
    QDD_TRY(slab_dslash_begin(g, din, false, true, nrhs, s));
    // FP32 spinors: the operator widens and writes the host layout
    const bool direct = arith == QDD_PREC_F32 && prec == QDD_PREC_F32;
    // FP64-class arithmetic in fixed point: the input is converted on its way in, the
    // operator writes the host layout and goes back to the input at single sites, so
    // the output must not reuse the input's staging, and a device buffer that is both
    // is copied first.  FP64 arithmetic has its result in the same buffer b, which
    // is there before the copy is acquired: nothing is allocated under its lock.
    const size_t bytes = V * 12 * sizeof(double2) * nrhs;
    const bool overlap = on_device && (const char *)in < (const char *)out + bytes && (const char *)out < (const char *)in + bytes;
    FxLock fl;
    if (arith != QDD_PREC_F32) {
        if (!on_device || overlap) QDD_TRY(st->b.ensure(g->ctx, bytes));
        if (g->slab && !on_device) QDD_TRY(st->c.ensure(g->ctx, bytes));
        const qdd_status room = optional_room(st->a_s, g->ctx, fx_exponent_bytes(V, nrhs));
        if (room == QDD_OK) QDD_TRY(fx_acquire(g, arith == QDD_PREC_DF64, true, s, fl));
        else if (room != QDD_EBUDGET) return room;
    }
    const bool fixed = fl.owns_lock();
    if (!fixed && !direct) QDD_TRY(st->b.ensure(g->ctx, V * 12 * eb * nrhs));
    // (a sharded field corrects the output's boundary planes from the input)
    DevMem &oio = g->slab ? st->c : fixed ? st->b : st->io;
    QDD_TRY(stage_out(g, oio, out, nrhs, on_device, s, &dout));
    if (fixed && overlap) {
        QDD_CUDA(cudaMemcpyAsync(st->b.p, din, bytes, cudaMemcpyDeviceToDevice, s));
        din = st->b.as<double>();
    }
    const FxField fxa{st->a.p, st->a_s.as<int>()};
    if (fixed) QDD_TRY(launch_spinor_in_fx(g, din, fxa, nrhs, s));
    else QDD_TRY(launch_spinor_in(g, din, st->a.p, st->a_s.as<float>(), prec, nrhs, s));
    if (fixed) {
        QDD_TRY(launch_dslash_fx(g, fxa, {din, kFxHost64}, (double2 *)dout, true, nullptr, nrhs, s));
    } else if (direct) {
        if (!g->have_clover) {
            set_error("set_clover has not been called");
            return QDD_EINVAL;
        }
        QDD_TRY(launch_dslash_host(g, fp, st->a.p, (double2 *)dout, nrhs, s));
    } else {
        QDD_TRY(launch_dslash(g, arith, fp, st->a.p, st->a_s.as<float>(), prec, st->b.p, st->b_s.as<float>(), prec,
                              nullptr, nrhs, s));
        QDD_TRY(launch_spinor_out(g, st->b.p, st->b_s.as<float>(), dout, prec, nrhs, s));
    }
    QDD_TRY(slab_dslash_end(g, (double2 *)dout, false, nrhs, s));
    return finish_out(g, oio, out, nrhs, on_device, s);
}

qdd_status qdd_sap_apply(qdd_gauge *g, const double *eta, double *psi, double *rho, int nrhs, int nmr, int n_half,
                         qdd_prec prec, int on_device, void *stream)
{
    clear_error();
    if (!g || !eta || !psi || nrhs < 1 || nmr < 0 || n_half < 1 || !is_sap_prec(prec)) {
        set_error("invalid argument");
        return QDD_EINVAL;
    }
    std::lock_guard<std::mutex> lk(g->mu);
    QDD_CUDA(cudaSetDevice(g->ctx->device));
    cudaStream_t s = (cudaStream_t)stream;
    auto &st = g->stage;  // under g->mu
    if (!st) st.reset(new Staging());
    const size_t V = g->hg.V;
    const qdd_prec ssp = spinor_store(prec);                                 // rho storage
    const size_t eb = elem_bytes(ssp);
    const qdd_prec pp = prec == QDD_PREC_F64 ? QDD_PREC_F64 : QDD_PREC_F32;  // psi storage
    const bool scaled = prec == QDD_PREC_F16S || prec == QDD_PREC_BF16S;
    const double *din = nullptr;
    QDD_TRY(stage_in(g, st->io, eta, nrhs, on_device, s, &din));
    QDD_TRY(st->a.ensure(g->ctx, V * 12 * eb * nrhs));                  // rho
    QDD_TRY(st->b.ensure(g->ctx, sap_face_bytes(g->hg, prec, nrhs)));   // face slots
    QDD_TRY(st->c.ensure(g->ctx, V * 12 * elem_bytes(pp) * nrhs));      // psi
    QDD_TRY(st->err.ensure(g->ctx, sizeof(int)));
    if (!st->host_err) QDD_CUDA(cudaMallocHost((void **)&st->host_err, sizeof(int)));
    if (scaled) QDD_TRY(st->a_s.ensure(g->ctx, V * 4 * nrhs));
    QDD_CUDA(cudaMemsetAsync(st->err.p, 0, sizeof(int), s));
    QDD_TRY(launch_spinor_in(g, din, st->a.p, st->a_s.as<float>(), ssp, nrhs, s));
    if (n_half < 2) QDD_CUDA(cudaMemsetAsync(st->c.p, 0, V * 12 * elem_bytes(pp) * nrhs, s));
    SapBuffers b{st->a.p, st->b.p, st->c.p, st->a_s.as<float>()};
    {
        SeqScope seq(g->ctx->timer, K_SAP, s);
        for (int hs = 0; hs < n_half; hs++) {
            // a sharded field exchanges the face slots that cross its slab
            // boundaries while the interior domains are swept
            if (g->slab)
                QDD_TRY(slab_sap_halfsweep(g, prec, b, hs & 1, nmr, nrhs, hs < 2, hs >= 1, st->err.as<int>(), s,
                                           hs + 1 < n_half || rho));
            else
                QDD_TRY(launch_sap_halfsweep(g, prec, b, hs & 1, nmr, nrhs, hs < 2, hs >= 1, 0, st->err.as<int>(), s,
                                             hs >= 1, false));
        }
    }
    if (rho)  // bring the residual of the next colour up to date
        QDD_TRY(launch_sap_halfsweep(g, prec, b, n_half & 1, nmr, nrhs, 0, 1, 1, st->err.as<int>(), s));
    double *dout = nullptr;
    QDD_TRY(stage_out(g, st->io, psi, nrhs, on_device, s, &dout));
    QDD_TRY(launch_spinor_out(g, st->c.p, nullptr, dout, pp, nrhs, s));
    QDD_CUDA(cudaMemcpyAsync(st->host_err, st->err.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    QDD_TRY(finish_out(g, st->io, psi, nrhs, on_device, s));
    if (rho) {
        QDD_TRY(stage_out(g, st->io, rho, nrhs, on_device, s, &dout));
        QDD_TRY(launch_spinor_out(g, st->a.p, st->a_s.as<float>(), dout, ssp, nrhs, s));
        QDD_TRY(finish_out(g, st->io, rho, nrhs, on_device, s));
    }
    const int err = *st->host_err;
    if (err) {
        set_error("device wait ran out in the Schwarz kernel (flags %d)", err);
        return QDD_ETIMEOUT;
    }
    return QDD_OK;
}

void qdd_default_params(qdd_solve_params *p)
{
    if (!p) return;
    p->tol = 1e-10;
    p->restart_m = 16;
    p->max_restarts = 50;
    p->nmr = 4;
    p->ncy = 4;
    p->sap_prec = QDD_PREC_F32;
    p->arnoldi_prec = QDD_PREC_F64;
    p->use_sap = 1;
    p->nrhs = 1;
    p->reorth = 1;
    p->relax_eta = 0.0;
    p->dr_k = 0;
}

qdd_status qdd_solve(qdd_gauge *g, const double *b, double *x, int on_device, const qdd_solve_params *p,
                     qdd_report *rep, void *stream)
{
    clear_error();
    if (!g || !b || !x || !p) {
        set_error("null argument");
        return QDD_EINVAL;
    }
    std::lock_guard<std::mutex> lk(g->mu);
    QDD_CUDA(cudaSetDevice(g->ctx->device));
    if (!g->ws) g->ws = make_workspace();
    return solve_impl(g, g->ws.get(), b, x, on_device, p, rep, (cudaStream_t)stream);
}

qdd_status qdd_cdot_multi(qdd_ctx *ctx, const double *v, int nvec, int64_t ld, const double *w, int64_t n,
                          double *out, void *stream)
{
    clear_error();
    if (!ctx || !v || !w || !out || nvec < 1 || nvec > 64 || n < 1 || ld < n) {
        set_error("invalid argument");
        return QDD_EINVAL;
    }
    QDD_CUDA(cudaSetDevice(ctx->device));
    cudaStream_t s = (cudaStream_t)stream;
    std::lock_guard<std::mutex> lk(ctx->red_mu);
    QDD_TRY(blas_scratch_ensure(ctx, ctx->red_scratch));
    QDD_TRY(blas_cdot_multi(ctx, (const double2 *)v, nvec, ld, (const double2 *)w, n, (double2 *)out,
                            ctx->red_scratch.as<double2>(), s));
    QDD_CUDA(cudaStreamSynchronize(s));
    ctx->timer.resolve();
    return QDD_OK;
}

qdd_status qdd_layout(const int L[4], const int dom[4], int *site_of, uint16_t *nbl, int *nbd)
{
    clear_error();
    if (!L || !dom) return QDD_EINVAL;
    HostGeom hg;
    QDD_TRY(make_geometry(L, dom, hg));
    if (site_of) std::memcpy(site_of, hg.site_of.data(), hg.site_of.size() * sizeof(int));
    if (nbl) std::memcpy(nbl, hg.nbl.data(), hg.nbl.size() * sizeof(uint16_t));
    if (nbd) std::memcpy(nbd, hg.nbd.data(), hg.nbd.size() * sizeof(int));
    return QDD_OK;
}

double qdd_load_model(double n_domains_per_colour, double n_slots)
{
    if (!(n_domains_per_colour > 0) || !(n_slots > 0)) return 0.0;
    double x = n_domains_per_colour / n_slots;
    return x / std::ceil(x);
}

double qdd_domain_working_set(const int dom[4], int link_bytes, int n_full, int n_even)
{
    if (!dom) return 0.0;
    double vd = (double)dom[0] * dom[1] * dom[2] * dom[3];
    return vd * ((72.0 + 72.0) * link_bytes + (24.0 * n_full + 12.0 * n_even) * 4.0);
}

}  // extern "C"
