"""The calls this library is timed on.

Each case is one call that a program using the library makes, through the
package's binding (paper_1502_04025_gb300.qdd), with torch CUDA tensors as its
buffers: the full-lattice operator, the Schwarz preconditioner, the fused
multi-dot of the Gram-Schmidt step, the multigrid V-cycle, the preparation of a
new gauge configuration, and whole solves.  Lattices, domain shapes, couplings
and solver settings are those of the repository's workload configurations and
tests, or lie between them.

Every entry point takes and returns FP64 spinors.  Where the arithmetic behind
a result is single precision (or less), the program keeps the result as
complex64, as a mixed-precision outer solver does; FP64 and double-float
results stay complex128.

Inputs: links U = exp(i eps H), H a Gaussian combination of the Gell-Mann
matrices (the repository's recipe, drawn on the GPU), Gaussian or Z2 sources.
"""
import math

import numpy as np
import torch

from paper_1502_04025_gb300 import inputs, qdd

# ------------------------------------------------------------------- the cases

_EASY = {"eps": 0.5, "csw": 1.0, "kappa": 0.125}   # the 16^3x32 workload's couplings
_ROUGH = {"eps": 0.7, "csw": 1.5, "kappa": 0.1355}  # the 32^3x64 and 48^3x96 workloads' couplings


def _lat(L, dom, couplings):
    return {**{f"L{k}": int(v) for k, v in enumerate(L)}, **{f"d{k}": int(v) for k, v in enumerate(dom)}, **couplings}


def listed():
    return [
        # the smallest call in real use: one operator application on a test-size lattice, all latency and launches
        {"name": "D f32 8^4", "kind": "D", "prec": "f32", "nrhs": 1, **_lat((8, 8, 8, 8), (4, 4, 4, 4), _EASY)},
        # the operator on a production lattice, larger than L2: the benchmark's operator line
        {"name": "D f32 32^3x64", "kind": "D", "prec": "f32", "nrhs": 1,
         **_lat((32, 32, 32, 64), (4, 4, 4, 4), _ROUGH)},
        # the FP64 operator (a program's own true-residual check), on extents and domains that are no powers of two
        {"name": "D f64 24x16x12x32", "kind": "D", "prec": "f64", "nrhs": 1,
         **_lat((24, 16, 12, 32), (6, 4, 2, 4), _EASY)},
        # the Gram-Schmidt step of an outer Krylov solver kept in the caller's program: <v_i, w> of five vectors
        {"name": "dots 5 x 16^3x32", "kind": "dots", "nvec": 5, "V": 16 ** 3 * 32},
        # one preconditioner application of the 16^3x32 workload (FP32 links, 8x4^3 domains)
        {"name": "sap f32 16^3x32", "kind": "sap", "prec": "f32", "nrhs": 1, "nmr": 4, "n_half": 8,
         **_lat((16, 16, 16, 32), (8, 4, 4, 4), _EASY)},
        # the same of the large single-source workloads (BF16 storage, 4^4 domains)
        {"name": "sap bf16 32^3x64", "kind": "sap", "prec": "bf16", "nrhs": 1, "nmr": 4, "n_half": 8,
         **_lat((32, 32, 32, 64), (4, 4, 4, 4), _ROUGH)},
        # a propagator's twelve spin-colour sources in one application (FP16 storage)
        {"name": "sap f16 16^3x32 12 src", "kind": "sap", "prec": "f16", "nrhs": 12, "nmr": 4, "n_half": 8,
         **_lat((16, 16, 16, 32), (4, 4, 4, 4), _ROUGH)},
        # the paper's half precision and five MR steps, on a 24-site extent split into 6-site domains
        {"name": "sap h16 24x16x16x24", "kind": "sap", "prec": "h16", "nrhs": 1, "nmr": 5, "n_half": 6,
         **_lat((24, 16, 16, 24), (6, 4, 4, 4), _EASY)},
        # a new gauge configuration: links in, clover term built, the first operator application on it
        {"name": "set-up 16^3x32", "kind": "set-up", **_lat((16, 16, 16, 32), (8, 4, 4, 4), _EASY)},
        # one multigrid V-cycle (a caller's own flexible solver near the critical kappa)
        {"name": "V-cycle 16^3x32", "kind": "vcycle", "nv": 8, "coarse_iters": 12, "post_ncy": 4,
         **_lat((16, 16, 16, 32), (8, 4, 4, 4), {"eps": 0.5, "csw": 1.0, "kappa": 0.138})},
        # whole solves to 1e-10: the 16^3x32 workload, and the large workloads' settings on 32^3x64
        {"name": "solve f32 16^3x32", "kind": "solve", "prec": "f32", "arnoldi": "df64", "nrhs": 1, "nmr": 4,
         "ncy": 4, **_lat((16, 16, 16, 32), (8, 4, 4, 4), _EASY)},
        {"name": "solve bf16 32^3x64", "kind": "solve", "prec": "bf16", "arnoldi": "df64", "nrhs": 1, "nmr": 4,
         "ncy": 4, **_lat((32, 32, 32, 64), (4, 4, 4, 4), _ROUGH)},
    ]


_SHAPES = [(4, 4, 4, 4), (4, 4, 4, 4), (8, 4, 4, 4), (6, 4, 4, 4), (4, 4, 4, 6), (6, 4, 2, 4), (4, 4, 2, 2)]


def _draw_lattice(rng, vmin, vmax):
    """A domain shape and an even number of domains per direction; the volume log-uniform in [vmin, vmax]."""
    target = math.exp(rng.uniform(math.log(vmin), math.log(vmax)))
    while True:
        dom = rng.choice(_SHAPES)
        nb = [2, 2, 2, 2]
        while math.prod(dom) * math.prod(nb) < 0.7 * target:
            nb[rng.randrange(4)] += 2
        L = [a * b for a, b in zip(nb, dom)]
        if max(L) <= 64 and vmin <= math.prod(L) <= vmax:
            return L, dom


def draw(rng):
    kind = rng.choice(["D", "D", "sap", "sap", "sap", "dots", "set-up", "vcycle", "solve", "solve"])
    couplings = dict(rng.choice([_EASY, _ROUGH]))
    if kind == "dots":
        return {"kind": kind, "nvec": rng.randint(1, 17), "V": int(math.exp(rng.uniform(math.log(1000), math.log(1e6))))}
    if kind == "D":
        prec = rng.choice(["f32", "f32", "f64", "df64", "bf16", "f16", "h16"])
        L, dom = _draw_lattice(rng, 4096, 500000 if prec in ("f64", "df64") else 1 << 21)
        nrhs = rng.randint(1, max(1, min(4, (1 << 20) // math.prod(L))))
        return {"kind": kind, "prec": prec, "nrhs": nrhs, **_lat(L, dom, couplings)}
    if kind == "sap":
        prec = rng.choice(["f32", "f32", "bf16", "bf16", "f16", "h16", "f64"])
        L, dom = _draw_lattice(rng, 4096, 50000 if prec == "f64" else 1 << 20)
        nrhs = rng.randint(1, max(1, min(12, 250000 // math.prod(L)))) if prec != "f64" else 1
        return {"kind": kind, "prec": prec, "nrhs": nrhs, "nmr": rng.randint(2, 6), "n_half": rng.randint(2, 8),
                **_lat(L, dom, couplings)}
    if kind == "set-up":
        L, dom = _draw_lattice(rng, 4096, 500000)
        return {"kind": kind, **_lat(L, dom, couplings)}
    if kind == "vcycle":
        L, dom = _draw_lattice(rng, 4096, 150000)
        return {"kind": kind, "nv": rng.randint(4, 12), "coarse_iters": rng.randint(6, 16), "post_ncy": rng.randint(1, 4),
                **_lat(L, dom, {"eps": 0.5, "csw": 1.0, "kappa": rng.choice([0.125, 0.13, 0.138])})}
    prec = rng.choice(["f32", "bf16", "f16", "h16", "f64"])
    L, dom = _draw_lattice(rng, 4096, 9000 if prec == "f64" else 1 << 20)
    nrhs = rng.randint(1, max(1, min(4, 150000 // math.prod(L)))) if prec != "f64" else 1
    return {"kind": "solve", "prec": prec, "arnoldi": "f64" if prec == "f64" else rng.choice(["df64", "df64", "f64"]),
            "nrhs": nrhs, "nmr": rng.randint(3, 5), "ncy": rng.randint(2, 4), **_lat(L, dom, couplings)}


# -------------------------------------------------------------------- inputs

def _geometry(case):
    L = tuple(case[f"L{k}"] for k in range(4))
    dom = tuple(case[f"d{k}"] for k in range(4))
    return L, dom, math.prod(L)


def _generator(seed, stream):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 16 + stream)


def _mm(a, b):
    """Products of 3x3 matrices (..., 3, 3)."""
    return sum(a[..., :, k, None] * b[..., None, k, :] for k in range(3))


def _links(V, eps, seed):
    """Links (V, 4, 3, 3): exp(i eps H) by a Taylor series of a 16th, squared four times, re-unitarised."""
    lam = torch.from_numpy(inputs.gell_mann()).cuda()
    gen = _generator(seed, 0)
    out = torch.empty((V, 4, 3, 3), dtype=torch.complex128, device="cuda")
    step = 1 << 19
    for s in range(0, V, step):
        n = min(step, V - s)
        h = torch.randn((n * 4, 8), dtype=torch.float64, device="cuda", generator=gen)
        X = (0.5j * eps / 16.0) * (h.to(torch.complex128) @ lam.reshape(8, 9)).reshape(n * 4, 3, 3)
        E = torch.eye(3, dtype=torch.complex128, device="cuda").expand_as(X)
        for k in range(10, 0, -1):
            E = torch.eye(3, dtype=torch.complex128, device="cuda") + _mm(X, E) / k
        for _ in range(4):
            E = _mm(E, E)
        a, b = E[:, 0], E[:, 1]
        a = a / a.abs().square().sum(-1, keepdim=True).sqrt()
        b = b - (a.conj() * b).sum(-1, keepdim=True) * a
        b = b / b.abs().square().sum(-1, keepdim=True).sqrt()
        c = torch.linalg.cross(a, b).conj()
        out[s:s + n] = torch.stack((a, b, c), 1).reshape(n, 4, 3, 3)
    return out


def _spinors(V, n, seed, stream, z2=False):
    gen = _generator(seed, stream)
    shape = (V, 4, 3, 2) if n == 1 else (n, V, 4, 3, 2)
    if z2:
        a = (1.0 - 2.0 * torch.randint(0, 2, shape, device="cuda", generator=gen).double()) / math.sqrt(2.0)
    else:
        a = torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen)
    return torch.view_as_complex(a)


_context = []


def _ctx():
    """One library context per process, as a program keeps it."""
    if not _context:
        _context.append(qdd.qdd_create(torch.cuda.current_device()))
    return _context[0]


class _Field:
    """A gauge field of the library, destroyed with its owner."""

    def __init__(self, L, dom, links, csw, kappa):
        self.g = qdd.qdd_create_gauge_field(_ctx(), L, dom, links)
        qdd.qdd_set_clover(self.g, csw, kappa)

    def __del__(self):
        qdd.qdd_destroy_gauge(self.g)


def _inputs(case, seed):
    """The tensors of a case: links and source, or the vectors of the dots."""
    if case["kind"] == "dots":
        n = case["V"] * 12
        v = _spinors(case["V"], case["nvec"], seed, 1).reshape(case["nvec"], n)
        v = v / v.abs().square().sum(-1, keepdim=True).sqrt()  # basis vectors have norm 1
        return {"v": v.contiguous(), "w": _spinors(case["V"], 1, seed, 2).reshape(n)}
    L, _, V = _geometry(case)
    z2 = case["kind"] == "solve" and case["prec"] == "bf16"  # the large workload's noise source
    return {"U": _links(V, case["eps"], seed), "b": _spinors(V, case.get("nrhs", 1), seed, 1, z2)}


def prepare(case, seed):
    st = {"case": case, **_inputs(case, seed)}
    if case["kind"] in ("dots", "set-up"):
        return st
    L, dom, V = _geometry(case)
    st["field"] = _Field(L, dom, st.pop("U"), case["csw"], case["kappa"])
    if case["kind"] == "vcycle":
        qdd.qdd_mg_setup(st["field"].g, _spinors(V, case["nv"], seed, 3), nv=case["nv"], setup_iters=3, setup_ncy=2,
                         nmr=4, post_ncy=case["post_ncy"], coarse_iters=case["coarse_iters"], sap_prec="f32")
    if case["kind"] == "solve":
        st["params"] = qdd.qdd_default_params(
            tol=1e-10, restart_m=16, nmr=case["nmr"], ncy=case["ncy"], sap_prec=case["prec"],
            arnoldi_prec=case["arnoldi"], relax_eta=0.0 if case["prec"] == "f64" else 1e-6, reorth=0,
            max_restarts=200, nrhs=case["nrhs"])
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "dots":
        return qdd.qdd_cdot_multi(_ctx(), st["v"], st["w"])
    if kind == "set-up":
        L, dom, _ = _geometry(case)
        field = _Field(L, dom, st["U"], case["csw"], case["kappa"])
        return qdd.qdd_apply_D(field.g, st["b"], "f64")
    g = st["field"].g
    if kind == "D":
        y = qdd.qdd_apply_D(g, st["b"], case["prec"], nrhs=case["nrhs"])
        return y if case["prec"] in ("f64", "df64") else y.to(torch.complex64)
    if kind == "sap":
        z = qdd.qdd_sap_apply(g, st["b"], case["nmr"], case["n_half"], case["prec"], nrhs=case["nrhs"])
        return z if case["prec"] == "f64" else z.to(torch.complex64)
    if kind == "vcycle":
        return qdd.qdd_mg_vcycle(g, st["b"]).to(torch.complex64)
    return qdd.qdd_solve(g, st["b"], st["params"])[0]


# ---------------------------------------------------------------------- work

_STORE = {"f64": 16, "df64": 16, "f32": 8, "h16": 4, "f16": 4, "bf16": 4}  # bytes of a complex link or clover entry
_D_FLOPS = 1848


def _sap_flops(dom, nmr):
    """Per site and visit of its domain: the hops inside it, MR with even-odd preconditioning, the inflow."""
    c = sum(2.0 / d for d in dom)  # hops of a site that leave the domain
    hops = (8 - c) * 144 + (7 - c) * 24
    return 0.5 * (504 + hops + 24 + nmr * (2 * (hops + 528) + 336) + hops + 528 + 2 * 168 * c)


def work(case):
    kind = case["kind"]
    if kind == "dots":
        n = 12.0 * case["V"]
        return {"bytes": 16 * n * (case["nvec"] + 1) + 16 * case["nvec"], "flops": 8 * n * case["nvec"]}
    _, dom, V = _geometry(case)
    r = case.get("nrhs", 1)
    if kind == "set-up":  # links and source in, the result out; 24 leaf products, the inverse blocks, D
        return {"bytes": V * (576 + 384.0), "flops": V * (24 * 3 * 198 + 2 * 1000 + _D_FLOPS)}
    if kind == "vcycle":  # P twice, links and clover, source and result; transfer, D and the smoother
        return {"bytes": V * (2 * case["nv"] * 96 + 72 * 8 + 384.0),
                "flops": V * (2 * 96.0 * case["nv"] + _D_FLOPS + case["post_ncy"] * _sap_flops(dom, 4))}
    field = 72 * _STORE[case["prec"]]
    if kind == "D":
        return {"bytes": V * (field + 384.0 * r), "flops": float(V) * r * _D_FLOPS}
    if kind == "sap":
        return {"bytes": V * (field + 384.0 * r), "flops": V * r * 0.5 * case["n_half"] * _sap_flops(dom, case["nmr"])}
    # a solve: about five steps, each the preconditioner, D and Gram-Schmidt against the basis so far
    steps = 5
    return {"bytes": V * (field + 384.0 * r),
            "flops": V * r * steps * (case["ncy"] * _sap_flops(dom, case["nmr"]) + _D_FLOPS + 12 * 16.0 * (steps + 1) / 2)}


# --------------------------------------------------------------- 64-bit values

def _gammas():
    sig = np.array([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]], dtype=np.complex128)
    g = np.zeros((4, 4, 4), dtype=np.complex128)
    for k in range(3):
        g[k, :2, 2:], g[k, 2:, :2] = -1j * sig[k], 1j * sig[k]
    g[3, :2, 2:] = g[3, 2:, :2] = np.eye(2)
    return g


class _Dirac:
    """The Wilson-clover operator and the Schwarz method on fields (T, Z, Y, X, ...), in plain torch."""

    def __init__(self, L, U, csw, kappa):
        self.dims, self.kappa = tuple(reversed(L)), kappa
        self.U = [u.contiguous() for u in U.reshape(*self.dims, 4, 3, 3).unbind(4)]
        self.gamma = torch.from_numpy(_gammas()).cuda()
        G = _gammas()
        blocks = torch.zeros((*self.dims, 2, 2, 3, 2, 3), dtype=torch.complex128, device="cuda")
        for mu in range(4):
            for nu in range(mu + 1, 4):
                F = self._field_strength(mu, nu)
                s = 0.5j * (G[mu] @ G[nu] - G[nu] @ G[mu])
                for ch in range(2):
                    for i in range(2):
                        for j in range(2):
                            c = 1j * kappa * csw * s[2 * ch + i, 2 * ch + j]
                            if c != 0:
                                blocks[..., ch, i, :, j, :] += complex(c) * F
        self.A = blocks.reshape(*self.dims, 2, 6, 6)
        self.A += torch.eye(6, dtype=torch.complex128, device="cuda")

    def _at(self, f, mu, d):
        """f(n + d mu) at n."""
        return torch.roll(f, -d, 3 - mu)

    def _field_strength(self, mu, nu):
        um, un, dag = self.U[mu], self.U[nu], lambda m: m.conj().transpose(-1, -2)
        P = _mm(_mm(um, self._at(un, mu, 1)), _mm(dag(self._at(um, nu, 1)), dag(un)))
        Q = P.clone()
        # the other three leaves are plaquettes of the neighbouring corners, turned to start at n
        W = _mm(_mm(self._at(un, mu, 1), dag(self._at(um, nu, 1))), _mm(dag(un), um))  # at n+mu; roll to n
        Q += self._at(W, mu, -1)
        W = _mm(_mm(dag(un), um), _mm(self._at(un, mu, 1), dag(self._at(um, nu, 1))))  # at n+nu
        Q += self._at(W, nu, -1)
        W = _mm(_mm(dag(self._at(um, nu, 1)), dag(un)), _mm(um, self._at(un, mu, 1)))  # at n+mu+nu
        Q += self._at(self._at(W, mu, -1), nu, -1)
        F = (Q - dag(Q)) / 8.0
        tr = F.diagonal(dim1=-2, dim2=-1).sum(-1) / 3.0
        return F - tr[..., None, None] * torch.eye(3, dtype=torch.complex128, device="cuda")

    def clover(self, A, x):
        y = x.reshape(*self.dims, 2, 6)
        return sum(A[..., :, :, j] * y[..., :, None, j] for j in range(6)).reshape(x.shape)

    def hops(self, x, inside=None):
        """H x; inside: per direction and sign, 1 where the hop stays in its domain (the others are dropped)."""
        out = torch.zeros_like(x)
        for mu in range(4):
            for sg in (1, -1):
                if sg > 0:
                    y = self._at(x, mu, 1)
                    y = sum(self.U[mu][..., None, :, b] * y[..., :, None, b] for b in range(3))
                else:
                    y = sum(self.U[mu][..., None, b, :].conj() * x[..., :, None, b] for b in range(3))
                    y = self._at(y, mu, -1)
                if inside is not None:
                    y = y * inside[mu, sg]
                out += y - sg * torch.einsum("st,...tc->...sc", self.gamma[mu], y)
        return out

    def apply(self, x):
        return self.clover(self.A, x) - self.kappa * self.hops(x)

    def schwarz(self, dom, eta, nmr, n_half):
        x = [torch.arange(n, device="cuda").reshape([-1 if 3 - mu == k else 1 for k in range(4)])
             for mu, n in enumerate(reversed(self.dims))]
        shape = (*self.dims, 1, 1)
        inside = {}
        for mu in range(4):
            last, first = (x[mu] % dom[mu]) == dom[mu] - 1, (x[mu] % dom[mu]) == 0
            inside[mu, 1] = (~last).expand(self.dims).reshape(shape).double()
            inside[mu, -1] = (~first).expand(self.dims).reshape(shape).double()
        odd = ((x[0] + x[1] + x[2] + x[3]) % 2 == 1).expand(self.dims).reshape(shape).double()
        block = [x[mu] // dom[mu] for mu in range(4)]
        colour = ((block[0] + block[1] + block[2] + block[3]) % 2).expand(self.dims).reshape(shape)
        index = torch.zeros(self.dims, dtype=torch.int64, device="cuda")
        for mu in (3, 2, 1, 0):
            index = index * (self.dims[3 - mu] // dom[mu]) + block[mu]
        index, nd = index.reshape(-1), int(index.max()) + 1

        def dot(a, b):
            p = (a.conj() * b).sum((-1, -2)).reshape(-1)
            return torch.zeros(nd, dtype=p.dtype, device="cuda").index_add_(0, index, p)[index].reshape(shape)

        Ainv, k = torch.linalg.inv(self.A), self.kappa
        psi, rho = torch.zeros_like(eta), eta.clone()
        for h in range(n_half):
            on = (colour == h % 2).double()
            even, oddm = on * (1 - odd), on * odd
            re, ro = rho * even, rho * oddm
            r = re + k * even * self.hops(oddm * self.clover(Ainv, ro), inside)
            xe = torch.zeros_like(r)
            for _ in range(nmr):
                t = oddm * self.clover(Ainv, -k * self.hops(r, inside))
                p = even * (self.clover(self.A, r) + k * self.hops(t, inside))
                pp = dot(p, p)
                a = torch.where(pp.real > 0, dot(p, r) / pp, torch.zeros_like(pp))
                xe, r = xe + a * r, r - a * p
            delta = xe + oddm * self.clover(Ainv, ro + k * self.hops(xe, inside))
            psi = psi + delta
            rho = rho - self.apply(delta)
        return psi

    def solve(self, b):
        """BiCGStab to the limit of 64 bits."""
        x, r = torch.zeros_like(b), b.clone()
        rt, p = r.clone(), r.clone()
        dot = lambda a, c: torch.vdot(a.reshape(-1), c.reshape(-1))  # noqa: E731
        rho, stop = dot(rt, r), 1e-14 * float(torch.linalg.vector_norm(b))
        for _ in range(400):
            v = self.apply(p)
            alpha = rho / dot(rt, v)
            s = r - alpha * v
            t = self.apply(s)
            om = dot(t, s) / dot(t, t)
            x = x + alpha * p + om * s
            r = s - om * t
            if float(torch.linalg.vector_norm(r)) <= stop:
                break
            new = dot(rt, r)
            p = r + (new / rho) * (alpha / om) * (p - om * v)
            rho = new
        return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "vcycle":
        return None  # the setup alone is dozens of Schwarz applications: past 20 seconds in 64 bits
    if kind == "dots":
        t = _inputs(case, seed)
        return torch.stack([(torch.conj(v) * t["w"]).sum() for v in t["v"]])
    L, dom, V = _geometry(case)
    r = case.get("nrhs", 1)
    cost = {"sap": 8.0 * V * r * case.get("n_half", 0) * (2 * case.get("nmr", 0) + 5), "solve": 8.0 * V * r * 150}
    if cost.get(kind, 0.0) > 3e9:
        return None  # over about 20 seconds
    t = _inputs(case, seed)
    D = _Dirac(L, t.pop("U"), case["csw"], case["kappa"])
    out = []
    for b in (t["b"].reshape(r, V, 4, 3)):
        b = b.reshape(*D.dims, 4, 3)
        y = D.schwarz(dom, b, case["nmr"], case["n_half"]) if kind == "sap" else (
            D.solve(b) if kind == "solve" else D.apply(b))
        out.append(y.reshape(V, 4, 3))
    return out[0] if r == 1 else torch.stack(out)
