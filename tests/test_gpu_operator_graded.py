"""FP64 and DF64 operators on spinors and links whose entries differ widely in size.

Componentwise, as FP64 arithmetic is: the error of an output component is at
most 64 units of 2^-53 of the sum of the moduli of the products it is made of
(|A||x| + kappa sum |U||h|, h the projected neighbour): fewer than 64 operations
per component, errors of fixed-point sums below FP64's bound by construction.
The reference runs in extended precision (the oracle multiplies before it
projects, so where a projection cancels it is itself off by more than that).
"""
import numpy as np
import pytest

from paper_1502_04025_gb300 import inputs
from tests.test_gpu_links_of_two_sizes import magnitudes

pytestmark = pytest.mark.gpu



def apply_extended(L, U, A, kappa, x):
    """D x in extended precision, hops projected first."""
    R, ext = tuple(reversed(L)), np.clongdouble
    U, A, x = U.reshape(R + (4, 3, 3)).astype(ext), A.reshape(R + (12, 12)).astype(ext), x.reshape(R + (4, 3)).astype(ext)
    out = np.einsum("...ij,...j->...i", A, x.reshape(R + (12,))).reshape(R + (4, 3))
    low = {0: lambda l: -1j * l[..., ::-1, :], 1: lambda l: np.stack([-l[..., 1, :], l[..., 0, :]], -2),
           2: lambda l: np.stack([-1j * l[..., 0, :], 1j * l[..., 1, :]], -2), 3: lambda l: l}
    back_low = {0: lambda w: 1j * w[..., ::-1, :], 1: lambda w: np.stack([w[..., 1, :], -w[..., 0, :]], -2),
                2: lambda w: np.stack([1j * w[..., 0, :], -1j * w[..., 1, :]], -2), 3: lambda w: w}
    k = np.longdouble(kappa)
    for mu in range(4):
        for q in (-1, 1):
            xn = np.roll(x, q, 3 - mu)
            h = xn[..., :2, :] + q * low[mu](xn[..., 2:, :])
            u = U[..., mu, :, :]
            if q > 0:
                u = np.roll(np.conj(np.swapaxes(u, -1, -2)), 1, 3 - mu)
            w = np.einsum("...ab,...sb->...sa", u, h)
            out[..., :2, :] -= k * w
            out[..., 2:, :] -= k * q * back_low[mu](w)
    return out.reshape(-1, 4, 3)


GEOMS = [((8, 8, 8, 8), (4, 4, 4, 4)), ((12, 8, 4, 4), (6, 4, 2, 2))]


@pytest.fixture(scope="module")
def env():
    from paper_1502_04025_gb300 import qdd

    c = qdd.qdd_create(0, 0)
    yield qdd, c
    qdd.qdd_destroy(c)


def source(L, kind, rng):
    x = inputs.gaussian_source(L, 2003)
    V = x.shape[0]
    if kind == "colour":
        x[:, :, 1] *= 1e-9
        x[:, :, 2] *= 1e-18
    elif kind == "one colour":
        x[:, :, 1:] = 0
    elif kind == "spin":
        x[:, 2:] *= 1e-12
    elif kind == "components":
        x *= 10.0 ** rng.uniform(-15, 0, x.shape)
    elif kind == "sites":
        x *= 10.0 ** rng.uniform(-15, 15, (V, 1, 1))
    elif kind == "point":
        x[:] = 0
        x[V // 3, 1, 2] = 1.0 + 0.5j
    elif kind == "slice":
        t = np.arange(V) // (L[0] * L[1] * L[2])
        x[t != 1] = 0
    elif kind == "even":
        n = np.arange(V)
        p = (n % L[0] + n // L[0] % L[1] + n // (L[0] * L[1]) % L[2] + n // (L[0] * L[1] * L[2])) & 1
        x[p == 1] = 0
    return x


KINDS = ["gauss", "colour", "one colour", "spin", "components", "sites", "point", "slice", "even"]


def links(L, kind, rng):
    if kind == "unit":
        return inputs.unit_gauge_field(L)
    if kind == "weak":
        return inputs.gauge_field(L, 1e-6, 1003)
    U = inputs.gauge_field(L, 0.7, 1003)
    if kind == "phases":  # not SU(3): antiperiodic in t, and a phase per site
        R = U.reshape(-1, 4, 3, 3)
        R *= np.exp(1j * rng.uniform(-3, 3, (R.shape[0], 4, 1, 1)))
        R[-L[0] * L[1] * L[2]:, 3] *= -1
    return U


@pytest.mark.parametrize("L,dom", GEOMS)
@pytest.mark.parametrize("prec", ["f64", "df64"])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("field", ["rough", "weak", "unit", "phases"])
def test_every_component_to_fp64(env, L, dom, prec, kind, field):
    """Host buffers, device buffers, and a device buffer that is both input and output."""
    import torch

    qdd, c = env
    rng = np.random.default_rng(11)
    csw, kappa = (1.5, 0.1355) if field != "unit" else (0.0, 0.125)
    U = links(L, field, rng)
    x = source(L, kind, rng)
    g = qdd.qdd_create_gauge_field(c, L, dom, U)
    qdd.qdd_set_clover(g, csw, kappa)
    blocks = qdd.qdd_get_clover(g, x.shape[0])
    A = np.zeros((x.shape[0], 12, 12), np.complex128)
    A[:, :6, :6], A[:, 6:, 6:] = blocks[:, 0], blocks[:, 1]
    want = apply_extended(L, U, A, kappa, x)
    bound = 64 * 2.0 ** -53 * magnitudes(L, U, A, kappa, x)
    xd = torch.from_numpy(x).cuda()
    outs = [qdd.qdd_apply_D(g, x, prec), qdd.qdd_apply_D(g, xd, prec).cpu().numpy()]
    outs.append(qdd.qdd_apply_D(g, xd, prec, out=xd).cpu().numpy())
    qdd.qdd_destroy_gauge(g)
    for y in outs:
        err = np.abs(y.reshape(-1, 4, 3) - want)
        assert (err <= bound).all(), (err - bound).max()
    assert np.array_equal(outs[0], outs[1]) and np.array_equal(outs[0], outs[2])


@pytest.mark.parametrize("prec", ["f64", "df64"])
@pytest.mark.parametrize("kind", KINDS)
def test_no_hops_and_no_clover_is_the_identity(env, prec, kind):
    qdd, c = env
    L, dom = GEOMS[1]
    x = source(L, kind, np.random.default_rng(12))
    g = qdd.qdd_create_gauge_field(c, L, dom, inputs.gauge_field(L, 0.7, 1003))
    qdd.qdd_set_clover(g, 0.0, 0.0)
    y = qdd.qdd_apply_D(g, x, prec)
    qdd.qdd_destroy_gauge(g)
    assert np.array_equal(y, x)


@pytest.mark.parametrize("arnoldi", ["f64", "df64"])
@pytest.mark.parametrize("sap", ["f32", "bf16"])
def test_solve_of_a_point_source(env, ora, arnoldi, sap):
    """Twelve sources at a point: graded at the start and around the source, FP64 and FP32 directions and residuals."""
    qdd, c = env
    L, dom = (8, 8, 8, 8), (4, 4, 4, 4)
    U = inputs.gauge_field(L, 0.5, 1001)
    A = ora.clover(L, U, 1.0, 0.12)
    g = qdd.qdd_create_gauge_field(c, L, dom, U)
    qdd.qdd_set_clover(g, 1.0, 0.12)
    b = inputs.point_sources(L, 100)
    x, rep = qdd.qdd_solve(g, b, tol=1e-11, nrhs=12, sap_prec=sap, arnoldi_prec=arnoldi)
    qdd.qdd_destroy_gauge(g)
    for k in range(12):
        r = b[k] - ora.apply_D(L, U, A, 0.12, np.ascontiguousarray(x[k]))
        assert np.linalg.norm(r) <= 1.01e-11 * np.linalg.norm(b[k])


@pytest.mark.parametrize("nrhs", [1, 2])
@pytest.mark.parametrize("sites", ["one", "few", "most"])
def test_lists_of_every_length(env, sites, nrhs):
    """Sites left to FP64 arithmetic, from a single one (a warp per site) to more than the kernel's
    warps take (a thread per site), in host layout and planes: a solve's residual and directions too."""
    qdd, c = env
    L, dom = (24, 16, 12, 16), (6, 4, 2, 4)
    rng = np.random.default_rng(13)
    U = inputs.gauge_field(L, 0.7, 1003)
    V = int(np.prod(L))
    x = np.stack([inputs.gaussian_source(L, 2003 + k) for k in range(nrhs)])
    at = {"one": [V // 2], "few": rng.choice(V, 300, replace=False), "most": np.arange(V)}[sites]
    x[:, at] *= 10.0 ** rng.uniform(-18, 0, (nrhs, len(at), 4, 3))
    x[:, at, :, 1:] *= 1e-18
    csw, kappa = 1.5, 0.1355
    g = qdd.qdd_create_gauge_field(c, L, dom, U)
    qdd.qdd_set_clover(g, csw, kappa)
    blocks = qdd.qdd_get_clover(g, V)
    y = qdd.qdd_apply_D(g, x if nrhs > 1 else x[0], "f64", nrhs=nrhs).reshape(nrhs, V, 4, 3)
    _, rep = qdd.qdd_solve(g, x if nrhs > 1 else x[0], nrhs=nrhs, tol=1e-10, sap_prec="f32", arnoldi_prec="f64")
    qdd.qdd_destroy_gauge(g)
    A = np.zeros((V, 12, 12), np.complex128)
    A[:, :6, :6], A[:, 6:, 6:] = blocks[:, 0], blocks[:, 1]
    for k in range(nrhs):
        err = np.abs(y[k] - apply_extended(L, U, A, kappa, x[k]))
        assert (err <= 64 * 2.0 ** -53 * magnitudes(L, U, A, kappa, x[k])).all()
    assert rep["converged"] and rep["true_rel_res"] <= 1e-10
