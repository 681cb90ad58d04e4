"""The solver's vector updates on elements whose parts differ widely in size.

With kappa = c_sw = 0 the operator is the identity, so one step of plain GMRES
gives v = b / |b|, h = <v, v>, x = |b| / h v: x equals b to a few roundings of
each part.  h's and y's imaginary parts are the rounding of sums of products
re * im of v, at most 2^-53 (64 + n / 25600) sum |re||im| of |v| = 1, which moves
a part by that times the other part.
"""
import numpy as np
import pytest

from paper_1502_04025_gb300 import inputs

pytestmark = pytest.mark.gpu

L, DOM = (8, 4, 4, 8), (4, 2, 2, 2)


@pytest.fixture(scope="module")
def env():
    from paper_1502_04025_gb300 import qdd

    c = qdd.qdd_create(0, 0)
    yield qdd, c
    qdd.qdd_destroy(c)


def field(qdd, c, L, dom):
    g = qdd.qdd_create_gauge_field(c, L, dom, inputs.unit_gauge_field(L))
    qdd.qdd_set_clover(g, 0.0, 0.0)
    return g


def close(x, b):
    """Part by part, with the rotation by the rounding of h."""
    x, b = x.reshape(-1), b.reshape(-1)
    unit = 2.0 ** -53
    rot = unit * (64 + b.size / 25600) * (np.abs(b.real) * np.abs(b.imag)).sum() / (np.abs(b) ** 2).sum()
    assert (np.abs(x.real - b.real) <= 16 * unit * np.abs(b.real) + 4 * rot * np.abs(b.imag)).all()
    assert (np.abs(x.imag - b.imag) <= 16 * unit * np.abs(b.imag) + 4 * rot * np.abs(b.real)).all()


@pytest.mark.parametrize("geom", [(L, DOM), ((16, 16, 8, 12), (4, 4, 4, 2))])
@pytest.mark.parametrize("small", [0.0, 1e-3, 1e-6, 1e-10, 1e-14])
def test_small_parts_of_large_elements(env, geom, small):
    qdd, c = env
    L, dom = geom
    g = field(qdd, c, L, dom)
    rng = np.random.default_rng(5)
    b = inputs.gaussian_source(L, 7)
    tiny_im = rng.uniform(size=b.shape) < 0.5
    b = np.where(tiny_im, b.real + 1j * small * b.imag, small * b.real + 1j * b.imag)
    x, _ = qdd.qdd_solve(g, b, tol=1e-300, restart_m=1, max_restarts=0, use_sap=0, sap_prec="f64", allow_noconv=True)
    qdd.qdd_destroy_gauge(g)
    close(x, b)


@pytest.mark.parametrize("size", [1e-100, 1e-106, 1e-112, 1e-118, 1e-121, 1e-130, 1e100])
def test_zero_sums_take_small_terms_whole(env, size):
    """x = 0 + y v with y from inside the fixed-point range to below it."""
    qdd, c = env
    g = field(qdd, c, L, DOM)
    b = inputs.gaussian_source(L, 7) * size
    x, _ = qdd.qdd_solve(g, b, tol=1e-300, restart_m=1, max_restarts=0, use_sap=0, sap_prec="f64", allow_noconv=True)
    qdd.qdd_destroy_gauge(g)
    close(x, b)


@pytest.mark.parametrize("shape", [((16, 16, 8, 12), (4, 4, 4, 2)), ((24, 8, 8, 12), (4, 4, 4, 2))])
@pytest.mark.parametrize("m", [3, 5, 18, 24])
@pytest.mark.parametrize("use_sap", [0, 1])
def test_long_vectors(ora, env, shape, m, use_sap):
    """Vectors of several passes of the update's main loop and a remainder, FP64 and FP32 directions: the
    estimate of the small least-squares problem is the true residual as far as every update held (the
    bound of test_gpu_vector_updates)."""
    qdd, c = env
    L, dom = shape
    U = inputs.gauge_field(L, 0.5, 1001)
    g = qdd.qdd_create_gauge_field(c, L, dom, U)
    qdd.qdd_set_clover(g, 1.0, 0.12)
    b = inputs.gaussian_source(L, 2001)
    x, rep = qdd.qdd_solve(g, b, tol=1e-300, restart_m=m, max_restarts=0, use_sap=use_sap,
                           sap_prec="f32" if use_sap else "f64", reorth=2, allow_noconv=True)
    qdd.qdd_destroy_gauge(g)
    r = b - ora.apply_D(L, U, ora.clover(L, U, 1.0, 0.12), 0.12, x)
    assert abs(np.linalg.norm(r) / np.linalg.norm(b) - rep["est_rel_res"]) <= 1e-13
