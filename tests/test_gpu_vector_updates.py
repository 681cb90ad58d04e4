"""The vector updates of the solver (w - sum h v, x + sum y z) in fixed point.

In plain GMRES (no preconditioner, FP64 operator) every basis vector and the
solution pass through them, with 1 to 24 vectors per update, on vectors that
are dense, zero almost everywhere, and out of the range that fixed point takes.
The estimate of the small least-squares problem equals the true residual only
as far as orthogonality and updates hold: with m <= 24 steps, a few times
24 * 2^-53 of |b|; 1e-13 covers it with a factor of 30.
"""
import numpy as np
import pytest

from paper_1502_04025_gb300 import inputs

pytestmark = pytest.mark.gpu

L, DOM, CSW, KAPPA = (8, 4, 4, 8), (4, 2, 2, 2), 1.0, 0.12


@pytest.fixture(scope="module")
def problem():
    from oracle import pyoracle as ora
    from paper_1502_04025_gb300 import qdd

    U = inputs.gauge_field(L, 0.5, 1001)
    ctx = qdd.qdd_create(0, 0)
    g = qdd.qdd_create_gauge_field(ctx, L, DOM, U)
    qdd.qdd_set_clover(g, CSW, KAPPA)
    yield qdd, ora, g, U, ora.clover(L, U, CSW, KAPPA)
    qdd.qdd_destroy_gauge(g)
    qdd.qdd_destroy(ctx)


def source(kind):
    if kind == "point":
        return inputs.point_source(L, 1, 2, 100)
    size = {"gauss": 1.0, "large": 1e100, "small": 1e-130}[kind]
    return inputs.gaussian_source(L, 2001) * size


@pytest.mark.parametrize("kind", ["gauss", "point", "large", "small"])
@pytest.mark.parametrize("m", [1, 5, 16, 24])
@pytest.mark.parametrize("use_sap", [0, 1])
def test_cycles_of_m_steps(problem, kind, m, use_sap):
    qdd, ora, g, U, A = problem
    b = source(kind)
    x, rep = qdd.qdd_solve(g, b, tol=1e-300, restart_m=m, max_restarts=0, use_sap=use_sap, sap_prec="f64" if not use_sap else "f32",
                           reorth=2, allow_noconv=True)
    r = b - ora.apply_D(L, U, A, KAPPA, x)
    true = np.linalg.norm(r) / np.linalg.norm(b)
    assert abs(true - rep["est_rel_res"]) <= 1e-13
    # one cycle reduces the residual as minimal residual methods do on this system
    assert true < 0.7 ** m + 1e-13


@pytest.mark.parametrize("kind", ["gauss", "point"])
def test_two_sources_are_each_alone(problem, kind):
    qdd, ora, g, U, A = problem
    bs = np.stack([source(kind), inputs.gaussian_source(L, 2002)])
    x, _ = qdd.qdd_solve(g, bs, tol=1e-11, nrhs=2)
    for k in range(2):
        x1, _ = qdd.qdd_solve(g, np.ascontiguousarray(bs[k]), tol=1e-11)
        assert np.linalg.norm(x[k] - x1) <= 1e-9 * np.linalg.norm(x1)
