"""Memory held only for speed never makes a call fail that would fit without it."""
import numpy as np
import pytest

from paper_1502_04025_gb300 import inputs

pytestmark = pytest.mark.gpu

L, DOM = (16, 8, 8, 16), (4, 4, 4, 4)
V = int(np.prod(L))
COPY = V * (2 * 36 * 16 + 4)  # the optional copies of links and clover term


@pytest.fixture(scope="module")
def q():
    from paper_1502_04025_gb300 import qdd

    return qdd


def field(q, ctx):
    g = q.qdd_create_gauge_field(ctx, L, DOM, inputs.gauge_field(L, 0.5, 1001))
    q.qdd_set_clover(g, 1.0, 0.12)
    return g


@pytest.mark.parametrize("sap,kw", [
    ("bf16", {"arnoldi_prec": "f64", "relax_eta": 1e-6}),
    ("bf16", {"arnoldi_prec": "f32"}),
    ("h16", {"arnoldi_prec": "f64", "relax_eta": 1e-6}),
    ("f32", {"arnoldi_prec": "f32"}),
])
@pytest.mark.parametrize("short", [1, V * 96, V * 500, V * 1000, COPY])
def test_solve_that_fits_without_the_copies(q, sap, kw, short):
    """The copies are there when the solve begins; the budget lacks `short` bytes for them and everything else."""
    b = inputs.gaussian_source(L, 2001)

    def run(budget):
        ctx = q.qdd_create(0, budget)
        g = field(q, ctx)
        y = q.qdd_apply_D(g, b, "f64")
        x, rep = q.qdd_solve(g, b, tol=1e-9, sap_prec=sap, **kw)
        used = q.qdd_memory(ctx)[0]
        q.qdd_destroy_gauge(g)
        q.qdd_destroy(ctx)
        assert rep["converged"]
        return y, x, used

    y0, x0, used = run(0)
    y1, x1, used1 = run(used - short)
    assert used1 <= used - short
    assert np.abs(y0 - y1).max() <= 1e-13 * np.abs(y0).max()
    assert np.linalg.norm(x0 - x1) <= 1e-7 * np.linalg.norm(x0)


@pytest.mark.parametrize("use_sap", [0, 1])
def test_plain_solve_in_the_room_it_needs(q, use_sap):
    """The operator's exponents of a solve without Schwarz preconditioner are optional too."""
    b = inputs.gaussian_source(L, 2001)

    def run(budget):
        ctx = q.qdd_create(0, budget)
        g = field(q, ctx)
        x, rep = q.qdd_solve(g, b, tol=1e-6, restart_m=8, max_restarts=20, use_sap=use_sap, sap_prec="f64",
                             arnoldi_prec="f64")
        used = q.qdd_memory(ctx)[0]
        q.qdd_destroy_gauge(g)
        q.qdd_destroy(ctx)
        return x, used

    x0, used = run(0)
    x1, _ = run(used - COPY - (8 * V if not use_sap else 0))
    assert np.linalg.norm(x0 - x1) <= 1e-4 * np.linalg.norm(x0)
