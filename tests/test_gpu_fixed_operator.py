"""The FP64 and double-float precisions of the operator, computed in 64-bit fixed point.

Every real of a site keeps 57 bits below the site's largest one, and the hops
into a site are added at the largest scale of the nine sites involved, so an
output's error is bounded against the largest input component of those nine
sites, whatever the sizes of the others.  With |U| <= 1 (or u), |A| <= a and
kappa < 1/4 each output sums fewer than 12 a + 8 * 12 u kappa products, each
off by at most 2^-55 of that component, and is rounded to FP64 twice: 64 (a + u)
units of 2^-53 cover both this and the reference's own rounding.
"""
import numpy as np
import pytest

from paper_1502_04025_gb300 import inputs

pytestmark = pytest.mark.gpu

GEOMS = [((8, 8, 8, 8), (4, 4, 4, 4)), ((4, 4, 4, 4), (2, 2, 2, 2)), ((12, 8, 4, 4), (6, 4, 2, 2)),
         ((16, 8, 8, 8), (8, 4, 4, 4))]
CSW, KAPPA = 1.5, 0.1355


@pytest.fixture(scope="module")
def q():
    from paper_1502_04025_gb300 import qdd

    return qdd


@pytest.fixture(scope="module")
def ctx(q):
    c = q.qdd_create(0, 0)
    yield c
    q.qdd_destroy(c)


def near_max(L, x):
    """Per site, the largest input component of the site and its eight neighbours."""
    m = np.abs(x.view(np.float64)).reshape(tuple(reversed(L)) + (24,)).max(-1)
    out = m.copy()
    for ax in range(4):
        for d in (1, -1):
            out = np.maximum(out, np.roll(m, d, ax))
    return out.reshape(-1)


def check(L, x, got, want, size=1.0):
    err = np.abs((got - want).view(np.float64)).reshape(-1, 24).max(1)
    assert (err <= 64 * (1.5 + size) * 2.0 ** -53 * near_max(L, x)).all()


@pytest.mark.parametrize("L,dom", GEOMS)
@pytest.mark.parametrize("prec", ["f64", "df64"])
@pytest.mark.parametrize("scales", [0, 3, 200])
def test_sites_of_any_size(q, ctx, ora, L, dom, prec, scales):
    """Gaussian sites times 10^U(-scales, scales), some of them zero."""
    U = inputs.gauge_field(L, 0.7, 1003)
    A = ora.clover(L, U, CSW, KAPPA)
    x = inputs.gaussian_source(L, 2003)
    rng = np.random.default_rng(3)
    V = x.shape[0]
    x = x * (10.0 ** rng.uniform(-scales, scales, V) * (rng.uniform(size=V) > 0.2))[:, None, None]
    g = q.qdd_create_gauge_field(ctx, L, dom, U)
    q.qdd_set_clover(g, CSW, KAPPA)
    check(L, x, q.qdd_apply_D(g, x, prec), ora.apply_D(L, U, A, KAPPA, x))
    xs = np.stack([x, inputs.gaussian_source(L, 2004)])
    both = q.qdd_apply_D(g, xs, prec, nrhs=2)
    check(L, xs[1], both[1], ora.apply_D(L, U, A, KAPPA, xs[1]))
    q.qdd_destroy_gauge(g)


@pytest.mark.parametrize("prec", ["f64", "df64"])
@pytest.mark.parametrize("kind", ["fp32", "powers", "z2"])
def test_values_on_limb_boundaries(q, ctx, ora, prec, kind):
    """Few significant bits: the lower limbs take their extreme values, in one component and in sums of two."""
    L, dom = (8, 8, 8, 8), (4, 4, 4, 4)
    U = inputs.gauge_field(L, 0.7, 1003)
    A = ora.clover(L, U, CSW, KAPPA)
    x = inputs.gaussian_source(L, 2003)
    if kind == "fp32":
        x = x.astype(np.complex64).astype(np.complex128)
    elif kind == "z2":
        x = inputs.z2_source(L, 2003)
    else:
        rng = np.random.default_rng(9)
        x = (2.0 ** rng.integers(-60, 1, x.view(np.float64).shape) * rng.choice([-1, 1], x.view(np.float64).shape)).view(np.complex128)
    g = q.qdd_create_gauge_field(ctx, L, dom, U)
    q.qdd_set_clover(g, CSW, KAPPA)
    check(L, x, q.qdd_apply_D(g, x, prec), ora.apply_D(L, U, A, KAPPA, x))
    q.qdd_destroy_gauge(g)


@pytest.mark.parametrize("sap", ["f32", "bf16"])
@pytest.mark.parametrize("arnoldi", ["f64", "df64"])
def test_arnoldi_operator_on_fp32_directions(q, ctx, sap, arnoldi):
    """The estimate of the small least-squares problem is the true residual, to FP64 rounding, only if the
    Arnoldi steps applied the operator of the true residual to the FP32 directions z_j."""
    L, dom = (8, 8, 8, 16), (4, 4, 4, 4)
    g = q.qdd_create_gauge_field(ctx, L, dom, inputs.gauge_field(L, 0.5, 1001))
    q.qdd_set_clover(g, 1.0, 0.12)
    _, rep = q.qdd_solve(g, inputs.gaussian_source(L, 2001), tol=1e-10, sap_prec=sap, arnoldi_prec=arnoldi)
    assert rep["restarts"] == 0 and abs(rep["true_rel_res"] - rep["est_rel_res"]) <= 1e-14
    q.qdd_destroy_gauge(g)


@pytest.mark.parametrize("size", [1.0 + 1e-6, 1.5, 1000.0, 1e30])
def test_links_off_su3(q, ctx, ora, size):
    """Links of another size (not SU(3)) take another scale; far too large ones FP64 arithmetic."""
    L, dom = (8, 4, 4, 12), (4, 2, 2, 2)
    U = inputs.gauge_field(L, 0.7, 1003) * size
    x = inputs.gaussian_source(L, 2003)
    g = q.qdd_create_gauge_field(ctx, L, dom, U)
    q.qdd_set_clover(g, 0.0, KAPPA)  # A = 1
    A = ora.clover(L, U, 0.0, KAPPA)
    for prec in ("f64", "df64"):
        check(L, x, q.qdd_apply_D(g, x, prec), ora.apply_D(L, U, A, KAPPA, x), size)
    q.qdd_destroy_gauge(g)


@pytest.mark.parametrize("prec", ["f64", "df64"])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e304, 1e-305, 5e-324])
def test_extreme_values_stay_where_they_are(q, ctx, ora, prec, value):
    """One component out of range: the nine sites that read it are computed in FP64, all others are untouched."""
    L, dom = (8, 8, 8, 8), (4, 4, 4, 4)
    U = inputs.gauge_field(L, 0.7, 1003)
    A = ora.clover(L, U, CSW, KAPPA)
    x = inputs.gaussian_source(L, 2003)
    clean = x.copy()
    clean[77, 2, 1] = 0.0
    x[77, 2, 1] = value
    if abs(value) < 1:
        x[77] = clean[77] = 0.0
        x[77, 2, 1] = value
    g = q.qdd_create_gauge_field(ctx, L, dom, U)
    q.qdd_set_clover(g, CSW, KAPPA)
    got = q.qdd_apply_D(g, x, prec)
    marked = np.zeros(tuple(reversed(L)), bool)
    marked.reshape(-1)[77] = True
    near = marked.copy()
    for ax in range(4):
        near |= np.roll(marked, 1, ax) | np.roll(marked, -1, ax)
    near = near.reshape(-1)
    base = q.qdd_apply_D(g, clean, prec)
    assert np.array_equal(got[~near], base[~near])
    if np.isfinite(value):
        check(L, x, got, ora.apply_D(L, U, A, KAPPA, x))
    else:
        assert not np.isfinite(got[near]).all(axis=(1, 2)).any()
        # a hop keeps the two spins it does not touch: some components stay finite
        assert np.isfinite(got[near]).any()
    q.qdd_destroy_gauge(g)


def test_optional_copies_give_way_to_a_tight_budget(q):
    """What ran within a budget without the optional fixed-point copies still does: they are given up when an
    allocation needs their room, and built again (or replaced by FP64 arithmetic) afterwards."""
    L, dom = (16, 8, 8, 16), (4, 4, 4, 4)
    V = int(np.prod(L))
    U, b = inputs.gauge_field(L, 0.5, 1001), inputs.gaussian_source(L, 2001)

    def steps(budget):
        ctx = q.qdd_create(0, budget)
        g = q.qdd_create_gauge_field(ctx, L, dom, U)
        q.qdd_set_clover(g, 1.0, 0.12)
        y = q.qdd_apply_D(g, b, "f64")
        x, rep = q.qdd_solve(g, b, tol=1e-10, sap_prec="f32", arnoldi_prec="f32")
        z = q.qdd_apply_D(g, x, "f64")
        used = q.qdd_memory(ctx)[0]
        q.qdd_destroy_gauge(g)
        assert q.qdd_memory(ctx)[0] <= 1 << 20
        q.qdd_destroy(ctx)
        return y, x, z, used

    y0, x0, z0, used = steps(0)
    # without the copies, with the output buffer that FP64 arithmetic needs in their place
    budget = used - V * (2 * 36 * 16 + 4) + V * 192
    y1, x1, z1, used1 = steps(budget)
    assert used1 <= budget
    for a, c in ((y0, y1), (z0, z1)):
        assert np.abs(a - c).max() <= 1e-13 * np.abs(a).max()
    assert np.linalg.norm(x0 - x1) <= 1e-9 * np.linalg.norm(x0)
