"""FP64 and DF64 operators where products leave FP64's range, and within it near its ends."""
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


@pytest.mark.parametrize("prec", ["f64", "df64"])
@pytest.mark.parametrize("link,spinor,csw", [
    (1e-200, 1e-200, 0.0),   # hops below the range: FP64 gives D x = x
    (1e-20, 1e-260, 0.0),    # hops below the normal numbers, x well inside
    (1e-60, 1e-200, 0.0),
    (1e15, 1e260, 1.0),      # clover term near 1e60: the sums overflow
    (1e15, 1e100, 1.0),      # ... and do not
    (1.0, 1e200, 1e160),     # SU(3) links, a clover term that overflows with x
    (1.0, 1.0, 1e60),
    (1.0, 1e-260, 1e-40),
])
def test_products_at_the_ends_of_the_range(env, ora, prec, link, spinor, csw):
    """Where FP64 arithmetic gives infinities or NaN no finite number may stand, where it gives numbers those.

    The bound is 2^-43 of the site's largest result: 64 products per component, the clover entries
    themselves good to a few hundred units of 2^-53 of their largest.
    """
    qdd, c = env
    kappa = 0.12
    U = inputs.gauge_field(L, 0.7, 1003) * link
    x = inputs.gaussian_source(L, 2003) * spinor
    g = qdd.qdd_create_gauge_field(c, L, DOM, U)
    try:
        with np.errstate(all="ignore"):
            qdd.qdd_set_clover(g, csw, kappa)
            got = qdd.qdd_apply_D(g, x, prec).reshape(-1, 12).view(np.float64)
            want = ora.apply_D(L, U, ora.clover(L, U, csw, kappa), kappa, x).reshape(-1, 12).view(np.float64)
    finally:
        qdd.qdd_destroy_gauge(g)
    fin = np.isfinite(want)
    assert not np.isfinite(got[~fin]).any()
    big = np.where(fin, np.abs(want), 0).max(1)[:, None]
    with np.errstate(all="ignore"):
        assert (np.abs(got - want) <= 2.0 ** -43 * big)[fin].all()
