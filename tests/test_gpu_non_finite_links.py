"""A field with a link entry that is not finite has no clover term, and no operator is applied to it."""
import numpy as np
import pytest

from paper_1502_04025_gb300 import inputs

pytestmark = pytest.mark.gpu

L, DOM = (8, 8, 8, 8), (4, 4, 4, 4)


@pytest.mark.parametrize("entry", [(0, 0), (0, 2), (1, 1), (2, 0), (2, 2)])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf, complex(0, np.nan)])
@pytest.mark.parametrize("csw", [0.0, 1.0])
def test_one_entry(entry, value, csw):
    from paper_1502_04025_gb300 import qdd

    U = inputs.gauge_field(L, 0.7, 1003).reshape(-1, 4, 3, 3)
    U[1234, 1][entry] = value
    ctx = qdd.qdd_create(0, 0)
    g = qdd.qdd_create_gauge_field(ctx, L, DOM, U)
    try:
        assert qdd.qdd_link_compression(g) == (False, False)
        with pytest.raises(qdd.QddError, match="singular"):
            qdd.qdd_set_clover(g, csw, 0.1355)
        with pytest.raises(qdd.QddError, match="set_clover"):
            qdd.qdd_apply_D(g, inputs.gaussian_source(L, 2003), "f64")
    finally:
        qdd.qdd_destroy_gauge(g)
        qdd.qdd_destroy(ctx)
