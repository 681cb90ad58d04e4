"""Memory held only for speed is given up before the device's own memory runs out."""
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


def test_device_memory_that_runs_out_takes_the_copies_first(q):
    """A request beyond the device's memory, within the budget: what is optional has been given up before it fails,
    and everything works as before."""
    ctx = q.qdd_create(0, 1 << 42)
    g = field(q, ctx)
    b = inputs.gaussian_source(L, 2001)
    y = q.qdd_apply_D(g, b, "f64")
    held = q.qdd_memory(ctx)[0]
    with pytest.raises(q.QddError) as e:
        q.qdd_apply_D(g, b, "f64", nrhs=200000)  # staging of 630 GB, refused before the buffers are read
    assert "cudaMalloc" in str(e.value)
    assert q.qdd_memory(ctx)[0] <= held - COPY
    assert np.abs(q.qdd_apply_D(g, b, "f64") - y).max() <= 1e-13 * np.abs(y).max()
    q.qdd_destroy_gauge(g)
    q.qdd_destroy(ctx)
