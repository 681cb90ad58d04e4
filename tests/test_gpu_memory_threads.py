"""Optional copies given up while another thread uses and rebuilds them."""
import threading

import numpy as np
import pytest

from paper_1502_04025_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_allocations_against_a_thread_that_rebuilds_its_copy():
    """One thread applies the FP64 operator again and again, and has its fixed-point copy back whenever there is
    room; another needs that room for a moment, every time.  No call of either is refused."""
    from paper_1502_04025_gb300 import qdd

    La, Lb = (16, 8, 8, 16), (8, 8, 8, 8)
    dom, sources = (4, 4, 4, 4), 70
    Va, Vb = int(np.prod(La)), int(np.prod(Lb))
    base_a = Va * (3 * 576 + 3 * 192 + 8)           # links, clover forms, staging, exponents
    base_b = Vb * (3 * 576 + 288 * sources)          # the same and FP32 staging of all sources
    copies_b = Vb * 2200                             # FP32 copies of links (whole, two rows) and clover forms
    budget = base_a + base_b + copies_b + Va * 600   # room for half of the first field's copy
    assert base_a + Va * 1156 <= budget // 2
    ctx = qdd.qdd_create(0, budget)
    Ua, Ub = inputs.gauge_field(La, 0.5, 1001), inputs.gauge_field(Lb, 0.5, 1003)
    a = qdd.qdd_create_gauge_field(ctx, La, dom, Ua)
    qdd.qdd_set_clover(a, 1.0, 0.12)
    xa = inputs.gaussian_source(La, 2001)
    want = qdd.qdd_apply_D(a, xa, "f64")
    xb = np.stack([inputs.gaussian_source(Lb, 3000)] * sources)
    stop, errors, calls = threading.Event(), [], [0]

    def loop():
        try:
            while not stop.is_set():
                y = qdd.qdd_apply_D(a, xa, "f64")
                assert np.abs(y - want).max() <= 1e-13 * np.abs(want).max()
                calls[0] += 1
        except Exception as e:  # shown by the main thread
            errors.append(e)

    t = threading.Thread(target=loop)
    t.start()
    try:
        for _ in range(40):
            b = qdd.qdd_create_gauge_field(ctx, Lb, dom, Ub)
            qdd.qdd_set_clover(b, 1.0, 0.12)
            qdd.qdd_apply_D(b, xb, "f32", nrhs=sources)
            qdd.qdd_destroy_gauge(b)
    finally:
        stop.set()
        t.join()
    qdd.qdd_destroy_gauge(a)
    assert qdd.qdd_memory(ctx)[0] <= 1 << 20
    qdd.qdd_destroy(ctx)
    assert not errors, errors[0]
    assert calls[0] > 10
