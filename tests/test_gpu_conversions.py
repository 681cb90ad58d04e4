"""The conversions between the host layout (FP64) and the internal storages.

At kappa = c_sw = 0 the operator is the identity, so an application returns the
input as the storage holds it: for FP32 storage every value rounded to FP32,
bit for bit, from values on rounding ties, in FP32's subnormal range, zeros of
both signs and values far below FP32's range; for 16-bit storage a value within
one rounding of the site's scale.  Buffers off the 32-byte boundary take the
16-byte accesses and give the same bits.
"""
import numpy as np
import pytest

from paper_1502_04025_gb300 import inputs

pytestmark = pytest.mark.gpu

L, DOM, V = (8, 4, 4, 12), (4, 2, 2, 2), 8 * 4 * 4 * 12


@pytest.fixture(scope="module")
def field():
    from paper_1502_04025_gb300 import qdd

    ctx = qdd.qdd_create(0, 0)
    g = qdd.qdd_create_gauge_field(ctx, L, DOM, inputs.gauge_field(L, 0.5, 1001))
    qdd.qdd_set_clover(g, 0.0, 0.0)
    yield qdd, g
    qdd.qdd_destroy_gauge(g)
    qdd.qdd_destroy(ctx)


def values(lo, hi):
    """FP64 values with exponents in [lo, hi], a third of them on or next to a tie of the FP32 rounding."""
    rng = np.random.default_rng(5)
    n = V * 24
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    tie = rng.integers(0, 3, n)
    m = np.where(tie == 0, (m & ~np.uint64((1 << 29) - 1)) | np.uint64(1 << 28), m)  # exact ties
    m = np.where(tie == 1, m | np.uint64((1 << 52) - (1 << 28)), m)                  # carries into the exponent
    e = rng.integers(1023 + lo, 1024 + hi, n).astype(np.uint64)
    s = rng.integers(0, 2, n).astype(np.uint64)
    x = ((s << np.uint64(63)) | (e << np.uint64(52)) | m).view(np.float64)
    x[rng.integers(0, n, n // 16)] = 0.0
    x[rng.integers(0, n, n // 16)] = -0.0
    return x.view(np.complex128).reshape(V, 4, 3)


@pytest.mark.parametrize("lo,hi", [(-3, 3), (-170, -110), (-126, 100)])
@pytest.mark.parametrize("offset", [0, 1])
def test_fp32_storage_is_the_rounded_value(field, lo, hi, offset):
    import torch

    qdd, g = field
    x = values(lo, hi)
    buf = torch.zeros(V * 12 + 2, dtype=torch.complex128, device="cuda")
    xin = buf[offset:offset + V * 12].view(V, 4, 3)
    xin.copy_(torch.from_numpy(x))
    out = torch.zeros_like(buf)[offset:offset + V * 12].view(V, 4, 3)
    qdd.qdd_apply_D(g, xin, "f32", out=out)
    want = x.view(np.float64).astype(np.float32).astype(np.float64)
    # y = 1 * x - 0 * (hops): a zero may lose its sign, every other value keeps its bits
    assert np.array_equal(out.cpu().numpy().view(np.float64), want)


@pytest.mark.parametrize("prec,ulp", [("f16", 2.0 ** -11), ("bf16", 2.0 ** -8)])
@pytest.mark.parametrize("size", [1.0, 2.0 ** -90, 2.0 ** -110])
def test_16bit_storage_at_small_scales(field, prec, ulp, size):
    """In and out each round once, relative to the site's largest component, at any size of it."""
    qdd, g = field
    x = inputs.gaussian_source(L, 2001) * size
    y = qdd.qdd_apply_D(g, x, prec)
    scale = np.abs(x.view(np.float64)).reshape(V, 24).max(1)
    err = np.abs((y - x).view(np.float64)).reshape(V, 24).max(1)
    assert (err <= 2 * ulp * scale).all()
