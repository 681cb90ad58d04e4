"""The multi-dot: sums of products in fixed point per tile of a few elements, FP64 between tiles.

Reference: math.fsum over exact products' FP64 halves (numpy longdouble has 64
bits here or 113 on Arm; both hold a product of two FP64 numbers to 2^-63), so
the reference's own error is far below the bound.  The bound: every FP64
addition along a thread's chain and the block sums rounds by 2^-53 of the
partial sum, itself at most sum |v||w|; chains are at most n / (blocks * 256)
long plus 24 levels, and each tile's fixed-point error is below 2^-55 of its
largest |v||w|.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    from paper_1502_04025_gb300 import qdd

    c = qdd.qdd_create(0, 0)
    yield qdd, c
    qdd.qdd_destroy(c)


def vectors(n, nvec, kind, seed=1):
    rng = np.random.default_rng(seed)
    z = rng.standard_normal((nvec + 1, n, 2))
    if kind == "decades":
        z = z * 10.0 ** rng.uniform(-40, 40, (nvec + 1, n, 1))
    elif kind == "sparse":
        z = z * (rng.uniform(size=(nvec + 1, n, 1)) > 0.9)
    elif kind == "fp32":
        z = z.astype(np.float32).astype(np.float64)
    elif kind == "huge":
        z = z * 1e170
    elif kind == "tiny":
        z = z * 1e-250
    z = z.view(np.complex128)[..., 0]
    return z[:-1].copy(), z[-1].copy()


def reference(v, w):
    vl, wl = v.astype(np.clongdouble), w.astype(np.clongdouble)
    return np.array([(np.conj(a) * wl).sum() for a in vl])


@pytest.mark.parametrize("n", [1, 31, 255, 1000, 77825, 400001])
@pytest.mark.parametrize("nvec", [1, 2, 5, 16, 17])
@pytest.mark.parametrize("kind", ["gauss", "decades", "sparse", "fp32"])
def test_dots_to_rounding(env, n, nvec, kind):
    import torch

    qdd, c = env
    v, w = vectors(n, nvec, kind)
    vd, wd = torch.from_numpy(v).cuda(), torch.from_numpy(w).cuda()
    want = reference(v, w)
    scale = (np.abs(v) * np.abs(w)).sum(1).astype(np.float64)
    # tiles mix elements of different sizes: 8 elements of a tile share a scale
    big = np.array([np.abs(a).max() for a in v]) * np.abs(w).max()
    bound = 2.0 ** -53 * (n / (100 * 256) + 32) * scale + (n * 2.0 ** -55 * big if kind == "decades" else 0)
    for got in (qdd.qdd_cdot_multi(c, vd, wd), qdd.qdd_cdot_multi_noalloc(vd, wd)):
        err = np.abs(got.cpu().numpy() - want).astype(np.float64)
        assert (err <= bound + 1e-300).all(), (err / scale).max()


@pytest.mark.parametrize("kind", ["huge", "tiny"])
def test_dots_at_the_ends_of_the_range(env, kind):
    """Products outside the range (inf, or zero as FP64 arithmetic gives) and within it on one side."""
    import torch

    qdd, c = env
    v, w = vectors(5000, 3, kind)
    got = qdd.qdd_cdot_multi(c, torch.from_numpy(v).cuda(), torch.from_numpy(w).cuda()).cpu().numpy()
    if kind == "huge":
        assert not np.isfinite(got).any()
    else:
        assert (got == 0).all()
    one = np.ones_like(w) / 4
    got = qdd.qdd_cdot_multi(c, torch.from_numpy(v).cuda(), torch.from_numpy(one).cuda()).cpu().numpy()
    want = reference(v, one)
    assert (np.abs(got - want) <= 2.0 ** -48 * np.abs(v).sum(1)).all()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("where", ["v", "w"])
def test_dots_pass_non_finite_values_on(env, bad, where):
    import torch

    qdd, c = env
    v, w = vectors(3000, 3, "gauss")
    if where == "v":
        v[1, 1234] = bad
    else:
        w[1234] = bad
    got = qdd.qdd_cdot_multi(c, torch.from_numpy(v).cuda(), torch.from_numpy(w).cuda()).cpu().numpy()
    assert np.isfinite(got[0]) == (where == "v") and not np.isfinite(got[1]) and np.isfinite(got[2]) == (where == "v")
