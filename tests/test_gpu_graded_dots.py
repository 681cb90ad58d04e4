"""Multi-dots of vectors whose elements differ widely in size.

Reference: exact rational arithmetic on the elements that matter (few here).
The bound is FP64's own: at most 8 roundings of 2^-53 per tile of four elements
on sums of at most sum |v||w|, and the additions of a thread's chain (n over
the number of threads), of the warp and of the blocks: 2^-53 (64 + n / 25600).
"""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_1502_04025_gb300 import qdd

    c = qdd.qdd_create(0, 0)
    yield torch, qdd, c
    qdd.qdd_destroy(c)


def exact(v, w):
    """<v, w> and the sums of the magnitudes of its real and imaginary products, exactly."""
    re = im = sre = sim = Fraction(0)
    for k in np.flatnonzero((v != 0) & (w != 0)):
        ax, ay, bx, by = (Fraction(float(t)) for t in (v[k].real, v[k].imag, w[k].real, w[k].imag))
        re += ax * bx + ay * by
        im += ax * by - ay * bx
        sre += abs(ax * bx) + abs(ay * by)
        sim += abs(ax * by) + abs(ay * bx)
    return re, im, sre, sim


def check(torch, qdd, c, vs, w):
    n = w.size
    vd, wd = torch.from_numpy(np.stack(vs)).cuda(), torch.from_numpy(w).cuda()
    want = [exact(v, w) for v in vs]
    unit = Fraction(2) ** -53 * (64 + n // 25600)
    for got in (qdd.qdd_cdot_multi(c, vd, wd), qdd.qdd_cdot_multi_noalloc(vd, wd)):
        for z, (re, im, sre, sim) in zip(got.cpu().numpy(), want):
            assert abs(Fraction(float(z.real)) - re) <= unit * sre
            assert abs(Fraction(float(z.imag)) - im) <= unit * sim


@pytest.mark.parametrize("n", [600000, 1600000])
@pytest.mark.parametrize("small", [1e-3, 1e-12, 1e-17, 1e-120])
def test_point_sink_on_a_decayed_vector(env, n, small):
    """A unit vector at a place where w is small: the result is that one product."""
    torch, qdd, c = env
    rng = np.random.default_rng(7)
    w = rng.standard_normal((n, 2)).view(np.complex128)[:, 0]
    places = rng.integers(0, n, 5)
    w[places] *= small
    vs = []
    for k in places:
        v = np.zeros(n, np.complex128)
        v[k] = 1.0 + 0.5j
        vs.append(v)
    check(torch, qdd, c, vs, w)


@pytest.mark.parametrize("nvec", [1, 3, 8])
@pytest.mark.parametrize("decades", [1, 2, 5, 12, 20])
def test_opposite_decays(env, nvec, decades):
    """v decays where w grows: every product is of one size, far below the largest elements of both."""
    torch, qdd, c = env
    rng = np.random.default_rng(8)
    n = 700001
    # a few thousand elements spread over all threads' tiles, the rest zero
    at = np.sort(rng.choice(n, 20000, replace=False))
    grade = 10.0 ** rng.uniform(-decades, 0, at.size)
    w = np.zeros(n, np.complex128)
    w[at] = rng.standard_normal((at.size, 2)).view(np.complex128)[:, 0] * grade
    vs = []
    for _ in range(nvec):
        v = np.zeros(n, np.complex128)
        v[at] = rng.standard_normal((at.size, 2)).view(np.complex128)[:, 0] / grade
        vs.append(v)
    check(torch, qdd, c, vs, w)


@pytest.mark.parametrize("small", [0.0, 1e-4, 1e-10, 1e-20])
def test_nearly_real_vectors(env, small):
    """The imaginary part of the result is a sum of small products of its own."""
    torch, qdd, c = env
    rng = np.random.default_rng(9)
    n = 500000
    mask = rng.uniform(size=n) < 0.05
    mk = lambda: (rng.standard_normal(n) + 1j * small * rng.standard_normal(n)) * mask
    check(torch, qdd, c, [mk() for _ in range(3)], mk())


@pytest.mark.parametrize("tiles", [1, 2, 3])
@pytest.mark.parametrize("extra", [-1, 0, 1, 300, 40000])
@pytest.mark.parametrize("nvec", [1, 5, 8, 9, 17])
def test_lengths_around_whole_tiles(env, tiles, extra, nvec):
    """Small integers at every place: the sums are exact in every form, whatever the tiling (7 elements a thread
    and pass, 2 blocks of 256 threads per SM), so that one element left out or taken twice shows."""
    torch, qdd, c = env
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    n = 2 * nsm * 256 * 7 * tiles + extra
    g = torch.Generator(device="cuda").manual_seed(3)
    v = torch.randint(-8, 9, (nvec, n, 2), generator=g, device="cuda").double()
    w = torch.randint(-8, 9, (n, 2), generator=g, device="cuda").double()
    v, w = torch.view_as_complex(v), torch.view_as_complex(w)
    re = (v.real * w.real + v.imag * w.imag).sum(1)
    im = (v.real * w.imag - v.imag * w.real).sum(1)
    for got in (qdd.qdd_cdot_multi(c, v, w), qdd.qdd_cdot_multi_noalloc(v, w)):
        got = torch.as_tensor(got).cuda()
        assert torch.equal(got.real, re) and torch.equal(got.imag, im)
