"""The clover term's inverses where the blocks are far from the identity."""
import numpy as np
import pytest

from paper_1502_04025_gb300 import inputs

pytestmark = pytest.mark.gpu

L, DOM = (8, 8, 8, 8), (4, 4, 4, 4)


@pytest.fixture(scope="module")
def env():
    from paper_1502_04025_gb300 import qdd

    c = qdd.qdd_create(0, 0)
    yield qdd, c
    qdd.qdd_destroy(c)


@pytest.mark.parametrize("kc", [0.2, 0.6, 1.0, 2.0, 5.0, 30.0])
def test_inverses_as_good_as_with_pivoting(env, kc):
    """kappa c_sw up to values where A's diagonal is no larger than the rest of a block.

    Gauss-Jordan with partial pivoting leaves a residual A A^-1 - 1 of a few n^2 units times the growth
    of a 6x6 elimination (below 8 here) times |A||A^-1|: 64 * 6 units of 2^-53, in the largest norm.
    """
    qdd, c = env
    U = inputs.gauge_field(L, 0.7, 1003)
    g = qdd.qdd_create_gauge_field(c, L, DOM, U)
    V = int(np.prod(L))
    qdd.qdd_set_clover(g, kc / 0.125, 0.125)
    A = qdd.qdd_get_clover(g, V, 0).reshape(V, 2, 6, 6)
    S = qdd.qdd_get_clover(g, V, 1).reshape(V, 2, 6, 6)
    qdd.qdd_destroy_gauge(g)
    n = np.arange(V)
    odd = (n % 8 + n // 8 % 8 + n // 64 % 8 + n // 512) & 1 == 1
    a, s = A[odd].astype(np.clongdouble), S[odd].astype(np.clongdouble)
    res = np.abs(np.einsum("nbij,nbjk->nbik", a, s) - np.eye(6)).sum(-1).max(-1)
    size = np.abs(a).sum(-1).max(-1) * np.abs(s).sum(-1).max(-1)
    assert (res <= 64 * 6 * 2.0 ** -53 * size).all(), (res / size).max() * 2.0 ** 53


@pytest.mark.parametrize("kc", [0.2, 0.4, 0.6, 1.0, 2.0, 5.0, 30.0])
def test_inverse_errors_are_those_of_pivoting(env, ora, kc):
    """Forward errors over the condition number, against the oracle's inverse (Gauss-Jordan, partial pivoting) of
    the same blocks; the largest of 4096 blocks within a factor 4, which covers the scatter of maxima."""
    qdd, c = env
    U = inputs.gauge_field(L, 0.7, 1003)
    g = qdd.qdd_create_gauge_field(c, L, DOM, U)
    V = int(np.prod(L))
    qdd.qdd_set_clover(g, kc / 0.125, 0.125)
    A = qdd.qdd_get_clover(g, V, 0).reshape(V, 2, 6, 6)
    S = qdd.qdd_get_clover(g, V, 1).reshape(V, 2, 6, 6)
    qdd.qdd_destroy_gauge(g)
    full = np.zeros((V, 12, 12), np.complex128)
    full[:, :6, :6], full[:, 6:, 6:] = A[:, 0], A[:, 1]
    inv = ora.invert_clover(L, full)
    n = np.arange(V)
    odd = (n % 8 + n // 8 % 8 + n // 64 % 8 + n // 512) & 1 == 1
    a, gpu = A[odd].reshape(-1, 6, 6), S[odd].reshape(-1, 6, 6)
    ref = np.stack([inv[odd][:, :6, :6], inv[odd][:, 6:, 6:]], 1).reshape(-1, 6, 6)
    x = np.linalg.inv(a).astype(np.clongdouble)
    ax = a.astype(np.clongdouble)
    for _ in range(3):  # Newton's iteration in extended precision
        x = 2 * x - np.einsum("nij,njk,nkl->nil", x, ax, x)
    cond = np.abs(ax).sum(-1).max(-1) * np.abs(x).sum(-1).max(-1) * np.abs(x).max((-1, -2))
    err = lambda y: float((np.abs(y - x).max((-1, -2)) / cond).max() * 2.0 ** 53)
    assert err(gpu) <= 4 * err(ref), (err(gpu), err(ref))
