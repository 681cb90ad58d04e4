"""The clover term on weak fields, whose field strength is far below the entries of the leaves it is a difference of."""
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


@pytest.mark.parametrize("eps", [0.5, 1e-2, 1e-4, 1e-8])
def test_weak_fields_keep_their_field_strength(env, eps):
    """A - 1 is linear in a small field strength: as good relative to itself as FP64's sums.

    F is a difference of leaves whose entries differ from the unit matrix by about eps; FP64 products of three
    matrices round entries of that size by 2^-53 eps, and the diagonal's by 2^-53 of their imaginary part: 2^-40
    of the largest entry of A - 1 leaves room for the cancellation (F is of order eps, leaf entries of a few eps).
    Reference: the leaves in extended precision.
    """
    qdd, c = env
    U = inputs.gauge_field(L, eps, 1003)
    g = qdd.qdd_create_gauge_field(c, L, DOM, U)
    V = int(np.prod(L))
    csw, kappa = 1.0, 0.125
    qdd.qdd_set_clover(g, csw, kappa)
    A = qdd.qdd_get_clover(g, V, 0).reshape(V, 2, 6, 6)
    qdd.qdd_destroy_gauge(g)
    # the upper triangle's entries come from F's off-diagonal parts without the 1 of the diagonal
    F = strengths(U)
    G3 = [-F[0, 1] + se * F[2, 3] for se in (1, -1)]
    G1 = [-F[1, 2] + se * F[0, 3] for se in (1, -1)]
    G2 = [F[0, 2] + se * F[1, 3] for se in (1, -1)]
    for ch in range(2):
        want = np.zeros((V, 6, 6), np.clongdouble)
        kc = np.longdouble(csw) * np.longdouble(kappa)
        want[:, :3, :3] = kc * 1j * G3[ch]
        want[:, 3:, 3:] = -kc * 1j * G3[ch]
        want[:, :3, 3:] = kc * 1j * (G1[ch] - 1j * G2[ch])
        iu = np.triu_indices(6, 1)
        w = want[:, iu[0], iu[1]]
        err = np.abs(A[:, ch][:, iu[0], iu[1]] - w)
        assert (err.max() <= 2.0 ** -40 * np.abs(w).max()), err.max() / np.abs(w).max()


def strengths(U):
    U = U.reshape(tuple(reversed(L)) + (4, 3, 3)).astype(np.clongdouble)
    mul = lambda a, b: np.einsum("...ij,...jk->...ik", a, b)
    dag = lambda a: np.conj(np.swapaxes(a, -1, -2))
    sh = lambda a, mu, d: np.roll(a, -d, 3 - mu)
    F = {}
    for mu in range(4):
        for nu in range(mu + 1, 4):
            um, un = U[..., mu, :, :], U[..., nu, :, :]
            q = mul(mul(um, sh(un, mu, 1)), dag(mul(un, sh(um, nu, 1))))
            a, b = sh(um, mu, -1), sh(un, mu, -1)  # links at n - mu
            q = q + mul(mul(un, dag(sh(a, nu, 1))), mul(dag(b), a))
            e, f = sh(sh(um, mu, -1), nu, -1), sh(sh(un, mu, -1), nu, -1)
            q = q + mul(mul(dag(a), dag(f)), mul(e, sh(un, nu, -1)))
            h = sh(un, nu, -1)
            q = q + mul(mul(dag(h), sh(um, nu, -1)), mul(sh(sh(un, nu, -1), mu, 1), dag(um)))
            f8 = (q - dag(q)) / 8
            tr = np.trace(f8, axis1=-2, axis2=-1) / 3
            f8 = f8 - tr[..., None, None] * np.eye(3)
            F[mu, nu] = f8.reshape(-1, 3, 3)
    return F
