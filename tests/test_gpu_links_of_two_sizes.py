"""FP64 and DF64 operators on links that are not SU(3) and differ in size.

Against the oracle with a componentwise bound: each output component is a sum of
fewer than 64 products, each rounded a handful of times, so the error of both
sides together is at most 64 units of 2^-53 of the sum of the products'
magnitudes (|A||x| + kappa sum |U||h|), however small that is against the largest
link or spinor of the field.
"""
import numpy as np
import pytest

from paper_1502_04025_gb300 import inputs

pytestmark = pytest.mark.gpu

L, DOM, KAPPA = (8, 8, 8, 8), (4, 4, 4, 4), 0.1355


@pytest.fixture(scope="module")
def env():
    from paper_1502_04025_gb300 import qdd

    c = qdd.qdd_create(0, 0)
    yield qdd, c
    qdd.qdd_destroy(c)


def magnitudes(L, U, A, kappa, x):
    """Per output component, the sum of the moduli of the products it is made of."""
    R = tuple(reversed(L))
    U, A = np.abs(U).reshape(R + (4, 3, 3)), np.abs(A).reshape(R + (12, 12))
    x = x.reshape(R + (4, 3))
    out = np.einsum("...ij,...j->...i", A, np.abs(x).reshape(R + (12,))).reshape(R + (4, 3))
    low = {0: lambda l: -1j * l[..., ::-1, :], 1: lambda l: np.stack([-l[..., 1, :], l[..., 0, :]], -2),
           2: lambda l: np.stack([-1j * l[..., 0, :], 1j * l[..., 1, :]], -2), 3: lambda l: l}
    for mu in range(4):
        for back in (0, 1):
            xn = np.roll(x, 1 if back else -1, 3 - mu)
            h = np.abs(xn[..., :2, :] + (1 if back else -1) * low[mu](xn[..., 2:, :]))
            u = U[..., mu, :, :]
            if back:
                u = np.roll(np.swapaxes(u, -1, -2), 1, 3 - mu)
            w = kappa * np.einsum("...ab,...sb->...sa", u, h)
            out[..., :2, :] += w
            out[..., 2:, :] += w[..., ::-1, :] if mu < 2 else w
    return out.reshape(-1, 4, 3)


@pytest.mark.parametrize("prec", ["f64", "df64"])
@pytest.mark.parametrize("size", [2.0 ** 3, 2.0 ** 20, 2.0 ** 40, 2.0 ** 61, 2.0 ** -40, 0.0])
@pytest.mark.parametrize("base", [1.0, 0.3])
def test_one_link_of_another_size(env, ora, prec, size, base):
    """One link `size` times as large as the others, which no site away from it may notice."""
    qdd, c = env
    U = inputs.gauge_field(L, 0.7, 1003) * base
    U = U.reshape(-1, 4, 3, 3)
    U[1234, 2] *= size
    x = inputs.gaussian_source(L, 2003)
    A = ora.clover(L, U, 0.0, KAPPA)  # A = 1
    g = qdd.qdd_create_gauge_field(c, L, DOM, U)
    qdd.qdd_set_clover(g, 0.0, KAPPA)
    got, want = qdd.qdd_apply_D(g, x, prec), ora.apply_D(L, U, A, KAPPA, x)
    qdd.qdd_destroy_gauge(g)
    err, mag = np.abs(got - want).reshape(-1, 4, 3), magnitudes(L, U, A, KAPPA, x)
    assert (err <= 64 * 2.0 ** -53 * mag).all(), (err / mag).max()
