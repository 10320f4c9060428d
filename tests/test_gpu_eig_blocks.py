"""Back-transformation in blocks (orders from 512 on) of the dense symmetric eigensolver: orders around whole
blocks of 128 reflectors, trivial reflectors (matrices already tridiagonal, block diagonal or diagonal), against
LAPACK within 1e-12 of the norm, the bound of the solver at every order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_1711_09487_gb300 import build
    build.build()
    import paper_1711_09487_gb300 as pkg
    pkg.load()
    return pkg


def _check(R, H):
    ev, V = R.rfdd_sym_eig(H)
    ref = np.linalg.eigvalsh(H)
    nrm = np.abs(ref).max()
    np.testing.assert_allclose(ev / nrm, ref / nrm, atol=1e-12)
    np.testing.assert_allclose(V @ V.T, np.eye(len(H)), atol=1e-12)
    assert np.abs((H / nrm) @ V.T - V.T * (ev / nrm)).max() <= 1e-12


@pytest.mark.parametrize("n", [511, 512, 513, 514, 515, 640, 642, 643, 900])
def test_orders(R, n):
    g = np.random.default_rng(n)
    Q, _ = np.linalg.qr(g.standard_normal((n, n)))
    H = (Q * np.cumsum(0.5 + g.random(n))) @ Q.T
    _check(R, 0.5 * (H + H.T))


@pytest.mark.parametrize("kind", ["diagonal", "tridiagonal", "blocks"])
def test_trivial_reflectors(R, kind):
    n = 600
    g = np.random.default_rng(7)
    H = np.diag(np.cumsum(0.5 + g.random(n)))
    if kind == "tridiagonal":
        e = 0.3 * g.random(n - 1)
        H += np.diag(e, 1) + np.diag(e, -1)
    if kind == "blocks":
        A = g.standard_normal((150, 150))
        H[200:350, 200:350] += 0.01 * (A + A.T)
    _check(R, H)
