"""Eigenvalues and eigenvectors of the dense symmetric solver at the sizes where the lane-parallel
kernels change shape: around whole warps of eigenvalues, the smallest orders, very large and very
small scales, and spectra that mix isolated eigenvalues with clusters.  Tolerances are those of the
LAPACK comparison: 1e-12 of the norm (order x machine epsilon with two decades of room)."""
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


def _matrix(n, lam, seed):
    Q, _ = np.linalg.qr(np.random.default_rng(seed).standard_normal((n, n)))
    H = (Q * lam) @ Q.T
    return 0.5 * (H + H.T)


@pytest.mark.parametrize("scale", [1.0, 1e100, 1e-100])
@pytest.mark.parametrize("n", [1, 2, 3, 9, 31, 32, 33, 65, 257])
def test_orders_and_scales(R, n, scale):
    _check(R, scale * _matrix(n, np.cumsum(0.5 + np.random.default_rng(n).random(n)), n))


@pytest.mark.parametrize("n", [37, 130])
def test_isolated_and_clustered_together(R, n):
    lam = np.concatenate([np.full(5, 2.0), 3.0 + np.arange(n - 8), np.full(3, -1.0)])
    _check(R, _matrix(n, lam, 2 * n))
