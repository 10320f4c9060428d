"""Householder vectors that are kept unnormalised: graded matrices, whose reflectors differ in size by orders of
magnitude, and matrices far from one, where the reflector is scaled, against LAPACK within 1e-12 of the norm,
the bound of the solver at every order."""
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


@pytest.mark.parametrize("decades", [0, 6, -6, 14])
@pytest.mark.parametrize("scale", [1.0, 1e-14, 1e15, 1e-120, 1e120])
@pytest.mark.parametrize("n", [3, 64, 130, 640])
def test_graded(R, n, scale, decades):
    g = np.random.default_rng(n)
    A = g.standard_normal((n, n))
    d = 10.0 ** np.linspace(0.0, -abs(decades), n)[:: -1 if decades < 0 else 1]
    H = (A + A.T) * d[:, None] * d[None, :]
    ref = np.linalg.eigvalsh(H)
    nrm = np.abs(ref).max()
    ev, V = R.rfdd_sym_eig(scale * H)
    np.testing.assert_allclose(ev / scale / nrm, ref / nrm, atol=1e-12)
    np.testing.assert_allclose(V @ V.T, np.eye(n), atol=1e-12)
    assert np.abs((H / nrm) @ V.T - V.T * (ev / scale / nrm)).max() <= 1e-12
