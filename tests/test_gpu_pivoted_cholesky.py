"""Rayleigh-Ritz on bases with linearly dependent columns, through the steps that call the pivoted Cholesky:
orders below and above the number of CTAs, full rank and deficient.  The Ritz values of a basis that
spans the same space must not depend on how it was built (redundant columns dropped): the whole solve with a
deep, nearly dependent basis (psi = 5) and with a shallow one (psi = 1) returns the closed-form pairs."""
import numpy as np
import pytest

import rfdd_inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_1711_09487_gb300 import build
    build.build()
    import paper_1711_09487_gb300 as pkg
    pkg.load()
    return pkg


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("psi,nev_b", [(1, 1), (1, 20), (5, 100)])
@pytest.mark.parametrize("name", ["q1_2d_24", "q1_3d_12", "fd5_32"])
def test_dependent_and_full_rank_bases(R, name, psi, nev_b, precision):
    w = I.workload(name)
    rule = R.RFDD_GAUSS_LEGENDRE if w.rule == "gauss_legendre" else R.RFDD_MIDPOINT
    ev, X, rs, info = R.solve(w.A, w.M, w.part, w.p, w.alpha, w.beta, w.n_nodes, psi=psi, nev_b=nev_b,
                              precision=precision, quad_rule=rule)
    ex = w.exact[(w.exact > w.alpha) & (w.exact < w.beta)]
    assert len(ev) == len(ex) and np.abs(ev - ex).max() <= 1e-9 * ex.max() and rs.max() <= 1e-10
    kz = w.p * nev_b + 2 * psi * info["mu"]
    assert 0 < info["k"] <= kz
    M = w.M.to_scipy()
    assert np.abs(X.T @ (M @ X) - np.eye(len(ev))).max() <= 1e-9
