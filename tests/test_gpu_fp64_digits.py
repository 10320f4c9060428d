"""The FP64 factorisations on blocks large enough for the digit products of their updates (several strips,
ragged last panels), real and complex: solves with the factors against the dense shifted blocks, scaled
residual within 1e-13 (the bound of the FP64 solve residuals at every size), and a whole FP64 solve."""
import numpy as np
import pytest

import rfdd_inputs as I
from oracle import rfdd_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    from paper_1711_09487_gb300 import build
    build.build()
    import paper_1711_09487_gb300 as pkg
    pkg.load()
    return pkg


@pytest.mark.parametrize("name", ["q1_2d_64", "q1_3d_16", "q1_2d_49_p16"])
def test_block_solves(R, name):
    w = I.workload(name)
    blk = O.Blocks(w.A.to_scipy(), w.M.to_scipy(), w.part, w.p)
    z, wt = R.rfdd_quadrature(w.alpha, w.beta, w.n_nodes)
    h = R.rfdd_setup(w.A, w.M, w.part, w.p, R.rfdd_default_options(precision=R.RFDD_FP64))
    R.rfdd_factor(h, z, wt)
    g = np.random.default_rng(1)
    for l in (0, w.n_nodes - 1):
        for j in (0, w.p - 1):
            K = blk.B[j] - z[l] * blk.MB[j]
            B = g.standard_normal((K.shape[0], 70)) + 1j * g.standard_normal((K.shape[0], 70))
            X = R.rfdd_shifted_solve(h, l, 0, j, B)
            res = np.linalg.norm(K @ X - B) / (np.linalg.norm(K, 2) * np.linalg.norm(X) + np.linalg.norm(B))
            assert res <= 1e-13, (l, j, res)


def test_fp64_solve_matches_closed_form(R):
    w = I.workload("q1_2d_64")
    ev, X, rs, info = R.solve(w.A, w.M, w.part, w.p, w.alpha, w.beta, w.n_nodes, precision=R.RFDD_FP64)
    ex = w.exact[(w.exact > w.alpha) & (w.exact < w.beta)]
    assert len(ev) == len(ex) and np.abs(ev - ex).max() <= 1e-10 * ex.max() and rs.max() <= 1e-10
    M = w.M.to_scipy()
    assert np.abs(X.T @ (M @ X) - np.eye(len(ev))).max() <= 1e-10
