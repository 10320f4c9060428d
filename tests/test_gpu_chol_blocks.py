"""Block orthonormalisation (Cholesky-QR) at the block widths where its kernels change: below, at and
above whole warps of columns, the largest width kept in shared memory (160) and one more.  The
Krylov basis must be orthonormal to 1e-12, and V_j of the same widths must span the same filter: the
solve returns every eigenpair of the closed form."""
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
@pytest.mark.parametrize("block", [1, 7, 8, 9, 31, 32, 33, 64])
def test_krylov_basis_is_orthonormal(R, block, precision):
    w = I.workload("q1_3d_12")
    h = R.rfdd_setup(w.A, w.M, w.part, w.p, R.rfdd_default_options(block=block, precision=precision))
    z, wt = R.rfdd_quadrature(w.alpha, w.beta, w.n_nodes)
    R.rfdd_factor(h, z, wt)
    Q, tr = R.rfdd_lanczos(h)
    assert np.abs(Q.T @ Q - np.eye(Q.shape[1])).max() <= 1e-12
    assert np.all(np.isfinite(tr))


@pytest.mark.parametrize("nev_b", [1, 27, 133, 134, 140])
def test_vj_widths(R, nev_b):
    w = I.workload("q1_2d_33_p9")
    ev, X, rs, info = R.solve(w.A, w.M, w.part, w.p, w.alpha, w.beta, w.n_nodes, nev_b=nev_b)
    ex = w.exact[(w.exact > w.alpha) & (w.exact < w.beta)]
    assert len(ev) == len(ex) and np.abs(ev - ex).max() <= 1e-9 * ex.max() and rs.max() <= 1e-10
