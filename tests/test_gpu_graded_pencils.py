"""Pencils whose rows differ by many orders: D A D x = lambda D M D x for D of powers of two has the spectrum of (A, M)
exactly, while the entries along the rows of its factors and bases are graded.  The plain FP64 path has to reach the
residual target of 1e-10 and the closed-form eigenvalues at every grading at which FP64 multiply-adds do (up to 2^7; at
2^8 their residuals are at the target)."""
import numpy as np
import pytest
import scipy.sparse as sp

import rfdd_inputs as I

pytestmark = pytest.mark.gpu


def _csr(S):
    S = sp.csr_matrix(S)
    S.sort_indices()
    return I.Csr(S.shape[0], S.indptr.astype(np.int64), S.indices.astype(np.int32), S.data.copy())


def _graded(w, e, seed):
    D = sp.diags(2.0 ** np.random.default_rng(seed).integers(-e, e + 1, w.A.n))
    return _csr(D @ w.A.to_scipy() @ D), _csr(D @ w.M.to_scipy() @ D)


@pytest.mark.parametrize("e,seeds", [(2, (0, 1)), (3, (0, 1)), (5, (0, 1, 2)), (7, (0, 1, 2, 4))])
def test_fp64_solves(R, e, seeds):
    w = I.workload("q1_3d_12")
    ex = w.exact[(w.exact > w.alpha) & (w.exact < w.beta)]
    for seed in seeds:
        A, M = _graded(w, e, seed)
        ev, X, rs, info = R.solve(A, M, w.part, w.p, w.alpha, w.beta, w.n_nodes, precision=R.RFDD_FP64)
        assert len(ev) == len(ex) and np.abs(ev - ex).max() <= 1e-10 * ex.max() and rs.max() <= 1e-10, (seed, rs.max())
