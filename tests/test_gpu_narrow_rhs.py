"""Refined solves with few right-hand sides, at the widths where the residual kernel changes (1, 2 to 4, 5 to 16, more)
and with several nodes: (A - zeta M) X = R on the interior-first ordering against the dense pencil, scaled
residual within 1e-14 (FP64 refinement: a few units of rounding of the residual's own evaluation)."""
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
@pytest.mark.parametrize("name", ["q1_2d_24", "q1_2d_33_p9", "q1_3d_12"])
def test_widths(R, name, precision):
    w = I.workload(name)
    h = R.rfdd_setup(w.A, w.M, w.part, w.p, R.rfdd_default_options(precision=precision))
    z, wt = R.rfdd_quadrature(w.alpha, w.beta, w.n_nodes)
    R.rfdd_factor(h, z, wt)
    _, perm, _ = R.rfdd_layout(h)
    A = w.A.to_scipy()[perm][:, perm]
    M = w.M.to_scipy()[perm][:, perm]
    g = np.random.default_rng(1)
    for b in (1, 2, 3, 4, 5, 15, 16, 17, 33):
        l = b % w.n_nodes
        B = g.standard_normal((w.n, b)) + 1j * g.standard_normal((w.n, b))
        X = R.rfdd_shifted_solve(h, l, 2, 0, B)
        K = A - z[l] * M
        res = np.linalg.norm(K @ X - B) / (abs(K).sum(1).max() * np.linalg.norm(X) + np.linalg.norm(B))
        assert res <= 1e-14, (b, l, res)
