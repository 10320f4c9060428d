"""Tridiagonalisation by one cooperative launch, through the eigenvalue count: batches of blocks of
uneven order (subdomain blocks and the larger interface block) against the closed-form count."""
import numpy as np
import pytest

import rfdd_inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["q1_2d_24", "q1_2d_33_p9", "q1_2d_49_p16", "q1_3d_12"])
def test_counts_of_uneven_blocks(name):
    from paper_1711_09487_gb300 import build
    build.build()
    import paper_1711_09487_gb300 as R
    w = I.workload(name)
    h = R.rfdd_setup(w.A, w.M, w.part, w.p, R.rfdd_default_options())
    for sigma in (w.alpha, w.beta):
        assert R.rfdd_inertia(h, sigma) == int(np.count_nonzero(w.exact < sigma))
