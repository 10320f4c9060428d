"""Entries far below the largest of their row (of A) or column (of B) in the 16-bit split of the tensor-core GEMM: full
mantissas at ratios on both sides of 2^-15, where the lower half starts to lose bits, each brought out alone by a zero
against the large entry.

Bound: 2^-22 of the entry or 2^-38 of the largest one, whichever is more (both halves are rounded to nearest; the
lower one has a spacing of 2^-24 under a largest entry of 2^13 and more)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("engine", [1, 2, 3])
@pytest.mark.parametrize("side", ["row of A", "column of B"])
@pytest.mark.parametrize("below", [0, 8, 13, 14, 15, 16, 17, 20, 24, 30, 37, 41])
def test_small_entries(R, below, side, engine):
    g = np.random.default_rng(below)
    m, k = 150, 40
    x = ((1 + g.random((m, k))) + 1j * (1 + g.random((m, k)))) * 2.0 ** -below
    X = x.astype(np.complex64)
    X[:, 0] = 1.5 - 1j
    E = np.eye(k, dtype=np.complex64)
    E[0, 0] = 0.0  # the large entry meets only zeros
    A, B = (X, E) if side == "row of A" else (E.T.copy(), X.T.copy())
    C = R.rfdd_cgemm(A, B, np.zeros((A.shape[0], B.shape[1]), np.complex64), 1.0, 0.0, engine)
    got = C if side == "row of A" else C.T
    want = X.astype(np.complex128) * (np.arange(k) > 0)
    for part in (np.real, np.imag):
        err, val = np.abs(part(got).astype(float) - part(want)), np.abs(part(want))
        assert np.all(err <= np.maximum(2.0 ** -22 * val, 2.0 ** -38 * 1.5))
