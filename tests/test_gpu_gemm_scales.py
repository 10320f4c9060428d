"""Row and column scales of the tensor-core GEMM whose product leaves the range of a float although the results do
not: sums that are normal FP32 numbers from rows and columns near 2^-62, the same brought up by a large alpha,
huge rows against huge columns without common entries (exactly zero), and scales on different sides of one,
with an alpha that is no power of two among them.

Bound of the sums: 2e-6 k (largest of the row) (largest of the column), that of the GEMM at every scale, and two
steps of the smallest floats."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _rnd(g, m, n, e):
    return ((g.standard_normal((m, n)) + 1j * g.standard_normal((m, n))) * 2.0 ** e).astype(np.complex64)


@pytest.mark.parametrize("engine", [1, 2, 3])
@pytest.mark.parametrize("ea,eb,alpha", [(-62, -62, 1.0), (-110, -13, 1.0), (-62, -61, 2.0 ** 100), (-100, 100, 1.0),
                                         (100, -110, -1.0), (60, 55, 1.0), (-59, -59, 2.0 ** 30),
                                         (110, -120, 1.0), (-120, 110, -0.75), (-100, -22, 0.75), (70, -115, 3e-9)])
@pytest.mark.parametrize("m,n,k", [(5, 3, 2), (300, 281, 96)])
def test_sums_in_range(R, m, n, k, ea, eb, alpha, engine):
    g = np.random.default_rng(m + ea + 200)
    A, B = _rnd(g, m, k, ea), _rnd(g, k, n, eb)
    C = R.rfdd_cgemm(A, B, np.zeros((m, n), np.complex64), alpha, 0.0, engine)
    want = alpha * (A.astype(np.complex128) @ B.astype(np.complex128))
    scale = alpha * k * np.abs(A.astype(np.complex128)).max(1)[:, None] * np.abs(B.astype(np.complex128)).max(0)[None, :]
    assert np.all(np.abs(C - want) <= 2e-6 * np.abs(scale) + 2.0 ** -148)


@pytest.mark.parametrize("engine", [1, 2, 3])
def test_huge_without_common_entries(R, engine):
    A, B = np.zeros((140, 40), np.complex64), np.zeros((40, 70), np.complex64)
    A[:, :20] = 2.0 ** 100
    B[20:] = 2.0 ** 100
    C = R.rfdd_cgemm(A, B, np.zeros((140, 70), np.complex64), 1.0, 0.0, engine)
    assert not C.any()
