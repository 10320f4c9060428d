"""The scaled 16-bit split of the tensor-core GEMM: sizes at the edges of its tiles (MMA columns in
steps of 16, packed blocks of 64, narrow and wide tiles, K chunks of the packing) and rows and columns
of very different magnitude, which each carry a scale of their own.

Bound: every entry within 2e-6 k (largest of its row of A) (largest of its column of B) of the FP64
product, the FP32-level bound of the unscaled products (22-bit operands: 2^-22 per product, and the
FP32 accumulation of 2k terms), row by row and column by column; a scale that is wrong or lost shows
as an error of the order of the row itself."""
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


def _run(R, m, n, k, er, ec, engine=1, seed=0):
    g = np.random.default_rng(seed + m + 7 * n + 11 * k)
    A = g.standard_normal((m, k)) + 1j * g.standard_normal((m, k))
    B = g.standard_normal((k, n)) + 1j * g.standard_normal((k, n))
    A = (A * 2.0 ** g.integers(-er, er + 1, (m, 1))).astype(np.complex64)
    B = (B * 2.0 ** g.integers(-ec, ec + 1, (1, n))).astype(np.complex64)
    C0 = np.zeros((m, n), np.complex64)
    C = R.rfdd_cgemm(A, B, C0, -1.0, 1.0, engine)
    want = -(A.astype(np.complex128) @ B.astype(np.complex128))
    scale = np.abs(A).max(1, keepdims=True).astype(float) * np.abs(B).max(0, keepdims=True).astype(float) * k
    assert np.all(np.abs(C - want) <= 2e-6 * scale)


@pytest.mark.parametrize("n", [1, 7, 8, 9, 31, 32, 33, 96, 127, 128, 129, 257])
@pytest.mark.parametrize("k", [1, 31, 32, 33, 255, 256, 257, 600])
def test_tile_edges(R, n, k):
    _run(R, 130, n, k, 0, 0)


@pytest.mark.parametrize("engine", [1, 2, 3])
@pytest.mark.parametrize("er,ec", [(20, 0), (0, 20), (40, 40), (55, 5)])
def test_rows_and_columns_of_different_magnitude(R, er, ec, engine):
    _run(R, 300, 280, 300, er, ec, engine)


def test_zero_rows_and_columns_and_small_entries(R):
    g = np.random.default_rng(3)
    A = g.standard_normal((140, 70)).astype(np.complex64)
    B = g.standard_normal((70, 90)).astype(np.complex64)
    A[5] = 0
    B[:, 17] = 0
    A[7] *= np.float32(1e-37)
    C = R.rfdd_cgemm(A, B, np.zeros((140, 90), np.complex64), 1.0, 0.0, 1)
    want = A.astype(np.complex128) @ B.astype(np.complex128)
    assert np.all(C[5] == 0) and np.all(C[:, 17] == 0)
    assert np.abs(C[7] - want[7]).max() <= 2e-6 * 70 * np.abs(A[7]).max() * np.abs(B).max()
    # an entry far below the largest of its row keeps its own leading bits down to 2^-39 of that one
    A = np.zeros((1, 2), np.complex64)
    A[0] = [1.0, 2.0 ** -20]
    B = np.array([[0.0], [1.0]], np.complex64)
    C = R.rfdd_cgemm(A, B, np.zeros((1, 1), np.complex64), 1.0, 0.0, 1)
    assert abs(C[0, 0] - 2.0 ** -20) <= 2.0 ** -39


def test_infinities_and_nan_stay_in_their_rows(R):
    g = np.random.default_rng(4)
    A = g.standard_normal((66, 40)).astype(np.complex64)
    B = g.standard_normal((40, 70)).astype(np.complex64)
    A[3, 2] = np.inf
    A[9, 1] = np.nan
    C = R.rfdd_cgemm(A, B, np.zeros((66, 70), np.complex64), 1.0, 0.0, 1)
    bad = ~np.isfinite(C.real) | ~np.isfinite(C.imag)
    assert bad[3].all() and bad[9].all() and not np.delete(bad, [3, 9], 0).any()
