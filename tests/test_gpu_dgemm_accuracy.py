"""Digit products at least as accurate as a sum in FP64: operands whose digits all have one sign, so that whatever the
planes leave out adds up over K; small entries beside the largest ones of their rows; and products at the edges of the
read-backs (every 128 terms) and of the shares of a split K, against extended precision.

Bound, entry by entry: k 2^-57 (largest |a| of its row) (largest |b| of its column) + 2^-51 |c|, after column k of A was
divided and row k of B multiplied by the power of two of the column's largest entry.  The operands are integers of 2^-62 of a power of two P at most twice the row's largest entry, rounded to nearest (2^-63 P each), and the planes
left out are below 2^-59.1 P Q a term: 2^-57 of the two largest entries.  2^-51 stands for the roundings of the two
64-bit sums, of their sum and of alpha and beta."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _check(R, A, B, rows, cols):
    """A (m x k) B (k x n) at the given rows and columns."""
    C = R.rfdd_dgemm(A, B, np.zeros((A.shape[0], B.shape[1])))
    al, bl = A[rows].astype(np.longdouble), B[:, cols].astype(np.longdouble)
    want = np.stack([(al[i][:, None] * bl).sum(0) for i in range(len(rows))])
    k = A.shape[1]
    top = np.abs(A).max(0)
    p2 = 2.0 ** np.floor(np.log2(np.where(top > 0, top, 1.0)))
    bound = (k * 2.0 ** -57 * np.abs(A[rows] / p2).max(1)[:, None] * np.abs(B[:, cols] * p2[:, None]).max(0)[None, :]
             + 2.0 ** -51 * np.abs(want))
    err = np.abs(C[np.ix_(rows, cols)] - want)
    assert np.all(err <= bound), float((err / bound).max())


def _one_sign(g, shape):
    """1 + a fraction whose every base-128 and base-256 digit is large: bits 0111111 repeated, a few of them random."""
    frac = sum(63 * 2.0 ** (-7 * i) for i in range(1, 8))
    return 1.0 + frac / 2 + g.integers(0, 64, shape) * 2.0 ** -52


@pytest.mark.parametrize("k", [1000, 4096, 20000])
def test_digits_of_one_sign(R, k):
    g = np.random.default_rng(k)
    A, B = _one_sign(g, (130, k)), _one_sign(g, (k, 520))
    _check(R, A, B, np.arange(0, 130, 13), np.arange(0, 520, 31))


@pytest.mark.parametrize("k", [127, 128, 129, 255, 511, 512, 513, 640, 30000, 30001])
def test_read_back_edges(R, k):
    g = np.random.default_rng(k)
    m, n = (900, 600) if k < 1000 else (70, 67)
    A, B = g.standard_normal((m, k)), g.standard_normal((k, n))
    _check(R, A, B, np.r_[0, 1, m // 2, m - 1], np.arange(0, n, 7))


@pytest.mark.parametrize("below", [2, 9, 10, 20, 40, 52])
def test_entries_below_the_largest_of_their_row(R, below):
    """Every row and column has an entry 2^below above the others, each at a place of its own."""
    g = np.random.default_rng(below)
    k = 3000
    A, B = g.standard_normal((200, k)), g.standard_normal((k, 200))
    A[np.arange(200), np.arange(200)] *= 2.0 ** below
    B[500 + np.arange(200), np.arange(200)] *= 2.0 ** below
    _check(R, A, B, np.arange(0, 200, 17), np.arange(0, 200, 11))


@pytest.mark.parametrize("ta,tb", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("span", [1, 30, 400])
def test_grading_along_the_sum_changes_no_bit(R, ta, tb, span):
    """op(A) D^-1 times D op(B), D powers of two that span 2 * span binary orders: the product of A and B, bit by bit."""
    g = np.random.default_rng(span)
    m, n, k = 190, 270, 1500
    A, B = g.standard_normal((m, k)), g.standard_normal((k, n))
    A[:, 7] = 0.0
    B[11] = 0.0
    d = 2.0 ** g.integers(-span, span + 1, k)
    Ad, Bd = A / d, B * d[:, None]
    st = lambda X, t: np.ascontiguousarray(X.T if t else X)
    C0 = np.zeros((m, n))
    got = R.rfdd_dgemm(st(Ad, ta), st(Bd, tb), C0, ta=ta, tb=tb)
    np.testing.assert_array_equal(got, R.rfdd_dgemm(st(A, ta), st(B, tb), C0, ta=ta, tb=tb))
    _check(R, A, B, np.arange(0, m, 19), np.arange(0, n, 23))


def test_infinities_meet_zero_and_graded_terms(R):
    """Infinities and NaN keep to their row and column, whatever the terms they stand in are scaled by."""
    g = np.random.default_rng(3)
    A, B = g.standard_normal((160, 3000)), g.standard_normal((3000, 150))
    ref = R.rfdd_dgemm(A, B, np.zeros((160, 150)))
    A[5, 7], A[9, 1], B[20, 3] = np.inf, np.nan, -np.inf
    A[:, 20] = 0.0
    B[7] *= 1e-250
    A[:, 7] *= 1e250
    C = R.rfdd_dgemm(A, B, np.zeros((160, 150)))
    rows, cols = np.delete(np.arange(160), [5, 9]), np.delete(np.arange(150), [3])
    assert not np.isfinite(C[[5, 9]]).any() and not np.isfinite(C[:, 3]).any()
    assert np.isfinite(C[np.ix_(rows, cols)]).all()
    assert np.abs(C - ref)[np.ix_(rows, cols)].max() <= 2 * np.abs(ref).max()  # column 20 left the sums, nothing else
