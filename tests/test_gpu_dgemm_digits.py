"""FP64 products by digit planes on the tensor cores (the large products of rfdd_dgemm engine 1): tile and
pass edges, transposes, symmetric products, leading dimensions, and rows and columns of very
different magnitude, against products in extended precision.

Bound, entry by entry: k 2^-48 (largest |a| of its row) (largest |b| of its column) + 2^-52 |c|.  Every operand is
a 55-bit integer times a power of two at most twice its row's largest entry (error 2^-54 of that
power), and the digit products left out are below 2^-51 of the product of the two powers, per term."""
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


def _check(R, A, B, C0, alpha, beta, ta=False, tb=False, sym=False, seed=0):
    got = R.rfdd_dgemm(A, B, C0, alpha, beta, ta=ta, tb=tb, sym=sym)
    a, b = (A.T if ta else A), (B.T if tb else B)
    m, k = a.shape
    n = b.shape[1]
    rows = np.unique(np.r_[0, m - 1, np.random.default_rng(seed).integers(0, m, 6)])
    cols = np.unique(np.r_[0, n - 1, np.random.default_rng(seed + 1).integers(0, n, 40)])
    al, bl = a[rows].astype(np.longdouble), b[:, cols].astype(np.longdouble)
    prod = np.stack([(al[i][:, None] * bl).sum(0) for i in range(len(rows))])
    want = beta * C0[np.ix_(rows, cols)].astype(np.longdouble) + alpha * prod
    bound = (abs(alpha) * k * 2.0 ** -48 * np.abs(a[rows]).max(1)[:, None] * np.abs(b[:, cols]).max(0)[None, :]
             + 2.0 ** -51 * (np.abs(want) + np.abs(beta * C0[np.ix_(rows, cols)]) + np.abs(alpha * prod)))
    err = np.abs(got[np.ix_(rows, cols)] - want)
    assert np.all(err <= bound), float((err / bound).max())
    return got


@pytest.mark.parametrize("ta,tb", [(False, False), (True, False), (False, True), (True, True)])
@pytest.mark.parametrize("m,n,k", [(128, 64, 8192), (129, 65, 8193), (700, 130, 1111), (48, 2000, 700),
                                   (300, 320, 48 * 20), (1000, 1003, 65)])
def test_shapes(R, m, n, k, ta, tb):
    g = np.random.default_rng(m + n + k)
    A = g.standard_normal((k, m) if ta else (m, k))
    B = g.standard_normal((n, k) if tb else (k, n))
    C0 = g.standard_normal((m, n))
    _check(R, A, B, C0, 1.0, 0.0, ta, tb)
    _check(R, A, B, C0, -0.75, 1.5, ta, tb)


@pytest.mark.parametrize("n,k", [(63, 20000), (64, 20000), (129, 8000), (390, 1000), (771, 5003)])
def test_symmetric(R, n, k):
    g = np.random.default_rng(n)
    Y = g.standard_normal((k, n))
    P = Y * (0.5 + g.random((k, 1)))
    G = _check(R, Y, P, np.zeros((n, n)), 1.0, 0.0, ta=True, sym=True)
    np.testing.assert_array_equal(G, G.T)


def test_many_passes_over_k(R):
    """digits of 2000 + 2000 vectors fill the workspace at about 23 000 terms: three passes"""
    g = np.random.default_rng(9)
    Y = g.standard_normal((50001, 2000))
    _check(R, Y, Y, np.zeros((2000, 2000)), 1.0, 0.0, ta=True, sym=True)


@pytest.mark.parametrize("span", [30, 300])
def test_scales(R, span):
    g = np.random.default_rng(span)
    A = g.standard_normal((200, 2000)) * 10.0 ** g.integers(-span // 2, span // 2, (200, 1))
    B = g.standard_normal((2000, 190)) * 10.0 ** g.integers(-span // 3, span // 3, (1, 190))
    _check(R, A, B, np.zeros((200, 190)), 1.0, 0.0)


def test_zeros_infinities_nan(R):
    g = np.random.default_rng(5)
    A, B = g.standard_normal((160, 3000)), g.standard_normal((3000, 150))
    A[3] = 0.0
    A[5, 7] = np.inf
    A[9, 1] = np.nan
    B[:, 11] = 0.0
    C = R.rfdd_dgemm(A, B, np.zeros((160, 150)))
    assert np.all(C[3] == 0.0)
    assert not np.isfinite(C[5]).any() and not np.isfinite(C[9]).any()
    ok = np.delete(np.arange(160), [5, 9])
    assert np.isfinite(C[ok]).all() and np.all(C[ok][:, 11] == 0.0)
