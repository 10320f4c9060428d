"""The one-launch pivoted Cholesky by itself: factors of full-rank and rank-deficient matrices around the number of
CTAs, more CTAs than the device has room for at once, and a barrier whose wait runs out, which has to come back as an error with nothing indexed by the
pivots that were never chosen.

Bound of the factors: k 2^-50 of the largest entry (k rounding errors of 2^-53 each, times eight)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _gram(k, rank, seed):
    Y = np.random.default_rng(seed).standard_normal((rank, k))
    d = 1.0 / np.sqrt((Y * Y).sum(0))
    return (Y * d).T @ (Y * d)


@pytest.mark.parametrize("k,rank", [(1, 1), (2, 2), (2, 1), (33, 33), (151, 150), (152, 152), (153, 7), (700, 305)])
def test_factor_and_rank(R, k, rank):
    G = _gram(k, rank, k + rank)
    r, perm, U = R.rfdd_pivoted_cholesky(G, 1e-12)
    assert r == rank and len(set(perm.tolist())) == r and perm.min() >= 0 and perm.max() < k
    assert np.abs(U.T @ U - G[np.ix_(perm, perm)]).max() <= k * 2.0 ** -50


def test_no_pivot_above_the_limit(R):
    assert R.rfdd_pivoted_cholesky(np.eye(40), 2.0)[0] == 0


@pytest.mark.parametrize("k", [40, 600])
def test_a_wait_that_runs_out_is_an_error(R, k):
    """One look at the counter instead of millions: the first CTA at the barrier gives up at once."""
    G = _gram(k, k, 1)
    with pytest.raises(R.RfddError) as e:
        R.rfdd_pivoted_cholesky(G, 1e-12, polls=1)
    assert e.value.code == R.RFDD_ECUDA and "timed out" in str(e.value)
    assert R.rfdd_pivoted_cholesky(G, 1e-12)[0] == k  # the next call is unaffected


@pytest.mark.parametrize("ctas", [1, 3, 2000])
def test_number_of_ctas_changes_no_bit(R, ctas):
    """2000 CTAs of this kernel are not resident together: the launch is refused and repeated with fewer."""
    G = _gram(2000, 300, 2)
    ref = R.rfdd_pivoted_cholesky(G, 1e-12)
    got = R.rfdd_pivoted_cholesky(G, 1e-12, ctas=ctas)
    assert got[0] == ref[0]
    np.testing.assert_array_equal(got[1], ref[1])
    np.testing.assert_array_equal(got[2], ref[2])
