"""The admission estimate against what a solve holds: the high-water mark of the stream-ordered pool over one solve stays
within rfdd_memory_estimate, in FP64 and in mixed precision with either form of the factors, with and without a
memory budget of that size (which bounds the digits of the FP64 products), and the solve still converges."""
import ctypes as C

import numpy as np
import pytest

import rfdd_inputs as I

pytestmark = pytest.mark.gpu

USED_CURRENT, USED_HIGH = 7, 8  # CUmemPool_attribute


class Pool:
    def __init__(self):
        self.cu, self.pool = C.CDLL("libcuda.so.1"), C.c_void_p()
        assert self.cu.cuDeviceGetDefaultMemPool(C.byref(self.pool), 0) == 0

    def get(self, attr):
        v = C.c_uint64()
        assert self.cu.cuMemPoolGetAttribute(self.pool, attr, C.byref(v)) == 0
        return v.value

    def restart(self):
        v = C.c_uint64(0)
        assert self.cu.cuMemPoolSetAttribute(self.pool, USED_HIGH, C.byref(v)) == 0
        return self.get(USED_CURRENT)


@pytest.mark.parametrize("budget", [False, True])
@pytest.mark.parametrize("precision,pack", [(0, -1), (1, 1), (1, 0)])
@pytest.mark.parametrize("name", ["q1_2d_40", "q1_3d_12", "q1_3d_16", "q1_2d_64"])
def test_high_water_mark(R, name, precision, pack, budget):
    w = I.workload(name)
    rule = R.RFDD_GAUSS_LEGENDRE if w.rule == "gauss_legendre" else R.RFDD_MIDPOINT
    opts = dict(precision=precision, pack_factors=pack, quad_rule=rule)
    h = R.rfdd_setup(w.A, w.M, w.part, w.p, R.rfdd_default_options(**opts))
    need = R.rfdd_memory_estimate(h, w.n_nodes, w.expected_nev)
    if budget:
        h = R.rfdd_setup(w.A, w.M, w.part, w.p, R.rfdd_default_options(mem_budget=need, **opts))
    pool = Pool()
    base = pool.restart()
    r = R.rfdd_solve(h, w.alpha, w.beta, w.n_nodes)
    high = pool.get(USED_HIGH) - base
    assert 0.3 * need <= high <= need, (high, need)
    ev = R.rfdd_result_get(r)[0]
    ex = w.exact[(w.exact > w.alpha) & (w.exact < w.beta)]
    assert len(ev) == len(ex) and np.abs(ev - ex).max() <= 1e-9 * ex.max()
