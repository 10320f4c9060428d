"""rfdd_cgemm_noalloc takes pointers to floats: operands that start on a 4-byte boundary give the bits of the same
operands on a 16-byte one (the packed values do not depend on how they were read), for each of A, B and C, at the
widths at which rows share a warp of the packing and at tile edges."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _place(torch, X, shift):
    """The floats of X on the device, `shift` floats after a 256-byte boundary."""
    buf = torch.zeros(X.size * 2 + 8, dtype=torch.float32, device="cuda")
    buf[shift:shift + 2 * X.size] = torch.from_numpy(X.view(np.float32).ravel().copy()).cuda()
    return buf, buf.data_ptr() + 4 * shift


@pytest.mark.parametrize("shifts", [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 1), (3, 2, 2)])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (130, 33, 32), (129, 65, 33), (300, 257, 100), (1024, 130, 128)])
def test_four_byte_boundaries(R, m, n, k, shifts):
    import torch
    g = np.random.default_rng(m + n + k)
    cplx = lambda r, c: (g.standard_normal((r, c)) + 1j * g.standard_normal((r, c))).astype(np.complex64)
    A, B, C = cplx(m, k), cplx(k, n), cplx(m, n)
    out = []
    for sh in ((0, 0, 0), shifts):
        bufs = [_place(torch, X, s) for X, s in zip((A, B, C), sh)]
        torch.cuda.synchronize()
        R.rfdd_cgemm_noalloc(m, n, k, bufs[0][1], k, bufs[1][1], n, bufs[2][1], n, -1.0, 1.0)
        got = bufs[2][0].cpu().numpy()
        out.append(got[sh[2]:sh[2] + 2 * m * n].view(np.complex64).reshape(m, n))
        assert not got[:sh[2]].any() and not got[sh[2] + 2 * m * n:].any()
    np.testing.assert_array_equal(out[0], out[1])
    want = C.astype(np.complex128) - A.astype(np.complex128) @ B.astype(np.complex128)
    assert np.abs(out[1] - want).max() <= 2e-6 * k * np.abs(A).max() * np.abs(B).max()
