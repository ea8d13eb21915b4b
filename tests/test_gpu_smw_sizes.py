"""The SMW recovery at the edges of its eliminations: one block in shared memory
(s <= 160), in place (the allocation-free call, s <= 256), the blocked LU with
its panels and triangular solves over a cluster (s > 160; panels of 16 columns,
blocks of 32 rows), each against LAPACK on the same Y.

I + V^T W has a random W(J,:) of 2-norm about 1, so its condition number stays
below about 1e3 and both solutions are within 1e3 * s * u < 1e-9 of each other.
"""
import ctypes as C

import numpy as np
import pytest
import scipy.sparse as sp

from gpu_helpers import lib, need_gpu, to_dev, torch

pytestmark = pytest.mark.gpu


def _case(s, seed):
    rng = np.random.default_rng(seed)
    n = 3 * s + 40
    J = np.sort(rng.choice(n, size=s, replace=False))
    A = sp.lil_matrix((n, n))
    A.setdiag(1.0)
    A = sp.csc_matrix(A)
    rows = np.concatenate([(np.arange(4) + j + 1) % n for j in J])
    A = sp.csc_matrix(A + sp.coo_matrix((np.ones(rows.size), (rows, np.repeat(J, 4))), shape=(n, n)))
    Y = rng.standard_normal((n, s + 1))
    Y[:, 1:] *= 0.5 / np.sqrt(s)
    W = Y[:, 1:]
    z = np.linalg.solve(np.eye(s) + W[J, :], Y[J, 0])
    return A, J, Y, Y[:, 0] - W @ z, np.linalg.norm(z)


@pytest.mark.parametrize("s", [1, 2, 31, 32, 33, 159, 160, 161, 176, 256, 257, 300, 1029])
def test_recovery_matches_lapack(s):
    need_gpu()
    sai = lib()
    A, J, Y, xo, co = _case(s, s)
    h = sai.split(to_dev(A), abs_tau=3.0, p_keep=1)
    assert h.s == s
    x, c = sai.smw_recover(h, torch.as_tensor(Y, device="cuda"))
    np.testing.assert_allclose(x.cpu().numpy(), xo, rtol=0, atol=1e-9 * np.abs(xo).max())
    assert c == pytest.approx(co, rel=1e-9)
    if s > 256:
        return
    L = sai.load()
    Yd = torch.as_tensor(Y, device="cuda")
    Jd = torch.as_tensor(J.astype(np.int32), device="cuda")
    xd = torch.empty(A.shape[0], dtype=torch.float64, device="cuda")
    cc = C.c_double()
    f = L.sai_smw_recover_noalloc
    f.argtypes = [C.c_int32, C.c_int32, C.c_void_p, C.c_void_p, C.c_void_p, C.POINTER(C.c_double), C.c_void_p]
    st = f(A.shape[0], s, Jd.data_ptr(), Yd.data_ptr(), xd.data_ptr(), C.byref(cc),
           torch.cuda.current_stream().cuda_stream)
    assert st == sai.SAI_OK
    np.testing.assert_allclose(xd.cpu().numpy(), xo, rtol=0, atol=1e-9 * np.abs(xo).max())


@pytest.mark.parametrize("s", [5, 170, 300])
def test_a_zero_pivot_is_singular(s):
    """W(J,:) = -I + a strictly lower triangular part: I + W(J,:) has a zero first row."""
    need_gpu()
    sai = lib()
    A, J, Y, _, _ = _case(s, s + 1)
    Y[J, 1:] = -np.eye(s) + np.tril(0.1 * np.ones((s, s)), -1)
    h = sai.split(to_dev(A), abs_tau=3.0, p_keep=1)
    with pytest.raises(sai.SaiError) as e:
        sai.smw_recover(h, torch.as_tensor(Y, device="cuda"))
    assert e.value.status == sai.SAI_SINGULAR
