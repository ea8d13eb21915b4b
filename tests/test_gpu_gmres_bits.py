"""A GMRES system gives the same bits and the same step count alone, with a few others and with many: at the edges of the
units that its sums are formed by (128 rows at least; sixteen units from 3585 rows on), of the blocks per cluster and of
the cluster form itself (10240 rows in FP64, 49152 in FP32), with short and long restarts, rows of equal length and with
every 64th row 40 entries longer. Every comparison is exact: no sum may depend on the other systems."""
import numpy as np
import pytest
import scipy.sparse as sp

from gpu_helpers import lib, need_gpu, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("uneven", [False, True])
@pytest.mark.parametrize("n,k,m,precision", [
    (1, 3, 5, 0), (33, 40, 7, 1), (255, 200, 10, 0), (256, 200, 10, 1), (513, 200, 20, 0), (1025, 120, 127, 0),
    (2047, 100, 12, 1), (2049, 80, 30, 0), (3584, 40, 30, 0), (3585, 40, 30, 1), (5000, 256, 10, 0), (6145, 70, 30, 0),
    (10240, 70, 20, 0), (10240, 10, 127, 0), (10241, 9, 20, 0), (12289, 60, 30, 1), (24577, 30, 30, 1),
    (36864, 25, 20, 1), (36864, 3, 127, 1), (36865, 9, 20, 1), (49152, 25, 20, 1), (49152, 3, 127, 1), (49153, 9, 20, 1)])
def test_bits_do_not_depend_on_the_other_systems(n, k, m, precision, uneven):
    need_gpu()
    sai = lib()
    rng = np.random.default_rng(n + m)
    A = sp.diags([-1.0 - 0.5 * rng.random(max(n - 1, 0)), np.full(n, 4.5), -np.ones(max(n - 1, 0))], (-1, 0, 1),
                 shape=(n, n))
    if uneven:
        rows = np.repeat(np.arange(0, n, 64), 40)
        A = A + sp.coo_matrix((0.01 * rng.standard_normal(rows.size), (rows, rng.integers(0, n, rows.size))), shape=(n, n))
    A = sp.csc_matrix(A)
    h = sai.split(to_dev(A), abs_tau=float("inf"))
    P = sai.precond_from_csc(to_dev(sp.csc_matrix(sp.diags(1.0 / A.diagonal()))))
    B = torch.as_tensor(rng.standard_normal((n, k)), device="cuda")
    thr = list(B.norm(dim=0).cpu().numpy() * 10.0 ** -np.linspace(3, 10, k))
    kw = dict(method=sai.GMRES, restart=m, maxit=100, precision=precision)
    X, it, _, _ = sai.krylov_solve(h, P, B, thr, **kw)
    for lo, hi in ((k - 1, k), (0, 2), (k // 3, k // 3 + k // 4 + 1), (0, k - 1)):
        x, i, _, _ = sai.krylov_solve(h, P, B[:, lo:hi].contiguous(), thr[lo:hi], **kw)
        assert i == it[lo:hi]
        assert torch.equal(x, X[:, lo:hi])
