"""The batched products at the edges of their blocks: 2048 rows per block, rows sorted by length within it, vectors of up
to 12288 rows staged in shared memory. One batch holds orders on both sides of each limit, with rows of up to 700
entries among rows of three or seven.

Tolerance: A is diagonally dominant by 2 with ||A|| <= 9, and the solver stops on the recursive residual; in at most 60
iterations the true one differs from it by less than 60 * 8 u * ||A|| ||x|| <= 1e-12 ||b||."""
import numpy as np
import pytest
import scipy.sparse as sp

from gpu_helpers import lib, need_gpu, to_dev, torch

pytestmark = pytest.mark.gpu


def _matrix(n, rng, bands):
    A = sp.diags([-1.0 - 0.5 * rng.random(n), np.full(n, 5.5), -np.ones(n)], (-1, 0, 1), shape=(n, n))
    for o in (-7, -3, 3, 7) if bands else ():  # rows long enough for staging
        if abs(o) < n:
            A = A + sp.diags([np.full(n - abs(o), 0.1)], (o,), shape=(n, n))
    rows, cols = [], []
    for i in {0, n // 2, n - 1}:
        length = min(n, int(rng.integers(1, 701)))
        rows.append(np.full(length, i))
        cols.append(rng.permutation(n)[:length])
    val = np.concatenate([0.3 / r.size * rng.uniform(-1, 1, r.size) for r in rows])
    A = sp.csc_matrix(A + sp.coo_matrix((val, (np.concatenate(rows), np.concatenate(cols))), shape=(n, n)))
    A.sort_indices()
    A.indptr, A.indices = A.indptr.astype(np.int64), A.indices.astype(np.int32)
    return A


@pytest.mark.parametrize("bands", [False, True])
@pytest.mark.parametrize("orders", [(1, 2, 31, 33), (255, 257, 2047, 2048, 2049, 6145), (24575, 24576, 24577, 700, 40001), (12287, 12288),
                                    (12289, 14337), (12288, 12289, 64)])
@pytest.mark.parametrize("kw", [dict(sai="spai", delta=0.4, mn=2, max_aug=5), dict(sai="psai", delta=0.4, tol=1e-3,
                                                                                  tol_mode=1, lmax=3)])
def test_batch_at_block_edges(orders, kw, bands):
    need_gpu()
    sai = lib()
    rng = np.random.default_rng(sum(orders))
    As = [_matrix(n, rng, bands) for n in orders]
    bs = [rng.standard_normal(n) for n in orders]
    xs, per, rep = sai.solve_batched([to_dev(A) for A in As], [torch.as_tensor(b, device="cuda") for b in bs],
                                     eps=1e-10, maxit=60, **kw)
    assert rep["status"] == sai.SAI_OK
    for A, b, x, r in zip(As, bs, xs, per):
        assert r["status"] == sai.SAI_OK and r["rr"] < 1e-10
        assert np.linalg.norm(b - A @ x.cpu().numpy()) <= (1e-10 + 1e-12) * np.linalg.norm(b)
