"""Batches too small to fill the GPU, whose products take smaller blocks of rows (down to 512), at the edges of those
blocks and of the staged form (12288 rows).

Tolerance: A is diagonally dominant by 2 with ||A|| <= 9, and the solver stops on the recursive residual; in at most 60
iterations the true one differs from it by less than 60 * 8 u * ||A|| ||x|| <= 1e-12 ||b||. A matrix gives the same bits
in a batch of its own and among others: its sums run over 256 rows at a time whatever the blocks are."""
import numpy as np
import pytest
import scipy.sparse as sp

from gpu_helpers import lib, need_gpu, to_dev, torch

pytestmark = pytest.mark.gpu


def _matrix(n, seed):
    rng = np.random.default_rng(seed)
    A = sp.diags([-1.0 - 0.5 * rng.random(n - 1), np.full(n, 5.5), -np.ones(n - 1)], (-1, 0, 1), shape=(n, n))
    for o in (-7, -3, 3, 7):
        A = A + sp.diags([np.full(n - abs(o), 0.1)], (o,), shape=(n, n))
    return sp.csc_matrix(A), rng.standard_normal(n)


@pytest.mark.parametrize("n", [300, 511, 512, 513, 1025, 2047, 2049, 5000, 12287, 12288, 12289, 13313, 20001])
def test_one_matrix(n):
    need_gpu()
    sai = lib()
    A, b = _matrix(n, n)
    dA, bd = to_dev(A), torch.as_tensor(b, device="cuda")
    xs, per, rep = sai.solve_batched([dA], [bd], eps=1e-10, maxit=60)
    assert rep["status"] == sai.SAI_OK and per[0]["rr"] < 1e-10
    assert np.linalg.norm(b - A @ xs[0].cpu().numpy()) <= (1e-10 + 1e-12) * np.linalg.norm(b)
    others = [_matrix(m, m) for m in (40000, 41000, 42000, 12000, 11000, 10000, 9000) * 10]  # enough for whole blocks
    As, bs = [dA] + [to_dev(a) for a, _ in others], [bd] + [torch.as_tensor(v, device="cuda") for _, v in others]
    many, _, _ = sai.solve_batched(As, bs, eps=1e-10, maxit=60)
    assert torch.equal(many[0], xs[0])
