"""The Krylov vector kernels at the edges of their row chunks.

The vector kernels take rows in chunks of 512 (below 16384 rows) or 2048, each
thread two pairs of neighbouring rows per 512; a system's sums are formed in an
order that depends on n alone. Checked on a nonsymmetric tridiagonal matrix with
M = diag(A)^-1: every system meets its threshold on the true residual, and
solved on its own it gives the same bits.

Tolerance: the solvers stop on the recursive (BiCGStab, CGS, BiCG) or estimated
(GMRES) residual; with ||A|| <= 6, ||x|| <= ||b|| / 2 (diagonal dominance by 2)
and at most 60 iterations the true residual differs from it by less than
60 * 8 u * ||A|| ||x|| <= 1e-12 ||b||.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from gpu_helpers import lib, need_gpu, to_dev, torch

pytestmark = pytest.mark.gpu

METHODS = ("bicgstab", "cgs", "bicg", "gmres")


def _system(n, k, seed):
    rng = np.random.default_rng(seed)
    A = sp.diags([-1.0 - 0.5 * rng.random(max(n - 1, 0)), np.full(n, 4.5), -1.0 * np.ones(max(n - 1, 0))], (-1, 0, 1),
                 shape=(n, n), format="csc")
    A.indptr, A.indices = A.indptr.astype(np.int64), A.indices.astype(np.int32)
    M = sp.csc_matrix(sp.diags(1.0 / A.diagonal()))
    M.indptr, M.indices = M.indptr.astype(np.int64), M.indices.astype(np.int32)
    return A, M, rng.standard_normal((n, k))


@pytest.mark.parametrize("n", [1, 2, 3, 511, 512, 513, 1537, 16383, 16384, 16385, 18433])
@pytest.mark.parametrize("method", METHODS)
def test_vector_kernels_at_chunk_edges(n, method):
    need_gpu()
    sai = lib()
    k = 5
    A, M, B = _system(n, k, n)
    h = sai.split(to_dev(A), abs_tau=float("inf"))
    P = sai.precond_from_csc(to_dev(M))
    Bd = torch.as_tensor(B, device="cuda")
    norms = np.linalg.norm(B, axis=0)
    thr = [1e-6 * norms[0], 1e-9 * norms[1], 2.0 * norms[2], 1e-10 * norms[3], 1e-3 * norms[4]]
    m = sai._METHOD[method]
    X, it, stt, st = sai.krylov_solve(h, P, Bd, thr, method=m, maxit=60, restart=30)
    assert st == sai.SAI_OK and stt == [0] * k
    R = np.linalg.norm(B - A @ X.cpu().numpy(), axis=0)
    assert np.all(R <= np.asarray(thr) + 1e-12 * norms), (R, thr)
    assert it[2] == 0  # its threshold is above ||b||
    for c in range(k):
        xc, itc, _, _ = sai.krylov_solve(h, P, Bd[:, c:c + 1].contiguous(), thr[c:c + 1], method=m, maxit=60,
                                         restart=30)
        assert itc[0] == it[c]
        assert torch.equal(xc[:, 0], X[:, c]), (method, n, c)


@pytest.mark.parametrize("n,k", [(63, 2), (511, 5), (513, 1), (1000, 9), (2049, 13), (3001, 17), (1537, 25), (4099, 32)])
@pytest.mark.parametrize("precision", [0, 1])
def test_block_gmres_block_sizes(n, k, precision):
    """Block sizes around the kernels' specialisations (4, 8, 12, 16, 24, 32) and row counts around their tiles
    (chunks of 512 rows, tiles of 64); restart 4, so that several cycles run. Tolerance as above."""
    need_gpu()
    sai = lib()
    A, M, B = _system(n, k, 7 * n + k)
    h = sai.split(to_dev(A), abs_tau=float("inf"))
    P = sai.precond_from_csc(to_dev(M))
    norms = np.linalg.norm(B, axis=0)
    thr = list(1e-10 * norms)
    X, it, stt, st = sai.krylov_solve(h, P, torch.as_tensor(B, device="cuda"), thr, method=sai.BGMRES, maxit=200,
                                      restart=4, precision=precision)
    assert st == sai.SAI_OK and stt == [0] * k
    R = np.linalg.norm(B - A @ X.cpu().numpy(), axis=0)
    assert np.all(R <= np.asarray(thr) + 1e-12 * norms), (R, thr)
