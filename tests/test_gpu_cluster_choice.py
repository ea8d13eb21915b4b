"""Orders around the limits at which the cluster forms are left: 10240 rows (12288 in refined GMRES) where most entries lie
far from the diagonal (a random permutation of a tridiagonal matrix), 14336 rows for more than 64 systems, 20480
(BiCGStab) and 49152 rows (refined GMRES) for a banded matrix; and the vector kernels of more than 256 systems at the
edges of their row chunks. Each against its true residual, and transposed.

Tolerance: the solvers stop on the recursive (BiCGStab) residual or on the true one (refined GMRES); with ||A|| <= 6 and
||x|| <= ||b|| / 2 the true residual differs from it by less than 60 * 8 u * ||A|| ||x|| <= 1e-12 ||b||."""
import numpy as np
import pytest
import scipy.sparse as sp

from gpu_helpers import lib, need_gpu, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scattered", [False, True])
@pytest.mark.parametrize("n,k,method", [
    (10240, 3, "bicgstab"), (10241, 3, "bicgstab"), (14336, 80, "bicgstab"), (14337, 8, "bicgstab"),
    (14337, 64, "bicgstab"), (14337, 65, "bicgstab"), (20480, 257, "bicgstab"), (9000, 257, "bicgstab"), (511, 300, "bicgstab"),
    (1537, 257, "bicgstab"), (16383, 40, "bicgstab"), (16384, 40, "bicgstab"), (12288, 3, "gmres32"),
    (12289, 3, "gmres32"), (36864, 2, "gmres32"), (36865, 2, "gmres32"), (49152, 2, "gmres32"), (49153, 2, "gmres32"),
    (10240, 5, "gmres"), (10241, 5, "gmres")])
def test_around_the_limits(n, k, method, scattered):
    need_gpu()
    sai = lib()
    rng = np.random.default_rng(n + k)
    A = sp.csc_matrix(sp.diags([-1.0 - 0.5 * rng.random(n - 1), np.full(n, 4.5), -np.ones(n - 1)], (-1, 0, 1)))
    if scattered:
        p = rng.permutation(n)
        A = sp.csc_matrix(A[p][:, p])
    h = sai.split(to_dev(A), abs_tau=float("inf"))
    P = sai.build_spai(h, delta=0.3, mn=3, max_aug=2)
    B = rng.standard_normal((n, k))
    norms = np.linalg.norm(B, axis=0)
    thr = list(norms * 10.0 ** -np.linspace(2, 10, k))
    kw = {"bicgstab": {}, "gmres": dict(method=sai.GMRES, restart=15),
          "gmres32": dict(method=sai.GMRES, restart=15, precision=1)}[method]
    Bd = torch.as_tensor(B, device="cuda")
    for transpose, Aop in ((False, A), (True, A.T)):
        X, it, stt, st = sai.krylov_solve(h, P, Bd, thr, maxit=60, transpose=transpose, **kw)
        assert st == sai.SAI_OK and stt == [0] * k
        R = np.linalg.norm(B - Aop @ X.cpu().numpy(), axis=0)
        assert np.all(R <= np.asarray(thr) + 1e-12 * norms), (R, thr)


@pytest.mark.parametrize("n", [1, 2, 511, 512, 513, 1537, 16383, 16384, 16385])
def test_vector_kernels_of_many_systems(n):
    """More systems than the cluster form takes: BiCGStab's vector kernels at the edges of their chunks of 512 rows (2048
    from 16384 on). 257 and 300 systems give the same bits: a system's sums depend on n alone."""
    need_gpu()
    sai = lib()
    rng = np.random.default_rng(n)
    A = sp.csc_matrix(sp.diags([-1.0 - 0.5 * rng.random(max(n - 1, 0)), np.full(n, 4.5), -np.ones(max(n - 1, 0))],
                               (-1, 0, 1), shape=(n, n)))
    h = sai.split(to_dev(A), abs_tau=float("inf"))
    P = sai.precond_from_csc(to_dev(sp.csc_matrix(sp.diags(1.0 / A.diagonal()))))
    B = rng.standard_normal((n, 300))
    norms = np.linalg.norm(B, axis=0)
    thr = list(norms * 10.0 ** -np.linspace(2, 10, 300))
    thr[3] = 2.0 * norms[3]
    Bd = torch.as_tensor(B, device="cuda")
    X, it, stt, st = sai.krylov_solve(h, P, Bd, thr, maxit=60)
    assert st == sai.SAI_OK and stt == [0] * 300 and it[3] == 0
    R = np.linalg.norm(B - A @ X.cpu().numpy(), axis=0)
    assert np.all(R <= np.asarray(thr) + 1e-12 * norms), (R, thr)
    x, i, _, _ = sai.krylov_solve(h, P, Bd[:, :257].contiguous(), thr[:257], maxit=60)
    assert i == it[:257] and torch.equal(x, X[:, :257])
