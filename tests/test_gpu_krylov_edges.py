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


@pytest.mark.parametrize("n", [64, 65, 2560, 2561, 5121, 10303, 20480, 20481])
@pytest.mark.parametrize("uneven", [False, True])
def test_bicgstab_in_clusters(n, uneven):
    """Orders around the cluster form's blocks (2560 rows; one, two, four or eight of them, more for fewer systems)
    and its limit of 20480; rows of equal length (sliced ELL) and with every 64th row 40 entries longer (CSR). The
    transposed solve too. Tolerance as above (||A|| grows to 7)."""
    need_gpu()
    sai = lib()
    k = 20
    A, M, B = _system(n, k, n + 1)
    if uneven:
        rng = np.random.default_rng(n)
        rows = np.repeat(np.arange(0, n, 64), 40)
        E = sp.coo_matrix((0.01 * rng.standard_normal(rows.size), (rows, rng.integers(0, n, rows.size))), shape=(n, n))
        A = sp.csc_matrix(A + E)
        A.sort_indices()
    h = sai.split(to_dev(A), abs_tau=float("inf"))
    P = sai.precond_from_csc(to_dev(M))
    norms = np.linalg.norm(B, axis=0)
    thr = list(norms * 10.0 ** -np.linspace(2, 10, k))
    thr[3] = 2.0 * norms[3]
    Bd = torch.as_tensor(B, device="cuda")
    for transpose, Aop in ((False, A), (True, A.T)):
        X, it, stt, st = sai.krylov_solve(h, P, Bd, thr, maxit=60, transpose=transpose)
        assert st == sai.SAI_OK and stt == [0] * k and it[3] == 0
        R = np.linalg.norm(B - Aop @ X.cpu().numpy(), axis=0)
        assert np.all(R <= np.asarray(thr) + 1e-12 * norms), (R, thr)
        for c in (0, 7, k - 1):
            xc, itc, _, _ = sai.krylov_solve(h, P, Bd[:, c:c + 1].contiguous(), thr[c:c + 1], maxit=60,
                                             transpose=transpose)
            assert itc[0] == it[c] and torch.equal(xc[:, 0], X[:, c]), (n, c)
    X, it, stt, st = sai.krylov_solve(h, P, Bd, thr, maxit=2)
    assert st == sai.SAI_MAXITER and max(it) == 2 and stt[3] == sai.SAI_OK and stt[k - 1] == sai.SAI_MAXITER


@pytest.mark.parametrize("n,k,m,precision", [
    (64, 1, 1, 0), (65, 3, 7, 1), (129, 40, 127, 0), (1000, 2, 127, 1), (2049, 5, 3, 0), (2304, 200, 20, 1),
    (10240, 4, 30, 0), (10241, 4, 30, 0), (16385, 20, 12, 1), (33333, 3, 30, 1), (49152, 2, 8, 1), (49153, 2, 8, 1)])
@pytest.mark.parametrize("uneven", [False, True])
def test_gmres_in_clusters(n, k, m, precision, uneven):
    """GMRES(m) around the limits of the cluster form (10240 rows in FP64, 49152 in FP32), with restart lengths from 1
    to the largest, one to eight blocks per cluster and more systems than clusters at once; rows of equal length and
    with every 64th row 40 entries longer. Tolerance as above; a system solved alone agrees within the two residuals."""
    need_gpu()
    sai = lib()
    A, M, B = _system(n, k, 3 * n + m)
    if uneven:
        rng = np.random.default_rng(n)
        rows = np.repeat(np.arange(0, n, 64), 40)
        E = sp.coo_matrix((0.01 * rng.standard_normal(rows.size), (rows, rng.integers(0, n, rows.size))), shape=(n, n))
        A = sp.csc_matrix(A + E)
        A.sort_indices()
    h = sai.split(to_dev(A), abs_tau=float("inf"))
    P = sai.precond_from_csc(to_dev(M))
    norms = np.linalg.norm(B, axis=0)
    thr = list(norms * 10.0 ** -np.linspace(3, 10, k))
    thr[0] = 2.0 * norms[0]
    Bd = torch.as_tensor(B, device="cuda")
    kw = dict(method=sai.GMRES, restart=m, maxit=400, precision=precision)
    X, it, stt, st = sai.krylov_solve(h, P, Bd, thr, **kw)
    assert st == sai.SAI_OK and stt == [0] * k and it[0] == 0
    R = np.linalg.norm(B - A @ X.cpu().numpy(), axis=0)
    assert np.all(R <= np.asarray(thr) + 1e-12 * norms), (R, thr)
    c = k - 1
    xc, itc, _, _ = sai.krylov_solve(h, P, Bd[:, c:c + 1].contiguous(), thr[c:c + 1], **kw)
    # the blocks per cluster, and so the order of the sums, depend on k: the two solutions differ by A^-1 times their
    # residuals, ||A^-1|| <= 1/2
    dx = np.linalg.norm((xc[:, 0] - X[:, c]).cpu().numpy())
    assert abs(itc[0] - it[c]) <= 1 and dx <= thr[c] + 1e-12 * norms[c]
    if k > 1:
        X, it, stt, st = sai.krylov_solve(h, P, Bd, thr, **dict(kw, maxit=2))
        assert st == sai.SAI_MAXITER and stt[c] == sai.SAI_MAXITER and it[c] == 2 and stt[0] == sai.SAI_OK


@pytest.mark.parametrize("n,k", [(700, 150), (4999, 20), (20480, 3)])
@pytest.mark.parametrize("method", ["bicgstab", "gmres", "gmres32"])
def test_cluster_rows_sorted_by_length(n, k, method):
    """A few rows far longer than the rest (around the steps of the sort by length: 511, 512, 607, 608 entries, and n),
    in the first, a middle and the last block. Their off-diagonal sums stay below 0.3, so the tolerance above holds."""
    need_gpu()
    sai = lib()
    A, M, B = _system(n, k, n)
    rng = np.random.default_rng(n)
    rows, cols = [], []
    for i, length in zip((0, 1, n // 2, n // 2 + 1, n - 1), (511, 512, 607, 608, n)):
        cols.append(rng.permutation(n)[:length])
        rows.append(np.full(length, i))
    val = np.concatenate([0.3 / r.size * rng.uniform(-1, 1, r.size) for r in rows])
    A = sp.csc_matrix(A + sp.coo_matrix((val, (np.concatenate(rows), np.concatenate(cols))), shape=(n, n)))
    A.sort_indices()
    h = sai.split(to_dev(A), abs_tau=float("inf"))
    P = sai.precond_from_csc(to_dev(M))
    norms = np.linalg.norm(B, axis=0)
    kw = {"bicgstab": {}, "gmres": dict(method=sai.GMRES, restart=20),
          "gmres32": dict(method=sai.GMRES, restart=20, precision=1)}[method]
    for transpose, Aop in ((False, A), (True, A.T)):
        X, it, stt, st = sai.krylov_solve(h, P, torch.as_tensor(B, device="cuda"), list(1e-9 * norms), maxit=100,
                                          transpose=transpose, **kw)
        assert st == sai.SAI_OK and stt == [0] * k
        R = np.linalg.norm(B - Aop @ X.cpu().numpy(), axis=0)
        assert np.all(R <= 1e-9 * norms + 1e-12 * norms), R / norms
