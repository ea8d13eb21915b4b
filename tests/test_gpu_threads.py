"""Calls from two host threads at once, each on a stream of its own.

The kernels with dynamic shared memory take as much as their problem needs; two threads with problems of different size
must not see each other's limits, and calls that capture graphs must not capture on one stream. Every call must succeed and give, bit for bit, what it gives alone: no sum of these
solvers depends on what else runs.
"""
import threading

import numpy as np
import pytest
import scipy.sparse as sp

from gpu_helpers import lib, need_gpu, to_dev, torch

pytestmark = pytest.mark.gpu


def _recovery(sai, s):
    rng = np.random.default_rng(s)
    n = 3 * s + 40
    J = np.sort(rng.choice(n, size=s, replace=False))
    rows = np.concatenate([(np.arange(4) + j + 1) % n for j in J])
    A = sp.csc_matrix(sp.identity(n) + sp.coo_matrix((np.ones(rows.size), (rows, np.repeat(J, 4))), shape=(n, n)))
    Y = rng.standard_normal((n, s + 1))
    Y[:, 1:] *= 0.5 / np.sqrt(s)
    h = sai.split(to_dev(A), abs_tau=3.0, p_keep=1)
    Yd = torch.as_tensor(Y, device="cuda")
    return lambda: sai.smw_recover(h, Yd)[0]


def _krylov(sai, n, k, **kw):
    rng = np.random.default_rng(n)
    A = sp.csc_matrix(sp.diags([np.full(n - 1, -1.5), np.full(n, 4.5), -np.ones(n - 1)], (-1, 0, 1)))
    h = sai.split(to_dev(A), abs_tau=float("inf"))
    P = sai.build_spai(h)
    B = rng.standard_normal((n, k))
    Bd = torch.as_tensor(B, device="cuda")
    thr = list(1e-10 * np.linalg.norm(B, axis=0))
    return lambda: sai.krylov_solve(h, P, Bd, thr, **kw)[0]


def _batch(sai, orders):
    rng = np.random.default_rng(sum(orders))
    As, bs = [], []
    for n in orders:
        d = [np.full(n - abs(o), 0.1) for o in (-7, -3, 3, 7)]
        A = sp.diags([np.full(n - 1, -1.5), np.full(n, 5.5), -np.ones(n - 1)] + d, (-1, 0, 1, -7, -3, 3, 7))
        As.append(to_dev(sp.csc_matrix(A)))
        bs.append(torch.as_tensor(rng.standard_normal(n), device="cuda"))
    return lambda: torch.cat(sai.solve_batched(As, bs, eps=1e-10)[0])


def _pair(kind):
    sai = lib()
    if kind == "recovery":
        return _recovery(sai, 700), _recovery(sai, 2000)
    if kind == "bicgstab":
        return _krylov(sai, 2000, 4), _krylov(sai, 20000, 4)
    if kind == "batch":
        return _batch(sai, (700, 900)), _batch(sai, (12000, 12100))
    kw = dict(method=sai.GMRES, restart=20)
    if kind == "gmres_graphs":  # beyond the cluster form: both capture their steps
        return _krylov(sai, 50000, 3, **kw), _krylov(sai, 20000, 5, **kw)
    return _krylov(sai, 500, 3, **kw), _krylov(sai, 10000, 3, **kw)


@pytest.mark.parametrize("kind", ["recovery", "bicgstab", "gmres", "gmres_graphs", "batch"])
def test_two_threads_with_problems_of_different_size(kind):
    need_gpu()
    calls = _pair(kind)
    alone = [f() for f in calls]
    torch.cuda.synchronize()
    failed = []
    start = threading.Barrier(2)

    def work(f, want):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                # the update's copy ring has more chances beside another thread's kernels
                for _ in range(1000 if kind == "gmres_graphs" else 60):
                    got = f()
                    if not torch.equal(got, want):
                        failed.append("other bits")
        except Exception as e:  # noqa: BLE001
            failed.append(repr(e))

    threads = [threading.Thread(target=work, args=a) for a in zip(calls, alone)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed[:3]
