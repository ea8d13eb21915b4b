"""A handle destroyed while work on it is in flight, and while another stream is in capture.

A handle's buffers come from a pool, so memory freed too early is handed to the next handle and a copy still running
reads that one's values; and a destruction may neither fail nor break a capture that runs meanwhile. Values are copied,
so every comparison is exact.
"""
import threading

import numpy as np
import pytest
import scipy.sparse as sp

from gpu_helpers import lib, need_gpu, to_dev, torch

pytestmark = pytest.mark.gpu


def _precond(sai, n, value):
    M = sp.csc_matrix(sp.diags([np.full(n, value), np.full(n - 1, 0.5 * value)], (0, 1), shape=(n, n)))
    return sai.precond_from_csc(to_dev(M))


def _copy_out(sai, P, v, stream):
    null = None
    st = sai.load().sai_precond_copy_out(P._h, null, null, v.data_ptr(), null, null, null, stream.cuda_stream)
    assert st == sai.SAI_OK


@pytest.mark.parametrize("nstreams", [1, 3, 20])  # 20: more streams than a handle keeps events for
@pytest.mark.parametrize("capture", [False, True])
@pytest.mark.parametrize("own", [False, True])  # created on the legacy stream, or on one of the caller's
def test_destroyed_with_copies_in_flight(nstreams, capture, own):
    need_gpu()
    with torch.cuda.stream(torch.cuda.Stream() if own else torch.cuda.default_stream()):
        _destroyed_with_copies_in_flight(nstreams, capture)


def _destroyed_with_copies_in_flight(nstreams, capture):
    sai = lib()
    n = 100000
    streams = [torch.cuda.Stream() for _ in range(nstreams)]
    a = torch.zeros(1024, device="cuda")
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        a.add_(0.0)
    torch.cuda.synchronize()
    for rep in range(3):
        P = _precond(sai, n, 1.0 + rep)
        out = [torch.zeros(P.nnz, dtype=torch.float64, device="cuda") for _ in streams]
        torch.cuda.synchronize()
        for s, v in zip(streams, out):
            with torch.cuda.stream(s):
                torch.cuda._sleep(20000000)  # some ten milliseconds
            _copy_out(sai, P, v, s)
        holder = [P]
        del P
        if capture:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=side, capture_error_mode="thread_local"):
                a.add_(1.0)
                t = threading.Thread(target=holder.clear)
                t.start()
                t.join()
                a.add_(1.0)
            before = float(a[0])
            g.replay()
            assert float(a[0]) == before + 2.0
        else:
            holder.clear()
        other = [_precond(sai, n, -7.0) for _ in range(4)]  # takes what was freed
        torch.cuda.synchronize()
        want = np.empty(2 * n - 1)
        want[0::2], want[1::2] = 1.0 + rep, 0.5 * (1.0 + rep)
        for v in out:
            got = v.cpu().numpy()
            assert np.array_equal(np.sort(got), np.sort(want))
        del other


def test_split_destroyed_behind_a_solve_on_another_stream():
    """Handles used on one stream and destroyed from a thread that works on another; the answers stay right."""
    need_gpu()
    sai = lib()
    n = 3000
    A = sp.csc_matrix(sp.diags([-np.ones(n - 1), np.full(n, 4.0), -np.ones(n - 1)], (-1, 0, 1)))
    dA = to_dev(A)
    b = np.random.default_rng(0).standard_normal(n)
    bd = torch.as_tensor(b, device="cuda")
    torch.cuda.synchronize()
    for _ in range(4):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            h = sai.split(dA)
            P = sai.build_spai(h)
            x, _, rep = sai.solve_with(dA, h, P, bd, eps=1e-10)
        with torch.cuda.stream(torch.cuda.Stream()):
            del h, P
            sai.split(dA)
        s.synchronize()
        assert rep["status"] == sai.SAI_OK
        assert np.linalg.norm(b - A @ x.cpu().numpy()) <= (1e-10 + 1e-12) * np.linalg.norm(b)


def test_memory_of_destroyed_handles_goes_back():
    """Sixteen handles of 120 MB in buffers of at most 32 MB: all but what the handles' pool keeps (256 MB; 512 MB allow
    for its granularity) is free again after a synchronisation."""
    need_gpu()
    sai = lib()
    n = 2000000
    M = to_dev(sp.identity(n, format="csc"))
    sai.precond_from_csc(M)  # the calls' own scratch
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    handles = [sai.precond_from_csc(M) for _ in range(16)]
    held = before - torch.cuda.mem_get_info()[0]
    assert held > 1500 << 20
    del handles
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] < 512 << 20
