"""Block GMRES's update in its two forms, on both sides of the orders at which the second is taken (256 rows per SM in
FP32, 640 in FP64, 384 in FP64 with at most four columns), with the block sizes at the ends of its specialisations; restart
4, so that several cycles run.

Tolerance: the true residuals are the stop tests at the restarts; with ||A|| <= 6 and ||x|| <= ||b|| / 2 the computed and
the true ones differ by less than 60 * 8 u * ||A|| ||x|| <= 1e-12 ||b||."""
import numpy as np
import pytest
import scipy.sparse as sp

from gpu_helpers import lib, need_gpu, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_sm,k,precision", [(256, 1, 1), (256, 11, 1), (256, 32, 1), (384, 4, 0), (640, 5, 0), (640, 12, 0)])
@pytest.mark.parametrize("past", [-1, 0, 1, 200])
def test_update_forms(per_sm, k, precision, past):
    need_gpu()
    sai = lib()
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + past
    rng = np.random.default_rng(n + k)
    A = sp.csc_matrix(sp.diags([-1.0 - 0.5 * rng.random(n - 1), np.full(n, 4.5), -np.ones(n - 1)], (-1, 0, 1)))
    h = sai.split(to_dev(A), abs_tau=float("inf"))
    P = sai.precond_from_csc(to_dev(sp.csc_matrix(sp.diags(1.0 / A.diagonal()))))
    B = rng.standard_normal((n, k))
    norms = np.linalg.norm(B, axis=0)
    X, it, stt, st = sai.krylov_solve(h, P, torch.as_tensor(B, device="cuda"), list(1e-10 * norms), method=sai.BGMRES,
                                      maxit=200, restart=4, precision=precision)
    assert st == sai.SAI_OK and stt == [0] * k
    R = np.linalg.norm(B - A @ X.cpu().numpy(), axis=0)
    assert np.all(R <= (1e-10 + 1e-12) * norms), R / norms
