"""BiCGStab on right-hand sides far from 1: scaled by a power of two, the systems converge as the unscaled ones do, on
either side of the limit between the cluster form and the kernels for larger orders.

rho = rhat^T r falls towards (eps ||b||)^2, below 2^-1040 for the smallest scale: a subnormal number of some 30 bits whose
reciprocal is not representable. Tolerance: the solver stops on the recursive residual; with ||A|| <= 6 and ||x|| <= ||b|| / 2 the true
one differs from it by less than 1e-12 ||b|| in at most 60 iterations."""
import numpy as np
import pytest
import scipy.sparse as sp

from gpu_helpers import lib, need_gpu, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [-492, -300, 0, 300, 492])
@pytest.mark.parametrize("n", [100, 2000, 20480, 20481])
def test_scaled_right_hand_sides(n, exponent):
    need_gpu()
    sai = lib()
    rng = np.random.default_rng(n)
    A = sp.csc_matrix(sp.diags([-1.0 - 0.5 * rng.random(n - 1), np.full(n, 4.5), -np.ones(n - 1)], (-1, 0, 1)))
    h = sai.split(to_dev(A), abs_tau=float("inf"))
    P = sai.precond_from_csc(to_dev(sp.csc_matrix(sp.diags(1.0 / A.diagonal()))))
    B = rng.standard_normal((n, 3))
    B /= np.linalg.norm(B, axis=0)
    X, it, stt, st = sai.krylov_solve(h, P, torch.as_tensor(np.ldexp(B, exponent), device="cuda"),
                                      [float(np.ldexp(1e-11, exponent))] * 3, maxit=60)
    assert st == sai.SAI_OK and stt == [0] * 3
    R = np.linalg.norm(B - A @ np.ldexp(X.cpu().numpy(), -exponent), axis=0)
    assert np.all(R <= 1e-11 + 1e-12), R
