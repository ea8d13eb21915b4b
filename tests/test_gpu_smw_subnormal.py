"""Pivots below the smallest normal number: their reciprocals overflow, so multipliers and unknowns must come from
divisions there, as they do for every other pivot up to rounding.

V^T W = -I + D with D a cyclic shift times values of 1e-310, so that I + V^T W = D has zeros on its diagonal and subnormal
pivots after interchanges; yhat(J) of order 1e-300 keeps z = D^-1 yhat(J) near 1e10. A z_t is one division, exact up to
half a unit roundoff u; x = yhat - W z adds s products, |W| < 0.5 sqrt(1/s) * 5: the sums differ by less than
(s + 2) u * s * 2.5 / sqrt(s) * max|z| <= 1e-12 max|z| for s <= 300.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from gpu_helpers import lib, need_gpu, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s", [2, 3, 33, 160, 161, 300])
def test_subnormal_pivots(s):
    need_gpu()
    sai = lib()
    rng = np.random.default_rng(s)
    n = 3 * s + 40
    J = np.sort(rng.choice(n, size=s, replace=False))
    rows = np.concatenate([(np.arange(4) + j + 1) % n for j in J])
    A = sp.csc_matrix(sp.identity(n) + sp.coo_matrix((np.ones(rows.size), (rows, np.repeat(J, 4))), shape=(n, n)))
    Y = rng.standard_normal((n, s + 1))
    Y[:, 1:] *= 0.5 / np.sqrt(s)
    shift = (np.arange(s) + 1) % s
    d = 1e-310 * rng.uniform(1.0, 2.0, s)
    Y[J, 1:] = -np.eye(s)
    Y[J, 1 + shift] = d  # row i of D: d_i in column i + 1
    Y[J, 0] = 1e-300 * rng.standard_normal(s)
    z = np.empty(s)
    z[shift] = Y[J, 0] / d
    x = Y[:, 0] - Y[:, 1:] @ z
    h = sai.split(to_dev(A), abs_tau=3.0, p_keep=1)
    assert h.s == s
    xs, c = sai.smw_recover(h, torch.as_tensor(Y, device="cuda"))
    np.testing.assert_allclose(xs.cpu().numpy(), x, rtol=0, atol=1e-12 * np.abs(z).max())
    assert c == pytest.approx(np.linalg.norm(z), rel=1e-12)
