"""The LM step where the FP32 factor fails and the FP64 factorisation takes over, in the
one-block form (2 n up to 90) and the cluster form, alone and in a batch.

Only baselines between even and odd antennas have data, and the offsets are zero: then
+x for the even and -x for the odd antennas changes no visibility to first order, so the
matrix without its damping is singular twice over and with lambda = 1e-8 has a condition
number of 2e8, while the right-hand side has nothing in those directions.  In FP32 its
last two pivots are rounding noise of either sign.  FP64 leaves 2e8 x 2^-53 x n, below
2e-6 of the step; 1e-5 is asserted."""
import numpy as np
import pytest

from test_gpu_lm import _problem

pytestmark = pytest.mark.gpu

LAM = 1e-8


def _weights(gp):
    import torch
    i, j = np.triu_indices(gp.m.n_ant, 1)
    w = torch.ones(gp.shape, device="cuda")
    w[:, torch.from_numpy((i + j) % 2 == 0).cuda()] = 0.0
    return w


def _opts():
    from paper_1709_08681_gb300 import _abi
    o = _abi.psc_solve_opts_default()
    o.lam0, o.lam_min = LAM, LAM
    return o


def _reference(gp, v, w):
    n = gp.m.n_ant
    _, g, H, X = gp.ctx.psc_residual_grad(np.zeros((n, 2)), v, w, 1e6, cross=True)
    A = np.zeros((n, 2, n, 2))
    k = np.arange(n)
    A[k, 0, k, 0], A[k, 0, k, 1], A[k, 1, k, 0], A[k, 1, k, 1] = H[:, 0], H[:, 1], H[:, 1], H[:, 2]
    i, j = np.triu_indices(n, 1)
    A[i, :, j, :] = X.reshape(-1, 2, 2)
    A[j, :, i, :] = X.reshape(-1, 2, 2).transpose(0, 2, 1)
    A = A.reshape(2 * n, 2 * n)
    A[np.arange(2 * n), np.arange(2 * n)] *= 1.0 + LAM
    scaled = A / np.sqrt(np.outer(np.diag(A), np.diag(A)))
    assert 1e7 < np.linalg.cond(scaled) < 1e10
    return np.linalg.solve(A, -g.reshape(-1)).reshape(n, 2)


@pytest.mark.parametrize("n_ant", [6, 44, 45, 46, 47, 100])
@pytest.mark.parametrize("seed", [3, 4, 5])
def test_step_of_an_ill_conditioned_system(n_ant, seed):
    from paper_1709_08681_gb300 import _abi
    gp, v = _problem(n_ant, seed)
    w = _weights(gp)
    ref = _reference(gp, v, w)
    gp.ctx.psc_lm_begin(np.zeros((n_ant, 2)), _opts())
    gp.ctx.psc_lm_iterate(v, w, 1e6, 2)
    lm, rep = gp.ctx.psc_lm_end()
    assert rep.n_eval == 2
    assert np.max(np.abs(lm - ref)) < 1e-5 * np.max(np.abs(ref))
    other, v2 = _problem(20, seed)                            # the same beside a system of the other form
    b = _abi.Batch([gp.ctx, other.ctx], [v, v2], [w, _weights(other)], [1e6, 1e6])
    b.psc_batch_begin([np.zeros((n_ant, 2)), np.zeros((20, 2))], _opts())
    b.psc_batch_iterate(2)
    lms, _ = b.psc_batch_end()
    b.close()
    assert np.array_equal(lms[0], lm)
