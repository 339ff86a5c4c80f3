"""Two visibilities of a thread, their rows taken two at a time: against the same
context with one visibility a thread (rows one at a time).  Both sum the same taps in
FP32 in another order: a sum of n <= 1000 taps of like size has an expected rounding
error below sqrt(n) 2^-24 = 2e-6 of its norm; 1e-5 bounds the two together.  Apertures
of few and many rows, odd and even, pairs that move little and by some cells, an odd
number of time steps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_grid,nt,span", [(1024, 37, 0.3), (1024, 37, 2.0), (512, 20, 1.0), (360, 33, 0.5), (256, 8, 1.0)])
def test_pair_rows_agree_with_single_rows(n_grid, nt, span):
    import cases
    import torch
    from gpu_cases import GpuProblem
    freqs = tuple(1.2e9 + 0.05e9 * k for k in range(7))
    m, _, lmt, img = cases.problem(("disk", 64, 24.0, n_grid), n_ant=7, n_time=nt, freqs=freqs, extent_m=300.0)
    m.uvw_m = cases.geometry(7, 300.0, nt, span, freqs)[0]
    gp = GpuProblem(m, img)
    vis = torch.randn(gp.shape, dtype=torch.complex64, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    out = []
    for kv in (1, 2):
        gp.ctx.psc_set_tiling(32, 4, kv)
        v = torch.empty_like(vis)
        d = torch.empty((4,) + tuple(vis.shape), dtype=vis.dtype, device="cuda")
        gp.ctx.psc_predict(0.5 * lmt, v, d)
        r = gp.ctx.psc_residual_grad(0.5 * lmt, vis, None, 1e6, cross=True)
        out.append([v.cpu().numpy()] + [x.cpu().numpy() for x in d] + [np.asarray(x) for x in r])
    for k, (x, y) in enumerate(zip(*out)):
        assert np.linalg.norm(x - y) < 1e-5 * np.linalg.norm(x), k
