"""Which fused kernel a context without a tiling runs, and that nothing else decides its
results' bits: not the staging mode's staged kernels where staging was refused."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (antennas, time steps, channels, hours): the track kernel with one and two
# visibilities per lane
ONE, TWO = (64, 20, 50, 0.02), (60, 45, 26, 0.05)


def _problem(n_ant, nt, nc, span):
    import cases
    import torch
    from gpu_cases import GpuProblem
    m, _, _, img = cases.problem(("disk", 512, 5.0, 1024), n_ant=3, n_time=1, freqs=(1.2e9,))
    m.uvw_m, m.freq_hz = cases.geometry(n_ant, 300.0, nt, span, tuple(np.linspace(1.2e9, 1.6e9, nc)))
    m.n_ant, m.diam_m = n_ant, 8.0
    gp = GpuProblem(m, img)
    vis = torch.empty(gp.shape, dtype=torch.complex64, device="cuda")
    gp.ctx.psc_predict(np.random.default_rng(n_ant).normal(0, 1e-4, (n_ant, 2)), vis, None)
    return gp, vis


def _batch(probs):
    from paper_1709_08681_gb300 import _abi
    return _abi.Batch([gp.ctx for gp, _ in probs], [v for _, v in probs], None, [1e6] * len(probs))


@pytest.mark.parametrize("shape,name", [(ONE, "track_kernel<1>"), (TWO, "track_kernel<2>")])
def test_unstaged_contexts_keep_the_bricks(shape, name):
    from paper_1709_08681_gb300 import _abi
    gp, vis = _problem(*shape)
    b = _batch([(gp, vis)])
    assert b.psc_batch_kernel() == name
    b.close()
    gp.ctx.psc_set_staging(_abi.PSC_STAGE_NEVER)
    b = _batch([(gp, vis)])
    assert b.psc_batch_kernel().startswith("eval_kernel")
    b.close()
    lm = np.random.default_rng(1).normal(0, 1e-4, (shape[0], 2))
    auto = gp.ctx.psc_residual_grad(lm, vis, None, 1e6, cross=True)
    gp.ctx.psc_set_track_tiling(0)                    # the brick kernel, by a call
    brick = gp.ctx.psc_residual_grad(lm, vis, None, 1e6, cross=True)
    assert auto[0] == brick[0] and all(np.array_equal(x, y) for x, y in zip(auto[1:], brick[1:]))
