"""Contexts without a tiling that take the track kernel or flat bricks of pairs by their
size are as exact as the rectangle (32, 4, 1): both against the FP64 oracle, on data whose residuals are
noise of a hundredth of the visibilities, where an error of the model's phase shows in
chi^2 most.  Boxes that the warps stage and boxes too wide for that (taps read from the
grid), one and two visibilities per lane.

Bound: half as far again as the rectangle, and on top what the FP32 roundings of one box
of one channel give where they are common to its visibilities: 2^-23 of V each, so
2 2^-23 |V| / |R| of chi^2 and 2^-23 of the normals, over the root of the number of
boxes; of the gradient's norm 2^-23 |V| / |R| over the root of the boxes of an antenna."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


SMALL, LARGE = ("disk", 512, 5.0, 1024), ("disk", 64, 24.0, 1024)


# (grid, dish m, antennas, time steps, channels, hours, array extent m, shape: per thread and per lane of the track kernel)
@pytest.mark.parametrize("spec,diam,n_ant,nt,nc,span,extent,shape", [
    (SMALL, 25.0, 60, 45, 26, 0.05, 300.0, (1, 2)),
    (SMALL, 25.0, 64, 20, 50, 0.02, 300.0, (1, 1)),
    (SMALL, 25.0, 60, 64, 19, 0.6, 1500.0, (1, 2)),      # the longest baselines' boxes do not fit the tile
    (SMALL, 25.0, 201, 8, 13, 0.7, 2200.0, (1, 1)),      # several cells a step: half of the boxes do not fit
    (LARGE, 12.0, 30, 201, 23, 0.3, 300.0, (2, 0)),      # flat bricks of pairs
])
def test_default_is_as_exact_as_the_rectangle(spec, diam, n_ant, nt, nc, span, extent, shape):
    import cases
    import torch
    from gpu_cases import GpuProblem
    from oracle import psc
    from paper_1709_08681_gb300 import inputs as I
    m, _, _, img = cases.problem(spec, n_ant=3, n_time=1, freqs=(1.2e9,))
    m.uvw_m, m.freq_hz = cases.geometry(n_ant, extent, nt, span, tuple(np.linspace(1.2e9, 1.6e9, nc)))
    m.n_ant, m.diam_m = n_ant, diam
    gp = GpuProblem(m, img)
    m.grid = gp.grid.cpu().numpy().astype(np.complex128)
    lm = np.random.default_rng(n_ant).normal(0, 1e-4, (n_ant, 2))
    V, _ = psc.predict(m, lm, False)
    scale = np.sqrt(np.mean(np.abs(V) ** 2))
    sigma = 1e-2 * scale
    vis = (V + I.complex_noise(V.shape, sigma, 3)).astype(np.complex64)
    w_scale = float(np.float32(1.0 / sigma ** 2))
    exact = psc.chi2_grad_normal(m, lm, vis.astype(np.complex128), np.full(V.shape, w_scale))
    dev = gp.upload(vis)
    assert gp.ctx.psc_get_shape()[2::2] == shape
    auto = gp.ctx.psc_residual_grad(lm, dev, None, w_scale, cross=True)
    gp.ctx.psc_set_tiling(32, 4, 1)
    rect = gp.ctx.psc_residual_grad(lm, dev, None, w_scale, cross=True)
    boxes = nc * len(m.uvw_m[0]) * -(-nt // (32 * max(shape[1], 1)))
    ratio = scale / np.sqrt(np.mean(np.abs(vis - V) ** 2))
    ulp = 2.0 ** -23
    floors = (2 * ulp * ratio / np.sqrt(boxes), ulp * ratio / np.sqrt(2 * boxes / n_ant), ulp / np.sqrt(boxes), ulp / np.sqrt(boxes))
    errs = [[float(np.linalg.norm(np.asarray(x) - y) / np.linalg.norm(y)) for x, y in zip(got, exact)] for got in (auto, rect)]
    print("errors of the default %s, of the rectangle %s, floors %s" % tuple(
        ["%.2g" % x for x in v] for v in (errs[0], errs[1], floors)))
    for a, r, f in zip(errs[0], errs[1], floors):
        assert a < 1.5 * r + f
