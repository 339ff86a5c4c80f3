"""Launch shapes picked by size.  Lanes that share a visibility's rows must give the
bits of the rectangle they stand for (a solve's stop rule depends on them): compared
with the same context after psc_set_tiling(32, 4, 1), staged and unstaged, with
ragged time and channel groups, at the grid's border, in predictions and sums.  The
large shapes (flat bricks, track kernel) are compared with that rectangle at FP32
summation accuracy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _both(ctx, vis, lm):
    import torch
    out = []
    for shape in ("auto", "rect"):
        if shape == "rect":
            ctx.psc_set_tiling(32, 4, 1)
        v = torch.empty_like(vis)
        d = torch.empty((4,) + tuple(vis.shape), dtype=vis.dtype, device=vis.device)
        ctx.psc_predict(lm, v, d)
        out.append((v, d) + tuple(ctx.psc_residual_grad(lm, vis, None, 1e6, cross=True)))
    return out


@pytest.mark.parametrize("spec,n_ant,nt,nc,span,extent", [
    (("disk", 64, 24.0, 1024), 7, 40, 5, 1.0, 300.0),      # staged, ragged
    (("disk", 64, 24.0, 1024), 9, 60, 1, 4.0, 900.0),      # unstaged, one channel, the border
    (("disk", 64, 24.0, 1024), 3, 1, 1, 1.0, 300.0),
    (("disk", 64, 24.0, 1024), 12, 33, 9, 1.0, 300.0),
    (("disk", 64, 24.0, 512), 6, 20, 6, 1.0, 300.0),       # an aperture of 7 cells
    (("gauss", 64, 41.25, 360), 6, 37, 3, 1.0, 300.0),     # cut by the window
])
def test_shared_rows_keep_every_bit(spec, n_ant, nt, nc, span, extent):
    import cases
    import torch
    from gpu_cases import GpuProblem
    freqs = tuple(1.2e9 + 0.1e9 * k for k in range(nc))
    m, _, lmt, img = cases.problem(spec, n_ant=n_ant, n_time=nt, freqs=freqs, extent_m=extent)
    m.uvw_m = cases.geometry(n_ant, extent, nt, span, freqs)[0]
    gp = GpuProblem(m, img)
    vis = torch.randn(gp.shape, dtype=torch.complex64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    a, r = _both(gp.ctx, vis, 0.5 * lmt)
    for x, y in zip(a, r):
        same = torch.equal(x, y) if torch.is_tensor(x) else np.array_equal(x, y)
        assert same


# (grid spec, dish m, n_ant, nt, nc): flat bricks of pairs, flat bricks, the track kernel with two and one per lane
@pytest.mark.parametrize("spec,diam,n_ant,nt,nc,span", [
    (("disk", 64, 24.0, 1024), 25.0, 30, 201, 23, 0.3),
    (("disk", 64, 24.0, 1024), 25.0, 30, 201, 23, 6.0),
    (("disk", 512, 5.0, 1024), 8.0, 60, 45, 26, 0.05),
    (("disk", 512, 5.0, 1024), 8.0, 64, 20, 50, 0.02),
])
def test_large_shapes_agree_with_the_rectangle(spec, diam, n_ant, nt, nc, span):
    import cases
    import torch
    from gpu_cases import GpuProblem
    freqs = tuple(np.linspace(1.2e9, 1.6e9, nc))
    m, _, lmt, img = cases.problem(spec, n_ant=3, n_time=1, freqs=(1.2e9,))
    m.uvw_m, m.freq_hz = cases.geometry(n_ant, 300.0, nt, span, freqs)
    m.n_ant, m.diam_m = n_ant, diam
    lm = np.random.default_rng(2).normal(0, 1e-4, (n_ant, 2))
    gp = GpuProblem(m, img)
    vis = torch.randn(gp.shape, dtype=torch.complex64, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    a, r = _both(gp.ctx, vis, lm)
    for k, (x, y) in enumerate(zip(a, r)):
        x, y = (v.cpu().numpy() if torch.is_tensor(v) else np.asarray(v) for v in (x, y))
        assert np.linalg.norm(x - y) < 1e-5 * np.linalg.norm(y), k
