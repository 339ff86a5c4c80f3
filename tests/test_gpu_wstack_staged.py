"""The stacked kernel's staged planes against its unstaged taps (PSC_STAGE_NEVER, held
to the oracle in test_gpu_wstack.py): bricks that touch one, two and many planes,
one and two visibilities per thread, the window's and the grid's edge.  Both sum
some 600 FP32 taps of the same values in another order: 1e-5 (the parity bound)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("planes", [2, 3, 40])
@pytest.mark.parametrize("tiling", [None, ("flat", 128, 1), ("flat", 64, 2), ("rect", 40, 3, 1)])
@pytest.mark.parametrize("extent", [300.0, 700.0])
def test_staged_matches_unstaged(planes, tiling, extent):
    import cases
    import torch
    from gpu_cases import GpuProblem
    from paper_1709_08681_gb300 import _abi
    nt, freqs = 130, (1.2e9, 1.3e9, 1.4e9)
    m, _, lmt, img = cases.problem(cases.DISK_SMALL, n_ant=5, n_time=2, freqs=freqs)
    m.uvw_m = cases.geometry(5, extent, nt, 0.5, freqs)[0]
    gp = GpuProblem(m, img)
    a, b = _abi.psc_snapshot_plane(gp.uvw, nt * 10)
    lo, hi = _abi.psc_wstack_range(gp.uvw, nt * 10, a, b)
    f0, f1 = (f / 299792458.0 for f in (min(freqs), max(freqs)))
    w_lo, w_hi = min(lo * f0, lo * f1) - 1e-3, max(hi * f0, hi * f1) + 1e-3
    ng = m.grid.shape[0]
    g = torch.Generator("cuda").manual_seed(planes)
    stack = torch.randn((planes, ng, ng), dtype=torch.complex64, device="cuda", generator=g)
    gp.ctx.psc_set_wstack(stack, planes, w_lo, (w_hi - w_lo) / (planes - 1) * (1 + 1e-9), a, b)
    if tiling is not None:
        (gp.ctx.psc_set_flat_tiling if tiling[0] == "flat" else gp.ctx.psc_set_tiling)(*tiling[1:])
    vis = torch.randn(gp.shape, dtype=torch.complex64, device="cuda", generator=g)
    out = []
    for mode in (_abi.PSC_STAGE_AUTO, _abi.PSC_STAGE_NEVER):
        gp.ctx.psc_set_staging(mode)
        V, dV = gp.predict(0.5 * lmt)
        out.append((V, dV) + tuple(gp.ctx.psc_residual_grad(0.5 * lmt, vis, None, 1.0, cross=True)))
    for k, (x, y) in enumerate(zip(*out)):
        assert np.linalg.norm(np.asarray(x) - np.asarray(y)) < 1e-5 * np.linalg.norm(np.asarray(y)), k
