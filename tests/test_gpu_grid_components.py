"""The component grid's half-plane pass: every row and column against the direct
sum in 64 bits, at the edges of its tiles (128 columns, 64 rows), of the groups of
64 fine steps and of the 16-component blocks, with the first row and column (which
have no mirror image) and the row v = 0 among them; and the w-plane grids, whose
complex fluxes leave no symmetry.  Bound: the component grid's own 1e-6 of the
largest cell (test_gpu_wsnap.py)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _direct(comp, ng, cell, wp=None):
    import torch
    c = torch.from_numpy(comp).cuda()
    u = (torch.arange(ng, dtype=torch.float64, device="cuda") - ng // 2) / (ng * cell)
    one = torch.ones((), dtype=torch.float64, device="cuda")
    s = c[:, 2].to(torch.complex128)
    if wp is not None:
        s = s * torch.polar(one, 2 * np.pi * wp * c[:, 3])
    a = torch.polar(one, 2 * np.pi * u[:, None] * c[None, :, 0]) * s
    return torch.polar(one, 2 * np.pi * u[:, None] * c[None, :, 1]) @ a.T


@pytest.mark.parametrize("ng,n", [(2, 1), (4, 3), (62, 16), (64, 17), (66, 31), (128, 33), (130, 48), (254, 200), (256, 1), (1030, 65)])
def test_every_cell(ng, n):
    import torch
    from paper_1709_08681_gb300 import _abi
    rng = np.random.default_rng(ng + n)
    cell = 1e-5
    comp = np.concatenate([rng.uniform(-0.4, 0.4, (n, 2)) * ng * cell, rng.uniform(0.1, 1.0, (n, 1))], 1)
    out = torch.full((ng, ng), float("nan"), dtype=torch.complex64, device="cuda")
    _abi.psc_model_grid_components(comp, ng, cell, out)
    ref = _direct(comp, ng, cell)
    assert float(torch.max(torch.abs(out - ref))) < 1e-6 * float(torch.max(torch.abs(ref)))
    planes = torch.full((2, ng, ng), float("nan"), dtype=torch.complex64, device="cuda")
    comp4 = np.concatenate([comp, -1e-4 * rng.uniform(0.0, 1.0, (n, 1))], 1)
    _abi.psc_model_grid_wstack(comp4, ng, cell, 2, -300.0, 500.0, planes)
    for p in range(2):
        ref = _direct(comp4, ng, cell, -300.0 + 500.0 * p)
        assert float(torch.max(torch.abs(planes[p] - ref))) < 1e-6 * float(torch.max(torch.abs(ref)))
