"""The stencil pass's grid reads at their edges: rows copied to shared memory
(apertures up to 16 cells), apertures too wide for that, a grid that is only
8-byte aligned, and visibilities whose aperture crosses the grid's border.  The
oracle and the bounds are those of test_gpu_features.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1709_08681_gb300 import _abi, inputs as I
from oracle import features as F, psc

import cases

SIG = 30.0 * I.ARCSEC


# (grid spec, support, array extent m, aligned): aperture radii of 14, 14 (crossing the border), 21 and 2.8 cells
@pytest.mark.parametrize("spec,support,extent,aligned", [
    (("disk", 64, 24.0, 1024), 32, 300.0, False),
    (("disk", 64, 24.0, 1024), 32, 1000.0, True),
    (("disk", 64, 24.0, 1536), 64, 300.0, True),
    (("disk", 64, 24.0, 206), 32, 300.0, True),
])
@pytest.mark.parametrize("nt,nc,stride", [(4, 8, 1), (30, 3, 7), (64, 1, 1)])
def test_rows_match_oracle(spec, support, extent, aligned, nt, nc, stride):
    freqs = tuple(1.3e9 + 0.03e9 * k for k in range(nc))
    m, _, lmt, img = cases.problem(spec, n_ant=5, n_time=nt, freqs=freqs, sigma_arcsec=30.0, support=support, extent_m=extent)
    V, _ = psc.predict(m, lmt, False)
    vobs = (V + I.complex_noise(V.shape, 1e-3, 9)).astype(np.complex64)
    ref = F.features(m, vobs, np.full(V.shape, 1e6, dtype=np.float32), SIG, stride)
    ng = m.grid.shape[0]
    buf = torch.zeros(ng * ng + 1, dtype=torch.complex64, device="cuda")
    grid = buf[0 if aligned else 1:][:ng * ng]
    grid.copy_(torch.from_numpy(m.grid.astype(np.complex64)).reshape(-1))
    uvw = torch.from_numpy(np.ascontiguousarray(m.uvw_m)).cuda()
    ctx = _abi.Context(5, nt, nc, uvw, m.freq_hz, "disk", m.diam_m, m.alpha_per_dlambda, 1, img.shape[0], ng, m.cell_rad,
                       support, 20, grid)
    got = ctx.psc_features(torch.from_numpy(vobs).cuda(), None, 1e6, SIG, stride).cpu().numpy()
    assert np.max(np.abs(got[:, :2] - ref[:, :2])) < 1e-4
    assert np.max(np.abs(got[:, 2:27] / ref[:, 2:27] - 1.0)) < 1e-5
    assert np.max(np.abs(got[:, 27:] - ref[:, 27:])) < 1e-5 * max(1.0, np.max(np.abs(ref[:, 27:])))
