"""The model grid by FFT against a 64-bit DFT: every pass structure (radices
2 to 16, an odd part, the longest transform) and the grids of a large odd part
that keep the matrix products.  The bound is the model grid's own (relative L2
1e-6, as in test_gpu_parity.py); rows and columns are checked one by one where
a wrong mirror row or a lost column would show."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(2, 2), (2, 4), (4, 8), (6, 6), (8, 16), (10, 32), (16, 64), (72, 72), (96, 384), (100, 300), (126, 254),
         (128, 128), (254, 508), (512, 1024), (700, 2800), (984, 3936), (62, 16384), (40, 1022), (1042, 1042), (16, 1042), (10, 1042)]


@pytest.mark.parametrize("n_img,n_grid", SIZES)
def test_model_grid_matches_the_dft(n_img, n_grid):
    import torch
    from paper_1709_08681_gb300 import _abi
    rng = np.random.default_rng(n_img * 20000 + n_grid)
    img = rng.normal(size=(n_img, n_img)).astype(np.float32)
    out = torch.full((n_grid, n_grid), float("nan"), dtype=torch.complex64, device="cuda")
    _abi.psc_model_grid(n_img, n_grid, 1e-5, 32, 20, torch.from_numpy(img).cuda(), out)
    p = torch.arange(n_img, dtype=torch.float64, device="cuda") - n_img // 2
    k = torch.arange(n_grid, dtype=torch.float64, device="cuda") - n_grid // 2
    e = torch.polar(torch.ones((), dtype=torch.float64, device="cuda"), 2 * np.pi * torch.remainder(k[:, None] * p, n_grid) / n_grid)
    t = e @ torch.from_numpy(img).cuda().to(torch.complex128)      # [gy][col]
    for rows in torch.arange(n_grid, device="cuda").split(2048):
        ref = t[rows] @ e.T
        d, r = (torch.linalg.vector_norm(v, dim=1) for v in (out[rows].to(torch.complex128) - ref, ref))
        assert float(torch.max(d / r)) < 2e-6                      # every row
        assert float(torch.linalg.vector_norm(d) / torch.linalg.vector_norm(r)) < 1e-6
