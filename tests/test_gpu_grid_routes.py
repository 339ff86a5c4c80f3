"""The model grid on both sides of the lines between transforms and matrix products, with
the checks and bounds of test_gpu_grid_fft.py; and a grid of a long odd part beside an
image of a few pixels, whose products are short: it may not take the direct DFT (45 times
as long as the power of two beside it; the products take 1.4 times as long)."""
import time

import pytest

import test_gpu_grid_fft as dft

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_img,n_grid", [
    (256, 1008), (248, 1008),       # odd part 63: up to (N + 256) / 8 in small grids
    (120, 1920), (112, 1920),       # 15: up to N / 8
    (136, 9216), (128, 9216),       # 9: up to N / 8 - 8
    (30, 1920), (28, 1920),         # 15: up to N / 2
    (50, 9216), (46, 9216),         # 9: up to N / 2 - 16
    (514, 1028), (514, 2052),       # 257, 513: up to N for images over 512
])
def test_both_sides_of_the_line(n_img, n_grid):
    dft.test_model_grid_matches_the_dft(n_img, n_grid)


def test_a_long_odd_part_takes_the_products():
    import torch
    from paper_1709_08681_gb300 import _abi
    img = torch.rand((64, 64), device="cuda")
    best = {}
    for n in (8192, 8176):                                       # 8176 = 16 x 511
        out = torch.empty((n, n), dtype=torch.complex64, device="cuda")
        for _ in range(8):
            torch.cuda.synchronize()
            t = time.perf_counter()
            _abi.psc_model_grid(64, n, 1e-5, 32, 20, img, out)
            torch.cuda.synchronize()
            best[n] = min(best.get(n, 1.0), time.perf_counter() - t)
    assert best[8176] < 8 * best[8192]
