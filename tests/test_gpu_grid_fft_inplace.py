"""An image that lies in the buffer that takes its model grid: the same grid as from an
image elsewhere, by transforms (with and without an odd part) and by matrix products."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_img,n_grid", [(2048, 4096), (1024, 1024), (1536, 1536), (40, 1022), (30, 1022)])
@pytest.mark.parametrize("at", [0.0, 0.4, 1.0])
def test_image_in_the_grid_buffer(n_img, n_grid, at):
    import torch
    from paper_1709_08681_gb300 import _abi
    img = torch.randn((n_img, n_img), device="cuda", generator=torch.Generator("cuda").manual_seed(n_img))
    want = torch.empty((n_grid, n_grid), dtype=torch.complex64, device="cuda")
    _abi.psc_model_grid(n_img, n_grid, 1e-5, 32, 20, img, want)
    out = torch.zeros((n_grid, n_grid), dtype=torch.complex64, device="cuda")
    flat = torch.view_as_real(out).reshape(-1)
    first = int(at * (flat.numel() - img.numel()))
    inside = flat[first:first + img.numel()]
    inside.copy_(img.reshape(-1))
    torch.cuda.synchronize()
    _abi.psc_model_grid(n_img, n_grid, 1e-5, 32, 20, inside, out)
    assert torch.equal(out, want)
