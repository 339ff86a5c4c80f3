"""Network outputs written into the buffer that holds the inputs: the bits of a forward
pass into a buffer of its own, with several rounds of blocks."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [5, 20000, 100000])
@pytest.mark.parametrize("at", [0.0, 0.7, 1.0])
def test_outputs_in_the_input_buffer(batch, at):
    import torch
    from paper_1709_08681_gb300 import _abi
    rng = np.random.default_rng(batch)
    net = _abi.Mlp(batch)
    params = (0.1 * rng.normal(size=net.n_params)).astype(np.float32)
    params[-52:] = 1.0
    net.psc_mlp_set_params(params)
    x = torch.randn((batch, 52), device="cuda", generator=torch.Generator("cuda").manual_seed(batch))
    want = torch.empty((batch, 2), device="cuda")
    net.psc_mlp_forward(x, want)
    flat = x.reshape(-1)
    first = int(at * (flat.numel() - 2 * batch))
    y = flat[first:first + 2 * batch]
    net.psc_mlp_forward(x, y)
    assert torch.equal(y.reshape(batch, 2), want)
