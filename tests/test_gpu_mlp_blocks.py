"""The network's row blocks and gradient splits at their edges: batches around
one and two blocks of 32 rows, around the change to blocks of 64, ragged splits of
the weight gradient, and a second, smaller batch after a larger one (stale rows
must not leak).  Oracle and tolerances as in test_gpu_mlp.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import mlp as O
from test_gpu_mlp import init_params, rel


@pytest.mark.parametrize("B,max_batch", [(31, 31), (32, 32), (33, 64), (65, 65), (255, 256), (257, 300), (2049, 2049),
                                         (4864, 4864), (4865, 4865), (5000, 8192)])
def test_blocks_match_oracle(B, max_batch):
    from paper_1709_08681_gb300 import _abi
    rng = np.random.default_rng(B)
    flat = init_params(7)
    net = _abi.Mlp(max_batch)
    net.psc_mlp_set_params(flat)
    for n in (B, max(1, B // 3)):
        x = rng.normal(0, 1, (n, O.N_IN)).astype(np.float32)
        t = rng.normal(0, 1, (n, O.N_OUT)).astype(np.float32)
        xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
        y = net.psc_mlp_forward(xd).cpu().numpy()
        yo, _ = O.forward(flat.astype(np.float64), x.astype(np.float64))
        assert rel(y, yo) < 2e-3
        loss, g = net.psc_mlp_grad(xd, td)
        lo, go = O.loss_and_grad(flat.astype(np.float64), x.astype(np.float64), t.astype(np.float64))
        assert abs(loss - lo) < 2e-3 * lo
        off = 0
        for name, shp in O.SHAPES:
            k = int(np.prod(shp))
            if name in O.TRAINED:
                assert rel(g[off:off + k], go[off:off + k]) < 2e-2, name
            else:
                assert np.all(g[off:off + k] == 0)
            off += k
