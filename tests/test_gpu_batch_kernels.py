"""Batches without tilings whose contexts take different fused kernels: two persistent
launches an iteration.  Each context's offsets must have the bits of a batch of its own
(same kernel, records summed in the same order).  Where contexts of one and two
visibilities per lane meet, those of two run with one: another FP32 summation order,
compared to 1e-4 of the largest offset (sums to 1e-6, times a condition below 100)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (antennas, time steps, channels, hours): bricks below the large sizes (rows shared
# among lanes, rectangle), flat bricks, the track kernel with one and two per lane
SHARED, RECT, FLAT = (6, 20, 4, 0.05), (20, 60, 8, 0.05), (12, 480, 64, 4.0)
ONE, TWO = (64, 20, 50, 0.02), (60, 45, 26, 0.05)


def _problem(n_ant, nt, nc, span):
    import cases
    import torch
    from gpu_cases import GpuProblem
    m, _, _, img = cases.problem(("disk", 512, 5.0, 1024), n_ant=3, n_time=1, freqs=(1.2e9,))
    freqs = tuple(np.linspace(1.2e9, 1.6e9, nc))
    m.uvw_m, m.freq_hz = cases.geometry(n_ant, 300.0, nt, span, freqs)
    m.n_ant, m.diam_m = n_ant, 8.0
    gp = GpuProblem(m, img)
    vis = torch.empty(gp.shape, dtype=torch.complex64, device="cuda")
    gp.ctx.psc_predict(np.random.default_rng(n_ant).normal(0, 1e-4, (n_ant, 2)), vis, None)
    return gp, vis


def _offsets(probs):
    from paper_1709_08681_gb300 import _abi
    b = _abi.Batch([gp.ctx for gp, _ in probs], [v for _, v in probs], None, [1e6] * len(probs))
    b.psc_batch_begin([np.zeros((gp.m.n_ant, 2)) for gp, _ in probs])
    b.psc_batch_iterate(2)
    lms, _ = b.psc_batch_end()
    name = b.psc_batch_kernel()
    b.close()
    return lms, name


@pytest.mark.parametrize("shapes", [(RECT, ONE), (TWO, SHARED, FLAT), (SHARED, ONE, RECT, ONE), (ONE, TWO, SHARED)])
def test_each_context_as_in_a_batch_of_its_own(shapes):
    probs = [_problem(*s) for s in shapes]
    single = [_offsets([p]) for p in probs]
    lms, name = _offsets(probs)
    assert [n.startswith("track") for _, n in single] == [s in (ONE, TWO) for s in shapes]
    assert name.startswith("eval_kernel")
    for s, x, (y, _) in zip(shapes, lms, single):
        if s is TWO and ONE in shapes:
            assert np.max(np.abs(x - y[0])) < 1e-4 * np.max(np.abs(y[0]))
        else:
            assert np.array_equal(x, y[0])
