"""Baselines that are not finite (as flagged ones may be) or absurdly long, in contexts whose
sizes would take them to the track kernel or to two visibilities a thread, whose taps
share rows and columns: such contexts keep one visibility a thread, the calls for the
others are refused, and every other visibility is as without them, to FP32 rounding (a
brick may read its cells another way)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SMALL, LARGE = ("disk", 512, 5.0, 1024), ("disk", 64, 24.0, 1024)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), 1e8])
@pytest.mark.parametrize("spec,n_ant,nt,nc,span", [
    (SMALL, 60, 45, 26, 0.05), (SMALL, 201, 1, 104, 0.0), (LARGE, 30, 201, 23, 0.3),
])
def test_such_contexts_keep_one_visibility_a_thread(spec, n_ant, nt, nc, span, bad):
    import cases
    import torch
    from gpu_cases import GpuProblem
    from paper_1709_08681_gb300 import _abi
    m, _, _, img = cases.problem(spec, n_ant=3, n_time=1, freqs=(1.2e9,))
    m.uvw_m, m.freq_hz = cases.geometry(n_ant, 300.0, nt, span, tuple(np.linspace(1.2e9, 1.6e9, nc)))
    m.n_ant, m.diam_m = n_ant, 12.0
    good = GpuProblem(m, img)
    assert good.ctx.psc_get_shape()[2:] != (1, 1, 0)
    good.ctx.psc_set_tiling(32, 4, 1)
    lm = np.random.default_rng(5).normal(0, 1e-4, (n_ant, 2))
    want = torch.empty(good.shape, dtype=torch.complex64, device="cuda")
    good.ctx.psc_predict(lm, want, None)
    m.uvw_m = m.uvw_m.copy()
    m.uvw_m[nt // 2, 7, 1] = bad
    gp = GpuProblem(m, img)
    assert gp.ctx.psc_get_shape()[2:] == (1, 1, 0)
    for call in (lambda: gp.ctx.psc_set_track_tiling(1), lambda: gp.ctx.psc_set_tiling(32, 4, 2)):
        with pytest.raises(_abi.PscError) as e:
            call()
        assert e.value.status == _abi.PSC_ERR_ARG
    got = torch.empty_like(want)
    gp.ctx.psc_predict(lm, got, None)
    got[nt // 2, 7] = want[nt // 2, 7]
    assert float(torch.linalg.vector_norm(got - want)) < 1e-6 * float(torch.linalg.vector_norm(want))
