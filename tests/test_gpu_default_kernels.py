"""Which fused kernel a context without a tiling runs, and that nothing else decides its
results' bits: not the staging mode's staged kernels where staging was refused, and not
what else a batch holds (other contexts without a tiling, or contexts with one)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (antennas, time steps, channels, hours): the track kernel with one and two
# visibilities per lane, flat bricks, the rectangle, rows shared among lanes
ONE, TWO = (64, 20, 50, 0.02), (60, 45, 26, 0.05)
FLAT, RECT, SHARED = (12, 480, 64, 4.0), (24, 60, 12, 0.05), (6, 20, 4, 0.05)


def _problem(n_ant, nt, nc, span):
    import cases
    import torch
    from gpu_cases import GpuProblem
    m, _, _, img = cases.problem(("disk", 512, 5.0, 1024), n_ant=3, n_time=1, freqs=(1.2e9,))
    m.uvw_m, m.freq_hz = cases.geometry(n_ant, 300.0, nt, span, tuple(np.linspace(1.2e9, 1.6e9, nc)))
    m.n_ant, m.diam_m = n_ant, 25.0
    gp = GpuProblem(m, img)
    vis = torch.empty(gp.shape, dtype=torch.complex64, device="cuda")
    gp.ctx.psc_predict(np.random.default_rng(n_ant).normal(0, 1e-4, (n_ant, 2)), vis, None)
    return gp, vis


def _batch(probs):
    from paper_1709_08681_gb300 import _abi
    return _abi.Batch([gp.ctx for gp, _ in probs], [v for _, v in probs], None, [1e6] * len(probs))


@pytest.mark.parametrize("shape,name", [(ONE, "track_kernel<1>"), (TWO, "track_kernel<2>")])
def test_unstaged_contexts_keep_the_bricks(shape, name):
    from paper_1709_08681_gb300 import _abi
    gp, vis = _problem(*shape)
    b = _batch([(gp, vis)])
    assert b.psc_batch_kernel() == name
    b.close()
    gp.ctx.psc_set_staging(_abi.PSC_STAGE_NEVER)
    b = _batch([(gp, vis)])
    assert b.psc_batch_kernel().startswith("eval_kernel")
    b.close()
    lm = np.random.default_rng(1).normal(0, 1e-4, (shape[0], 2))
    auto = gp.ctx.psc_residual_grad(lm, vis, None, 1e6, cross=True)
    gp.ctx.psc_set_track_tiling(0)                    # the brick kernel, by a call
    brick = gp.ctx.psc_residual_grad(lm, vis, None, 1e6, cross=True)
    assert auto[0] == brick[0] and all(np.array_equal(x, y) for x, y in zip(auto[1:], brick[1:]))


def _offsets(probs):
    b = _batch(probs)
    b.psc_batch_begin([np.zeros((gp.m.n_ant, 2)) for gp, _ in probs])
    b.psc_batch_iterate(2)
    lms, _ = b.psc_batch_end()
    b.close()
    return lms


def _alone(gp, vis):
    """The same two iterations without a batch."""
    gp.ctx.psc_lm_begin(np.zeros((gp.m.n_ant, 2)))
    gp.ctx.psc_lm_iterate(vis, None, 1e6, 2)
    return gp.ctx.psc_lm_end()[0]


# "set": a context that was given the rectangle (32, 4, 1) by a call
@pytest.mark.parametrize("shapes", [(ONE, TWO), (TWO, ONE, SHARED), (TWO, "set"), ("set", ONE, FLAT, RECT)])
def test_a_batch_does_not_change_its_contexts(shapes):
    probs = [_problem(*(RECT if s == "set" else s)) for s in shapes]
    for (gp, _), s in zip(probs, shapes):
        if s == "set":
            gp.ctx.psc_set_tiling(32, 4, 1)
    for lm, (gp, vis) in zip(_offsets(probs), probs):
        assert np.array_equal(lm, _offsets([(gp, vis)])[0])
        assert np.array_equal(lm, _alone(gp, vis))


def test_batches_refuse_contexts_beside_the_track_tiling():
    from paper_1709_08681_gb300 import _abi
    probs = [_problem(*s) for s in (ONE, TWO)]
    probs[1][0].ctx.psc_set_track_tiling(2)                   # ONE's context runs the track kernel, but not by a call
    with pytest.raises(_abi.PscError) as e:
        _batch(probs)
    assert e.value.status == _abi.PSC_ERR_ARG


BRICKS, SHARED_ROWS = "eval_kernel<false, false, false>", "eval_kernel<false, false, true>"


@pytest.mark.parametrize("shapes,name", [
    ((ONE, TWO), "track_kernel<1> + track_kernel<2>"), ((FLAT, TWO), BRICKS + " + track_kernel<2>"),
    ((RECT, FLAT), BRICKS), ((SHARED, SHARED), SHARED_ROWS),
    ((RECT, SHARED, ONE), BRICKS + " + " + SHARED_ROWS + " + track_kernel<1>"),      # each at its own registers
])
def test_the_kernels_of_a_batch_by_name(shapes, name):
    b = _batch([_problem(*s) for s in shapes])
    assert b.psc_batch_kernel() == name
    b.close()


# the shapes of test_gpu_auto_shape.py, one more, and what is picked for each: (grid, dish m, antennas,
# times, channels, hours, extent m), (t_tile or items, c_group, per thread, lanes, track)
LARGE, SMALL = ("disk", 64, 24.0, 1024), ("disk", 512, 5.0, 1024)
PICKED = [
    (LARGE, 25.0, 7, 40, 5, 1.0, 300.0, (32, 4, 1, 16, 0)), (LARGE, 25.0, 9, 60, 1, 4.0, 900.0, (32, 4, 1, 8, 0)),
    (LARGE, 25.0, 3, 1, 1, 1.0, 300.0, (32, 4, 1, 8, 0)), (LARGE, 25.0, 12, 33, 9, 1.0, 300.0, (32, 4, 1, 16, 0)),
    (("disk", 64, 24.0, 512), 25.0, 6, 20, 6, 1.0, 300.0, (32, 4, 1, 8, 0)),
    (("gauss", 64, 41.25, 360), 25.0, 6, 37, 3, 1.0, 300.0, (32, 4, 1, 16, 0)),
    (LARGE, 25.0, 30, 60, 23, 0.3, 300.0, (32, 4, 1, 1, 0)),
    (LARGE, 20.0, 30, 201, 23, 0.3, 300.0, (256, 0, 2, 1, 0)),         # the aperture inside the window
    (LARGE, 25.0, 30, 201, 23, 0.3, 300.0, (256, 0, 1, 1, 0)), (LARGE, 25.0, 30, 201, 23, 6.0, 300.0, (256, 0, 1, 1, 0)),
    (SMALL, 8.0, 60, 45, 26, 0.05, 300.0, (256, 0, 1, 1, 2)), (SMALL, 8.0, 64, 20, 50, 0.02, 300.0, (32, 4, 1, 1, 1)),
]


@pytest.mark.parametrize("spec,diam,n_ant,nt,nc,span,extent,shape", PICKED)
def test_the_shape_that_is_picked(spec, diam, n_ant, nt, nc, span, extent, shape):
    import cases
    from gpu_cases import GpuProblem
    freqs = tuple(1.2e9 + 0.1e9 * k for k in range(nc)) if nc < 20 else tuple(np.linspace(1.2e9, 1.6e9, nc))
    m, _, _, img = cases.problem(spec, n_ant=3, n_time=1, freqs=(1.2e9,))
    m.uvw_m, m.freq_hz = cases.geometry(n_ant, extent, nt, span, freqs)
    m.n_ant, m.diam_m = n_ant, diam
    ctx = GpuProblem(m, img).ctx
    assert ctx.psc_get_shape() == shape
    ctx.psc_set_tiling(32, 4, 1)
    assert ctx.psc_get_shape() == (32, 4, 1, 1, 0)
    if nt * nc >= 64:
        ctx.psc_set_flat_tiling(64, 1)
        assert ctx.psc_get_shape() == (64, 0, 1, 1, 0)
