"""Launches of one kernel with different amounts of shared memory: none may take from
another what it needs, neither from another thread's call nor from a batch made earlier."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _together(calls, repeats):
    """Each of calls in a thread of its own, repeats times; what they raised."""
    import torch
    raised, go = [], threading.Barrier(len(calls))

    def body(call):
        stream = torch.cuda.Stream()
        go.wait()
        try:
            for _ in range(repeats):
                call(stream)
        except Exception as e:
            raised.append(e)

    threads = [threading.Thread(target=body, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return raised


def test_threads_make_grids_of_different_sizes():
    import torch
    from paper_1709_08681_gb300 import _abi
    img = torch.randn((64, 64), device="cuda")
    sizes = (64, 64, 8192)
    outs = [torch.empty((n, n), dtype=torch.complex64, device="cuda") for n in sizes]
    torch.cuda.synchronize()
    raised = _together([lambda s, n=n, out=out: _abi.psc_model_grid(64, n, 1e-5, 32, 20, img, out, s)
                        for n, out in zip(sizes, outs)], 400)
    assert not raised, raised


def _problem(n_ant, nt, freqs, diam):
    import cases
    import torch
    from gpu_cases import GpuProblem
    m, _, _, img = cases.problem(("disk", 512, 5.0, 1024), n_ant=n_ant, n_time=nt, freqs=freqs)
    m.diam_m = diam
    gp = GpuProblem(m, img)
    vis = torch.randn(gp.shape, dtype=torch.complex64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    return gp, vis


def test_threads_form_features_of_different_apertures():
    probs = [_problem(4, 4, (1.3e9,) * 8, d) for d in (8.0, 8.0, 60.0)]
    expect = [gp.ctx.psc_features(vis, None, 1e6).cpu().numpy() for gp, vis in probs]
    raised = _together([lambda s, gp=gp, vis=vis: gp.ctx.psc_features(vis, None, 1e6) for gp, vis in probs], 5000)
    assert not raised, raised
    for (gp, vis), x in zip(probs, expect):
        assert np.array_equal(gp.ctx.psc_features(vis, None, 1e6).cpu().numpy(), x)


def test_a_smaller_context_leaves_a_batch_its_tables():
    from paper_1709_08681_gb300 import _abi
    large, small = _problem(5, 40, (1.3e9, 1.4e9), 60.0), _problem(5, 40, (1.3e9, 1.4e9), 8.0)
    for gp, _ in (large, small):
        gp.ctx.psc_set_track_tiling(2)
    b = _abi.Batch([large[0].ctx], [large[1]], None, [1e6])
    small[0].ctx.psc_residual_grad(np.zeros((5, 2)), small[1], None, 1e6)
    b.psc_batch_begin([np.zeros((5, 2))])
    b.psc_batch_iterate(1)
    lms, _ = b.psc_batch_end()
    b.close()
    assert np.all(np.isfinite(lms[0]))
