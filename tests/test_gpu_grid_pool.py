"""The memory that the model-grid calls keep between calls goes back: by
psc_release_workspace where there is no psc_ctx, and with the last psc_ctx of the CUDA
context that holds it, whatever lives in another."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NG, COMP = 1024, 500          # operands of 1024 x 512 x 6 x 3 bytes and more: over 8 MB are kept


def _components():
    rng = np.random.default_rng(1)
    return np.ascontiguousarray(np.column_stack([rng.normal(0, 1e-4, (COMP, 2)), rng.random(COMP)]))


def test_release_without_a_context():
    import torch
    from paper_1709_08681_gb300 import _abi
    out = torch.empty((NG, NG), dtype=torch.complex64, device="cuda")
    _abi.psc_model_grid_components(_components(), NG, 1e-5, out)        # kernels and tables are loaded
    _abi.psc_release_workspace()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    _abi.psc_model_grid_components(_components(), NG, 1e-5, out)
    assert torch.cuda.mem_get_info()[0] < free - (8 << 20)
    first = out.clone()
    torch.cuda.synchronize()
    _abi.psc_release_workspace()
    held = torch.cuda.mem_get_info()[0]
    _abi.psc_model_grid_components(_components(), NG, 1e-5, out)
    _abi.psc_release_workspace()
    assert torch.cuda.mem_get_info()[0] == held and torch.equal(out, first)


def test_a_second_cuda_context_gives_its_memory_back_by_itself():
    import torch
    from paper_1709_08681_gb300 import _abi
    from test_gpu_grid_contexts import _Driver
    import cases
    from gpu_cases import GpuProblem
    m, _, _, img = cases.problem(cases.DISK_SMALL, n_ant=3, n_time=2)
    here = GpuProblem(m, img)                                           # a psc_ctx that outlives the second context
    torch.cuda.synchronize()
    lib, drv, ctx = _abi.lib(), _Driver(), ctypes.c_void_p()
    comp, ng = _components(), m.grid.shape[0]

    def free():
        a, b = ctypes.c_size_t(), ctypes.c_size_t()
        drv("cuMemGetInfo_v2", ctypes.byref(a), ctypes.byref(b))
        return a.value

    drv("cuCtxCreate_v2", ctypes.byref(ctx), 0, 0)
    try:
        uvw, grid = drv.alloc(m.uvw_m.nbytes), drv.alloc(8 * ng * ng)
        data = np.ascontiguousarray(m.uvw_m)
        drv("cuMemcpyHtoD_v2", uvw, data.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(data.nbytes))

        def one():
            """A grid and a psc_ctx on it; the memory in use just before its end and after it."""
            c = comp.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
            assert lib.psc_model_grid_components(COMP, c, ng, 1e-5, grid.value, None) == 0
            p = _abi.Context(3, 2, 1, uvw.value, m.freq_hz, "disk", m.diam_m, m.alpha_per_dlambda, 1, img.shape[0], ng,
                             m.cell_rad, m.support, m.oversample, grid.value)
            before = free()
            p.close()
            return before, free()

        one()                                                           # kernels and tables are loaded
        before, after = one()
        assert after > before + (8 << 20)
    finally:
        drv("cuCtxDestroy_v2", ctx)
    assert here.predict(np.zeros((3, 2)), False)[0].shape == here.shape
