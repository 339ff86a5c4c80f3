"""Model grids in a second CUDA context of the process: the tables and workspaces that
the library keeps on the device belong to one context each.  The same kernels on the
same inputs, so the same bits in both, in the first also after the second is gone."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


class _Driver:
    def __init__(self):
        self.cu = ctypes.CDLL("libcuda.so.1")

    def __call__(self, name, *args):
        assert getattr(self.cu, name)(*args) == 0, name

    def alloc(self, n):
        p = ctypes.c_uint64()
        self("cuMemAlloc_v2", ctypes.byref(p), ctypes.c_size_t(n))
        return p


def _grids(drv, img, comp, sizes):
    from paper_1709_08681_gb300 import _abi
    lib, out = _abi.lib(), []
    src = drv.alloc(img.nbytes)
    drv("cuMemcpyHtoD_v2", src, img.ctypes.data_as(ctypes.c_void_p), ctypes.c_size_t(img.nbytes))
    for n in sizes:
        for kind in ("image", "components"):
            g = np.empty((n, n), np.complex64)
            dst = drv.alloc(g.nbytes)
            if kind == "image":
                gd = _abi.psc_grid_desc(img.shape[0], n, 1e-5, 34, 20)
                assert lib.psc_model_grid(ctypes.byref(gd), src.value, dst.value, None) == 0
            else:
                c = comp.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
                assert lib.psc_model_grid_components(len(comp), c, n, 1e-5, dst.value, None) == 0
            drv("cuMemcpyDtoH_v2", g.ctypes.data_as(ctypes.c_void_p), dst, ctypes.c_size_t(g.nbytes))
            drv("cuMemFree_v2", dst)
            out.append(g)
    drv("cuMemFree_v2", src)
    return out


def test_second_context_gives_the_same_grids():
    import torch
    torch.zeros(1, device="cuda")
    torch.cuda.synchronize()
    rng = np.random.default_rng(4)
    img = rng.random((64, 64), dtype=np.float32)
    comp = np.ascontiguousarray(np.column_stack([rng.normal(0, 1e-4, (50, 2)), rng.random(50)]))
    sizes, drv = (256, 360), _Driver()                 # a power of two, and tables of the call's own
    first = _grids(drv, img, comp, sizes)
    ctx = ctypes.c_void_p()
    drv("cuCtxCreate_v2", ctypes.byref(ctx), 0, 0)
    try:
        second = _grids(drv, img, comp, sizes)
    finally:
        drv("cuCtxDestroy_v2", ctx)                    # pops it
    again = _grids(drv, img, comp, sizes)
    for a, b, c in zip(first, second, again):
        assert np.isfinite(a).all() and np.abs(a).max() > 0
        assert np.array_equal(a, b) and np.array_equal(a, c)
