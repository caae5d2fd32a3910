"""pat_adjoint where the device's pool has no room for the weighted data: it needs the image only, as
it always did, and gives the same bits."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU, skipped there
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1707_02245_gb300 as P  # noqa: E402

DEV = torch.device("cuda:0")


class _PoolProps(ctypes.Structure):   # CUmemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("location_type", ctypes.c_int),
                ("location_id", ctypes.c_int), ("win32", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


def test_adjoint_in_a_pool_of_32_mib():
    from paper_1707_02245_gb300 import build
    build.build()
    P.load()
    n, n_det, n_t = 48, 8, (1 << 21) + 1          # 64 MiB of data
    a = 2 * np.pi * np.arange(n_det) / n_det
    det = np.stack([1.2 * np.cos(a), 1.2 * np.sin(a)], 1)
    g = P.Geometry(n, det, n_t, 0.0, 2.7 / n_t, 4)
    y = torch.randn(n_det, n_t, generator=torch.Generator(device=DEV).manual_seed(3), device=DEV)
    want, got = torch.empty(n, n, device=DEV), torch.full((n, n), float("nan"), device=DEV)
    P.pat_adjoint(g.handle, y, want)              # (also prepares the geometry)
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    dev, standard, pool = ctypes.c_int(), ctypes.c_void_p(), ctypes.c_void_p()
    assert cu.cuDeviceGet(ctypes.byref(dev), torch.cuda.current_device()) == 0
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(standard), dev) == 0
    props = _PoolProps(alloc_type=1, location_type=1, location_id=dev.value, max_size=32 << 20)
    assert cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) == 0
    assert cu.cuDeviceSetMemPool(dev, pool) == 0
    try:
        for _ in range(2):
            P.pat_adjoint(g.handle, y, got)
            torch.cuda.synchronize()
            assert torch.equal(got, want)
            got.fill_(float("nan"))
    finally:
        torch.cuda.synchronize()
        assert cu.cuDeviceSetMemPool(dev, standard) == 0
        assert cu.cuMemPoolDestroy(pool) == 0
    assert bool(want.any())
    g.close()
