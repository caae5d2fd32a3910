"""Where the solves' device memory comes from: from the pool that the application has set for the
device, if it has set one, else from a pool of the library's own, whose kept memory is given back
with the last geometry."""
import ctypes
import os
import subprocess
import sys

import pytest

import synthetic as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU, skipped there
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1707_02245_gb300 as P  # noqa: E402

DEV = torch.device("cuda:0")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MODELS = [dict(reg=0), dict(reg=1), dict(reg=3, wavelet_kind=0, wavelet_levels=2), dict(reg=3, wavelet_kind=1, wavelet_levels=2)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1707_02245_gb300 import build
    build.build()
    P.load()


class _PoolProps(ctypes.Structure):   # CUmemPoolProps
    _fields_ = [("alloc_type", ctypes.c_int), ("handle_types", ctypes.c_int), ("location_type", ctypes.c_int),
                ("location_id", ctypes.c_int), ("win32", ctypes.c_void_p), ("max_size", ctypes.c_size_t),
                ("usage", ctypes.c_ushort), ("reserved", ctypes.c_ubyte * 54)]


def test_solves_use_the_application_s_pool():
    cu = ctypes.CDLL("libcuda.so.1")
    USED_CURRENT, USED_HIGH = 7, 8     # CU_MEMPOOL_ATTR_USED_MEM_CURRENT / _HIGH
    det = S.detectors_full_circle(16, 1.2)
    r0, dr = S.radial_sampling(det, 96)
    g = P.Geometry(128, det, 96, r0, dr, 64)
    f = 0.1 * torch.randn(16, 96, generator=torch.Generator().manual_seed(1)).to(DEV)
    us = [torch.empty(128, 128, device=DEV) for _ in MODELS]

    def solve(i):
        P.pat_reconstruct(g.handle, f, P.make_params(alpha=0.02, iters=4, **MODELS[i]), us[i])
        return us[i].clone()

    before = [solve(i) for i in range(len(MODELS))]
    dev, standard, pool, v = ctypes.c_int(), ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_uint64()
    assert cu.cuDeviceGet(ctypes.byref(dev), torch.cuda.current_device()) == 0
    assert cu.cuDeviceGetDefaultMemPool(ctypes.byref(standard), dev) == 0
    props = _PoolProps(alloc_type=1, location_type=1, location_id=dev.value)   # pinned, on the device
    assert cu.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(props)) == 0
    assert cu.cuDeviceSetMemPool(dev, pool) == 0
    try:
        for i in range(len(MODELS)):
            zero = ctypes.c_uint64(0)
            assert cu.cuMemPoolSetAttribute(pool, USED_HIGH, ctypes.byref(zero)) == 0
            assert torch.equal(solve(i), before[i])
            assert cu.cuMemPoolGetAttribute(pool, USED_HIGH, ctypes.byref(v)) == 0
            assert v.value >= 8 * 128 * 128 * 4, (MODELS[i], v.value)   # of the workspace's many images
        torch.cuda.synchronize()
        assert cu.cuMemPoolGetAttribute(pool, USED_CURRENT, ctypes.byref(v)) == 0 and v.value == 0
    finally:
        torch.cuda.synchronize()
        assert cu.cuDeviceSetMemPool(dev, standard) == 0
        assert cu.cuMemPoolDestroy(pool) == 0
    assert torch.equal(solve(0), before[0])
    g.close()


def test_last_geometry_gives_the_kept_memory_back():
    """In a process of its own, where no other geometry lives."""
    code = r"""
import torch, synthetic as S, paper_1707_02245_gb300 as P
det = S.detectors_full_circle(16, 1.2)
r0, dr = S.radial_sampling(det, 96)
gs = [P.Geometry(384, det, 96, r0, dr, 64) for _ in range(2)]
f = 0.1 * torch.randn(16, 96, device="cuda:0")
u = torch.empty(384, 384, device="cuda:0")
def solve(g):
    P.pat_reconstruct(g.handle, f, P.make_params(reg=1, alpha=0.02, iters=4), u)
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]
for g in gs:
    solve(g)
kept = solve(gs[0])
gs[1].close()
one = solve(gs[0])
assert one >= kept
gs[0].close()
free = torch.cuda.mem_get_info()[0]
assert free >= one + 8 * 384 * 384 * 4, (kept, one, free)
print("given back")
"""
    env = dict(os.environ, PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "given back" in r.stdout, r.stdout + r.stderr
