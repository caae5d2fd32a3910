"""K^T where radius indexes lie beyond 2^24, which FP32 does not hold exactly: the kernel's positions
and arc weights are those of the integer index, as in K.

Bound: K and K^T evaluate the same FP32 positions and taps, so <K u, y> and <u, K^T y> differ by the
rounding of K's rows (a few 2^-24) and of K^T's fixed-point sums (2^-30 of the largest sum per
point, 40 000 points: 4e-5 of it at most); 1e-4 of the norms' product is allowed.
"""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU, skipped there
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1707_02245_gb300 as P  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1707_02245_gb300 import build
    build.build()
    P.load()


@pytest.mark.parametrize("exponent", [24, 25])
def test_adjoint_of_rows_past_exact_indexes(exponent):
    n, m, dist = 32, 16, 2000.0
    n_t = (1 << exponent) + 20001
    phi = 2 * math.pi * 0.5 / m
    det = np.array([[-dist * math.cos(phi), -dist * math.sin(phi)]])
    g = P.Geometry(n, det, n_t, 0.0, dist / (1 << exponent), m)
    gen = torch.Generator(device=DEV).manual_seed(exponent)
    u = torch.rand(n, n, generator=gen, device=DEV) + 0.5
    y = torch.randn(1, n_t, generator=gen, device=DEV)
    ku = torch.empty(1, n_t, device=DEV)
    kty, kty2 = torch.empty(n, n, device=DEV), torch.empty(n, n, device=DEV)
    P.pat_forward(g.handle, u, ku)
    P.pat_adjoint(g.handle, y, kty)
    P.pat_adjoint_noalloc(g.handle, y, kty2)
    torch.cuda.synchronize()
    assert int((ku != 0).sum()) > 10000
    assert bool((ku[0, (1 << exponent) + 10:] != 0).any())
    hit = ku[0] != 0
    scale = float(ku.double().norm() * (y[0] * hit).double().norm())
    lhs, rhs = float((ku.double() * y).sum()), float((u.double() * kty).sum())
    assert abs(lhs - rhs) <= 1e-4 * scale, (lhs, rhs, scale)
    # data premultiplied by the arc weights, and weighted in the kernel
    assert torch.equal(kty, kty2)
    g.close()
