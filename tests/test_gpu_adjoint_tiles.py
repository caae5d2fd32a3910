"""K^T at the edges of its pixel tiles and ray segments, against the FP64 oracle.

Tiles have a side of 32 pixels, a warp walks four segments in pairs of points, and the data
rows inside a reconstruction are padded to an even length.  So: image sides around multiples
of the tile, odd numbers of samples (the last pair is half
padding), segments shorter and longer than a warp's step, detectors inside the image (rays
in every direction through one tile) and a single datum.

Bounds: a point's FP32 position is off by a few 1e-5 pixel at these sizes, so the weights are
off by as much of 1 and the image by less than 1e-4 of its norm.
"""
import numpy as np
import pytest

import synthetic as S
from oracle import pat_oracle as O
from tests.problems import rel_l2

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


# n, detectors, radius of their circle, samples, angles
CASES = [(2, 1, 1.2, 1, 16), (31, 3, 1.2, 17, 48), (32, 5, 1.2, 33, 64), (33, 4, 0.5, 21, 200), (65, 2, 1.2, 301, 96),
         (192, 3, 1.2, 95, 64), (193, 3, 1.2, 385, 64), (200, 2, 0.4, 51, 128), (64, 140, 1.2, 255, 256),
         (96, 330, 0.9, 97, 256)]


@pytest.mark.parametrize("n,n_det,radius,n_t,m", CASES)
def test_adjoint_tile_edges(n, n_det, radius, n_t, m):
    det = S.detectors_full_circle(n_det, radius)
    r0, dr = S.radial_sampling(det, n_t)
    g = P.Geometry(n, det, n_t, r0, dr, m)
    og = O.Geometry(n=n, det_xy=det, n_t=n_t, r0=r0, dr=dr, quad_m=m)
    y = np.random.default_rng(n + n_t).standard_normal((n_det, n_t)).astype(np.float32)
    # an array off the 8-byte boundary, as a caller may pass
    buf = torch.empty(y.size + 1, device=DEV)
    buf[1:] = torch.from_numpy(y.ravel()).to(DEV)
    u = torch.empty(n, n, device=DEV)
    P.pat_adjoint(g.handle, buf[1:], u)
    ref = O.adjoint(og, y.astype(np.float64))
    assert rel_l2(u.cpu().numpy(), ref) <= 1e-4
    u2 = torch.empty(n, n, device=DEV)
    P.pat_adjoint_noalloc(g.handle, buf[1:], u2)
    assert torch.equal(u, u2)
    # inside a reconstruction: the data rows K writes for K^T, padded to an even length
    uo = torch.empty(n, n, device=DEV)
    P.pat_reconstruct(g.handle, torch.from_numpy(y).to(DEV), P.make_params(reg=P.PAT_TV, alpha=0.05, iters=3), uo)
    res = O.pdhg(O.problem_from_geometry(og, y.astype(np.float64), reg=O.REG_TV, alpha=0.05), 3, gap_every=0)
    assert rel_l2(uo.cpu().numpy(), res.u) <= 1e-3
    g.close()
