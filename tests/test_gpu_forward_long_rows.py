"""K of a detector with more than 2^18 radii (groups of 8 radii beyond the 16 bits a work unit once
kept for them) against the FP64 oracle.  Bound: positions are off by a few 1e-5 pixel at this
distance, so the taps' weights by as much of 1 and the rows by less than 1e-4 of their norm."""
import numpy as np
import pytest

from oracle import pat_oracle as O
from tests.problems import rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU, skipped there
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1707_02245_gb300 as P  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n,n_t", [(32, 300001), (400, 600003)])   # slabs and the global variant
def test_forward_of_long_rows(n, n_t):
    from paper_1707_02245_gb300 import build
    build.build()
    P.load()
    det = -2.0 * np.array([[np.cos(np.pi / 8), np.sin(np.pi / 8)]])   # one of the 8 angles points at the centre
    dr = 3.1 / n_t
    g = P.Geometry(n, det, n_t, 0.0, dr, 8)
    u = np.random.default_rng(n).uniform(0.5, 1.5, (n, n)).astype(np.float32)
    y = torch.full((1, n_t), float("nan"), device=DEV)
    P.pat_forward(g.handle, torch.from_numpy(u).to(DEV), y)
    ref = O.forward(O.Geometry(n=n, det_xy=det, n_t=n_t, r0=0.0, dr=dr, quad_m=8), u.astype(np.float64)).reshape(-1)
    got = y.cpu().numpy().reshape(-1).astype(np.float64)
    assert np.count_nonzero(ref[1 << 18:]) > 10000
    assert rel_l2(got, ref) <= 1e-4
    assert rel_l2(got[1 << 18:], ref[1 << 18:]) <= 1e-4
    g.close()
