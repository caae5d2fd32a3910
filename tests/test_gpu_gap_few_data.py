"""The duality gap where the data give K few CTAs and the image is large: the pixel terms are then
spread over CTAs that take pixels only, so that no thread adds up a long FP32 chain.

The states make every pixel's term the same number (columns alternate between 0 and c), whose
chain of 1024 FP32 additions drifts by 1e-5.  Bound: a thread adds at most 8 pixels (7 roundings
of 2^-24), a term takes a difference, two squares, their sum and a root (4 more), and what follows
carries 48 bits: 11 * 2^-24 = 6.6e-7 of the term's sum, 8e-7 with the data terms, which are far smaller.
"""
import numpy as np
import pytest

import synthetic as S
from oracle import pat_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU, skipped there
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1707_02245_gb300 as P  # noqa: E402

DEV = torch.device("cuda:0")
BOUND = 8e-7


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1707_02245_gb300 import build
    build.build()
    P.load()


def _geometry(n, n_det, n_t, m=64):
    det = S.detectors_full_circle(n_det, 1.2)
    r0, dr = S.radial_sampling(det, n_t)
    return (P.Geometry(n, det, n_t, r0, dr, m),
            O.Geometry(n=n, det_xy=det, n_t=n_t, r0=r0, dr=dr, quad_m=m))


# n, detectors, samples, K variant: the global variant, slabs of 3 CTAs and one slab per SM with its
# wider CTAs, each with clusters of pixels only; and a plan that fills the GPU by itself
@pytest.mark.parametrize("n,n_det,n_t,fwd", [(1024, 1, 16, P.PAT_FWD_AUTO), (1023, 1, 8, P.PAT_FWD_AUTO),
                                             (256, 1, 16, P.PAT_FWD_AUTO), (300, 2, 9, P.PAT_FWD_SLAB_ONE),
                                             (64, 1, 1, P.PAT_FWD_AUTO), (64, 64, 96, P.PAT_FWD_AUTO)])
@pytest.mark.parametrize("reg", [0, 1, 2])
def test_gap_terms_of_equal_pixels(n, n_det, n_t, fwd, reg):
    g, og = _geometry(n, n_det, n_t)
    if fwd != P.PAT_FWD_AUTO:
        P.pat_geometry_set_shapes(g.handle, forward=fwd)
    c = 0.1
    u = np.tile(np.where(np.arange(n) % 2 == 0, 0.0, c).astype(np.float32), (n, 1))
    r = np.zeros((2, n, n), np.float32)
    r[0] = np.tile(np.where(np.arange(n) % 2 == 0, -c, c).astype(np.float32), (n, 1)) / 4
    v, s = np.zeros((2, n, n), np.float32), np.zeros((3, n, n), np.float32)
    xi = np.zeros((2, n, n), np.float32)
    xi[0] = 1.0
    f = (0.01 * np.random.default_rng(n).standard_normal((n_det, n_t))).astype(np.float32)
    q = np.zeros(n_det * n_t, np.float32)
    pb = O.problem_from_geometry(og, f.astype(np.float64), reg=(O.REG_TV, O.REG_TGV, O.REG_DTV)[reg], alpha=1.0, beta=2.0,
                                 gamma=0.5, xi=xi.astype(np.float64) if reg == 2 else None)
    d = lambda a: a.astype(np.float64)  # noqa: E731
    ref = O.duality_gap(pb, d(u), d(q), d(r), d(v) if reg == 1 else None, d(s) if reg == 1 else None)
    tgv = reg == 1
    x = np.concatenate([u.ravel()] + ([v.ravel()] if tgv else []))
    y = np.concatenate([q, r.ravel()] + ([s.ravel()] if tgv else []))
    prm = P.make_params(reg=reg, alpha=1.0, beta=2.0, gamma=0.5, xi=torch.from_numpy(xi).to(DEV) if reg == 2 else None)
    got = P.pat_duality_gap(g.handle, torch.from_numpy(f).to(DEV), prm, torch.from_numpy(x).to(DEV), torch.from_numpy(y).to(DEV))
    assert abs(got["primal"] - ref["primal"]) <= BOUND * abs(ref["primal"])
    assert abs(got["dual"] - ref["dual"]) <= BOUND * abs(ref["dual"])
    g.close()


def test_few_data_in_a_batch():
    """Problems with and without CTAs of pixels only in one launch, on both a cluster size of their
    own and a shared one: a solve's result does not depend on its company."""
    probs = [_geometry(*a) for a in ((512, 1, 16), (384, 64, 96), (256, 2, 16), (256, 64, 96), (64, 1, 9), (400, 2, 8))]
    fs = [0.1 * torch.randn(o.n_det, o.n_t, generator=torch.Generator().manual_seed(i)).to(DEV) for i, (_, o) in enumerate(probs)]
    prm = [P.make_params(reg=i % 2, alpha=0.01, iters=20, gap_every=5) for i in range(len(probs))]
    alone, us = [], []
    for (g, o), f, p in zip(probs, fs, prm):
        us.append(torch.empty(o.n, o.n, device=DEV))
        alone.append(P.pat_reconstruct(g.handle, f, p, us[-1]))
    ub = [torch.empty_like(u) for u in us]
    infos = P.pat_reconstruct_batched([g.handle for g, _ in probs], fs, prm, ub)
    for a, b, u, v in zip(alone, infos, us, ub):
        assert torch.equal(u, v)
        for k in ("primal", "dual", "residual"):
            assert abs(a[k] - b[k]) <= 1e-6 * abs(a[k]), k
        assert a["iters_done"] == b["iters_done"] == 20
    for g, _ in probs:
        g.close()
