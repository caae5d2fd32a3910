"""K^T of a batch whose CTAs take several work items of a tile: the fixed-point sums are integers,
so a problem's solve has the bits it has alone, where every CTA takes one item."""
import pytest

import synthetic as S

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


# sets of (n, detectors, radius of their circle, samples) and how many of each: few heavy tiles cut
# into many items, one tile, more tiles than items, rays in every direction, empty work lists
@pytest.mark.parametrize("geoms,copies", [([(64, 64, 1.2, 127)], 24), ([(32, 40, 1.2, 65)], 150),
                                          ([(64, 48, 0.5, 96), (200, 9, 1.2, 301), (33, 4, 0.3, 21), (2, 1, 1.2, 1)], 12)])
@pytest.mark.parametrize("model", [dict(reg=0), dict(reg=3, wavelet_kind=1, wavelet_levels=1)])
def test_batched_adjoint_has_the_bits_of_a_single_one(geoms, copies, model):
    if model["reg"] == 3 and len(geoms) > 1:   # (a wavelet batch has one N)
        geoms = geoms[:1]
    gs, fs = [], []
    gen = torch.Generator().manual_seed(len(geoms) + copies)
    for n, n_det, radius, n_t in geoms:
        det = S.detectors_full_circle(n_det, radius)
        r0, dr = S.radial_sampling(det, n_t)
        gs.append(P.Geometry(n, det, n_t, r0, dr, 128))
        fs.append((0.1 * torch.randn(n_det, n_t, generator=gen)).to(DEV))
    prm = P.make_params(alpha=0.01, iters=6, gap_every=3, **model)
    alone = []
    for g, f in zip(gs, fs):
        alone.append(torch.empty(g.n, g.n, device=DEV))
        P.pat_reconstruct(g.handle, f, prm, alone[-1])
        assert bool(alone[-1].any()) or g.n == 2
    k = len(gs) * copies
    us = [torch.full_like(alone[i % len(gs)], float("nan")) for i in range(k)]
    P.pat_reconstruct_batched([gs[i % len(gs)].handle for i in range(k)], [fs[i % len(gs)] for i in range(k)], [prm] * k, us)
    for i, u in enumerate(us):
        assert torch.equal(u, alone[i % len(gs)]), i
    for g in gs:
        g.close()
