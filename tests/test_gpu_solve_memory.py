"""The solves' device memory is kept between calls and not cleared, so a solve must not depend on
what an earlier one left there: after a solve on data that are not numbers, every model gives the
bits it gave before, alone, in a batch and from several threads at once."""
import threading

import numpy as np
import pytest

import synthetic as S

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - collected on CPU, skipped there
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1707_02245_gb300 as P  # noqa: E402

DEV = torch.device("cuda:0")
MODELS = [dict(reg=0), dict(reg=1, beta=2.0), dict(reg=2), dict(reg=3, wavelet_kind=0, wavelet_levels=3),
          dict(reg=3, wavelet_kind=1, wavelet_levels=3)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_1707_02245_gb300 import build
    build.build()
    P.load()


@pytest.mark.parametrize("n,n_t", [(48, 95), (136, 271)])
def test_dirty_memory_does_not_reach_a_solve(n, n_t):
    w = S.workload_warm(5, n=n, n_det=24)
    g = P.Geometry(n, w["det_xy"], n_t, w["r0"], w["dr"], w["quad_m"])
    gen = torch.Generator(device=DEV).manual_seed(n)
    f = torch.randn(24, n_t, generator=gen, device=DEV) * 0.1
    nan = torch.full_like(f, float("nan"))
    xi = torch.randn(n, n, 2, generator=gen, device=DEV)
    xi = (xi / xi.norm(dim=2, keepdim=True)).permute(2, 0, 1).contiguous()

    def spoil(m, b=0, stream=None):
        with pytest.raises(P.PatError, match="not finite"):
            solve(m, nan, b, stream)

    def solve(m, data, b=0, stream=None):
        p = [P.make_params(alpha=0.02, iters=12, gap_every=5, xi=xi if m["reg"] == 2 else None, **m) for _ in range(b or 1)]
        u = [torch.full((n, n), float("nan"), device=DEV) for _ in range(b or 1)]
        if b:
            P.pat_reconstruct_batched([g.handle] * b, [data] * b, p, u, stream)
        else:
            P.pat_reconstruct(g.handle, data, p[0], u[0], stream)
        torch.cuda.synchronize()
        return torch.stack(u).cpu()

    clean = [solve(m, f) for m in MODELS]
    assert all(bool(torch.isfinite(c).all()) for c in clean)
    for m, c in zip(MODELS, clean):
        for dirty in MODELS:
            spoil(dirty)
        assert torch.equal(solve(m, f), c)
        spoil(dict(reg=1), b=3)
        assert torch.equal(solve(m, f, b=3), c.expand(3, n, n))
    got = [None] * len(MODELS)

    def work(i):
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        for _ in range(3):
            spoil(MODELS[(i + 1) % len(MODELS)], stream=s)
            got[i] = solve(MODELS[i], f, stream=s)

    ts = [threading.Thread(target=work, args=(i,)) for i in range(len(MODELS))]
    [t.start() for t in ts]
    [t.join() for t in ts]
    assert all(x is not None and torch.equal(x, c) for x, c in zip(got, clean))
    g.close()
