"""The convolution kernel that stages pixel tiles with their halo (32, 64 or 96 input channels on
images with enough 8 x 16 tiles), at the edges of its tiles: image sides just below, at and
above multiples of 8 and 16, output channels that fill one N tile, spill into a second or
leave one partly empty, and an output pointer off the 32-byte boundary its wide stores need.

Bound: products of bfloat16 values are exact in FP32 and the sum has 9 cin terms, accumulated
with an error below 2e-5 of the sum of their magnitudes (the bound of the other convolution
tests).
"""
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


@pytest.mark.parametrize("b,h,w,cin,cout,relu,shift", [
    (80, 15, 15, 32, 8, False, 0), (40, 16, 17, 32, 32, True, 0), (40, 17, 16, 32, 96, True, 4), (20, 33, 31, 64, 64, False, 4),
    (3, 97, 129, 64, 104, True, 0), (30, 16, 40, 64, 192, False, 0), (25, 31, 25, 96, 40, True, 0), (2, 160, 130, 96, 64, False, 4),
])
def test_halo_convolution_edges(b, h, w, cin, cout, relu, shift):
    g = torch.Generator(device=DEV).manual_seed(b + h + cin + cout)
    x = torch.randn(b, h, w, cin, generator=g, device=DEV).bfloat16()
    wt = (torch.randn(cout, 3, 3, cin, generator=g, device=DEV) / (3 * cin ** 0.5)).bfloat16()
    bias = torch.randn(cout, generator=g, device=DEV)
    buf = torch.full((b * h * w * cout + shift,), float("nan"), device=DEV)
    P.pat_conv3x3_forward(x, b, h, w, cin, wt, bias, cout, relu, buf[shift:])
    y = buf[shift:].reshape(b, h, w, cout)
    xd, wd = x.double().permute(0, 3, 1, 2), wt.double().permute(0, 3, 1, 2)
    conv = torch.nn.functional.conv2d
    ref = conv(xd, wd, bias.double(), padding=1)
    mag = conv(xd.abs(), wd.abs(), bias.double().abs(), padding=1)
    if relu:
        ref = ref.clamp(min=0)
    err = (y.double().permute(0, 3, 1, 2) - ref).abs()
    assert bool((err <= 2e-5 * mag).all()), float((err / mag).max())
    assert P.pat_nn_wait_timeouts() == 0


@pytest.mark.parametrize("b,h,w,cin,cout", [
    (90, 15, 15, 32, 32), (40, 17, 33, 32, 64), (20, 33, 31, 32, 128), (24, 25, 47, 64, 32), (10, 63, 65, 64, 64),
    (40, 9, 16, 96, 64), (13, 40, 49, 192, 64), (20, 24, 32, 128, 32),
    (2, 16, 16, 128, 128), (1, 9, 8, 160, 128), (3, 8, 9, 192, 192),   # other kernels, 4, 2 and 1 warps per sum of splits
    (90, 15, 15, 8, 32), (40, 17, 33, 32, 8), (24, 33, 31, 16, 24), (40, 24, 32, 64, 16), (28, 31, 41, 24, 128),
])
def test_halo_weight_gradient_edges(b, h, w, cin, cout):
    """The weight gradient of the wide layers: ragged pixel tiles of 16 x 8, one to three channel
    boxes of 32 or 64, fewer than 32 channels on either side, every width of the accumulators, and
    a last CTA with fewer tiles."""
    g = torch.Generator(device=DEV).manual_seed(h + w + cin + cout)
    x = torch.randn(b, h, w, cin, generator=g, device=DEV).bfloat16()
    dy = torch.randn(b, h, w, cout, generator=g, device=DEV).bfloat16()
    dw = torch.full((cout, 3, 3, cin), float("nan"), device=DEV)
    db = torch.full((cout,), float("nan"), device=DEV)
    P.pat_conv3x3_backward_weight(x, dy, b, h, w, cin, cout, dw, db)

    def reference(a, d):
        p = torch.nn.functional.pad(a.double(), (0, 0, 1, 1, 1, 1))
        d = d.double().reshape(-1, cout)
        return torch.stack([torch.stack([d.T @ p[:, i:i + h, j:j + w].reshape(-1, cin) for j in range(3)], 1)
                            for i in range(3)], 1)

    assert bool(((dw.double() - reference(x, dy)).abs() <= 2e-5 * reference(x.abs(), dy.abs())).all())
    assert bool(((db.double() - dy.double().sum((0, 1, 2))).abs() <= 2e-5 * dy.double().abs().sum((0, 1, 2))).all())
    assert P.pat_nn_wait_timeouts() == 0
