"""The network at sizes where its layers run on the kernels that stage pixel tiles with their halo:
bfloat16 outputs, slices of the skip concatenation as inputs and outputs, and ReLU masks taken
with the bias sums.

A batch of images against the images one at a time, which are too few tiles for those kernels and
take the others (checked against the oracle elsewhere).  Every forward kernel adds the same products
in the same order, so outputs, and the input gradients between layers, have equal bits.  A layer's
weight and bias gradient of the batch is the sum over the images up to the order of FP32
additions: up to 2^-24 of a running sum for each of some thousand, of random signs, so a few 1e-6
of the gradient's norm; 5e-5 is allowed.  A mask, tile or channel out of place gives 1e-2 or more.
"""
import numpy as np
import pytest

from oracle import unet_oracle as U

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


@pytest.mark.parametrize("batch,h,w,base,levels", [(8, 128, 128, 32, 3), (7, 104, 72, 32, 2), (12, 72, 88, 16, 3), (24, 40, 56, 64, 2)])
def test_batch_matches_single_images(batch, h, w, base, levels):
    net = P.pat_unet_create(8, 8, base, levels, seed=base + levels)
    n = P.pat_unet_num_params(net)
    gen = torch.Generator(device=DEV).manual_seed(h + w)
    x = torch.randn(batch, h, w, 8, generator=gen, device=DEV).bfloat16()
    dy = torch.randn(batch, h, w, 8, generator=gen, device=DEV)
    y, grad = torch.full((batch, h, w, 8), float("nan"), device=DEV), torch.full((n,), float("nan"), device=DEV)
    P.pat_unet_forward(net, x, batch, h, w, y)
    P.pat_unet_backward(net, dy, grad)
    whole = grad.double()
    total = torch.zeros(n, dtype=torch.float64, device=DEV)
    for i in range(batch):
        yi = torch.full((1, h, w, 8), float("nan"), device=DEV)
        P.pat_unet_forward(net, x[i:i + 1].contiguous(), 1, h, w, yi)
        P.pat_unet_backward(net, dy[i:i + 1].contiguous(), grad)
        assert torch.equal(yi[0], y[i]), i
        total += grad.double()
    k = 0
    for name, co, ci in U.unet_layout(8, 8, base, levels):
        for part, size in (("weights", co * 9 * ci), ("bias", co)):
            a, b = whole[k:k + size], total[k:k + size]
            assert float((a - b).norm()) <= 5e-5 * float(b.norm()), (name, part)
            k += size
    assert k == n
    P.pat_unet_destroy(net)
    assert P.pat_nn_wait_timeouts() == 0
    assert np.isfinite(float(whole.norm()))
