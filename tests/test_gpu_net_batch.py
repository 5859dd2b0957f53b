"""The BF16 network's persistent kernels on batches that give every CTA several
tiles, against the same images one at a time, which give it one or two.

On 152 SMs the shapes reach: weights kept for all tiles and weights in a ring
that runs on from tile to tile, tiles of one and of two pixel blocks with 16 to
128 output channels, two image stages and one, inputs too wide for shared
memory at once, images that are not whole tiles, and up to 34 tiles in a split
of the weight gradient.

Forward: the order of the sums does not depend on the tiling, so the bits are
those of the images alone.  Gradients: the loss is a mean, and 1/N of a power
of two scales every stored BF16 gradient exactly; so a batch's gradient is the
mean of its images' up to FP32 rounding of the sums, of order 1e-6 of a layer's
gradient.  A pixel lost or taken twice would change it by 1e-3 and more (one of
at most 5e5 terms of random sign), and the tolerance is 1e-4."""
import numpy as np
import pytest

from paper_2012_14707_gb300 import build as lbm_build
from paper_2012_14707_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base,levels,H,W,N", [
    (32, 4, 248, 232, 8), (96, 2, 72, 88, 8), (128, 2, 120, 136, 4), (512, 1, 40, 64, 4)])
def test_batch_is_its_images(base, levels, H, W, N):
    import torch

    lbm_build.build()
    torch.cuda.set_device(0)
    g = torch.Generator().manual_seed(base + H)
    x = torch.randn((N, H, W, 3), generator=g).cuda()
    t = torch.randn((N, H, W, 3), generator=g).cuda()
    y = torch.full((N, H, W, 3), float("nan"), device="cuda")
    one = torch.full((1, H, W, 3), float("nan"), device="cuda")
    net = lbm.Net(H, W, base=base, levels=levels, precision="bf16", max_batch=N, seed=11)
    p = net.get_params()
    rng = np.random.default_rng(5)
    net.set_params(p + (rng.standard_normal(p.size) * 0.02 * (p == 0)).astype(np.float32))  # biases
    net.forward(x.data_ptr(), N, y.data_ptr())
    assert torch.isfinite(y).all()
    whole, loss = net.gradients(x.data_ptr(), t.data_ptr(), N)
    parts, losses = [], []
    for k in range(N):
        net.forward(x[k:k + 1].contiguous().data_ptr(), 1, one.data_ptr())
        assert torch.equal(one[0], y[k]), k
        gk, lk = net.gradients(x[k:k + 1].contiguous().data_ptr(),
                               t[k:k + 1].contiguous().data_ptr(), 1)
        parts.append(gk.astype(np.float64))
        losses.append(lk)
    net.close()
    assert loss == pytest.approx(np.mean(losses), rel=1e-6)
    mean = np.mean(parts, axis=0)
    # layer by layer: weights, biases
    chans, prev = [], 3
    for l in range(levels):
        chans += [(3, prev, base << l), (3, base << l, base << l)]
        prev = base << l
    for l in range(levels - 2, -1, -1):
        chans += [(3, 3 * (base << l), base << l), (3, base << l, base << l)]
    chans.append((1, base, 3))
    off = 0
    for ks, ci, co in chans:
        for size in (ks * ks * ci * co, co):
            a, b = whole[off:off + size], mean[off:off + size]
            off += size
            assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b), (ks, ci, co, size)
    assert off == whole.size
