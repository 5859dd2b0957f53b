"""Rounding of the BF16 network's weight and bias gradients as they are summed
over the pixels of a large batch.

With weights that pass three channels through, every operand of the gradients
is known: the layers' input is the network's (rounded to BF16), the output
gradient 2 (y - t) / n (rounded to BF16).  The sums over 524,288 pixels in 64
bits are then exact values for the library's, whose products are exact and
whose sums are FP32.  All operands are positive, so sums grow about evenly and
an addition acts on half the final size on average.  An accumulator of the
tensor cores takes at most 32 additions that may truncate a unit in the last
place (2^-23 of its size); its sums, and those of at most 152 splits, are added
with rounding (2^-24): 16 * 2^-23 + (152 + 16) / 2 * 2^-24 = 6.9e-6.  Without a
limit on the accumulators 32 channels gave 7.6e-6 and 64 channels 2.2e-5."""
import numpy as np
import pytest

from paper_2012_14707_gb300 import build as lbm_build
from paper_2012_14707_gb300 import lbm

pytestmark = pytest.mark.gpu

TOLERANCE = 16 * 2.0 ** -23 + (152 + 16) / 2 * 2.0 ** -24


@pytest.mark.parametrize("base,H,W,N", [(32, 256, 256, 8), (64, 256, 256, 8), (32, 248, 232, 8),
                                        (128, 64, 64, 8), (20, 120, 72, 8)])
def test_gradients_against_sums_in_64_bits(base, H, W, N):
    import torch

    lbm_build.build()
    torch.cuda.set_device(0)
    g = torch.Generator().manual_seed(5)
    x = torch.randn((N, H, W, 3), generator=g).abs() + 0.5
    t = -torch.randn((N, H, W, 3), generator=g).abs() - 0.3
    shapes = [(3, 3, 3, base), (base,), (3, 3, base, base), (base,), (1, 1, base, 3), (3,)]
    params = [np.zeros(s, np.float32) for s in shapes]
    for p in params[::2]:
        for k in range(3):
            p[p.shape[0] // 2, p.shape[1] // 2, k, k] = 1.0
    net = lbm.Net(H, W, base=base, levels=1, precision="bf16", max_batch=N)
    net.set_params(np.concatenate([p.reshape(-1) for p in params]))
    xd, td = x.cuda(), t.cuda()
    got, _ = net.gradients(xd.data_ptr(), td.data_ptr(), N)
    net.close()

    y = xd.to(torch.bfloat16).float()          # every layer's input and output
    gz = (2.0 * (y - td) / np.float32(N * H * W * 3)).to(torch.bfloat16).double()
    y = y.double()
    yp = torch.nn.functional.pad(y.permute(0, 3, 1, 2), (1, 1, 1, 1)).permute(0, 2, 3, 1)
    w3 = torch.stack([torch.stack([torch.einsum("nhwc,nhwo->co", yp[:, a:a + H, b:b + W], gz)
                                   for b in range(3)]) for a in range(3)])
    w1, db = torch.einsum("nhwc,nhwo->co", y, gz)[None, None], gz.sum((0, 1, 2))
    off = 0
    for s, want in zip(shapes, (w3, db, w3, db, w1, db)):
        a = got[off:off + int(np.prod(s))].reshape(s).astype(np.float64)
        off += a.size
        a = a[..., :3, :3] if a.ndim == 4 else a[:3]
        want = want.cpu().numpy()
        assert np.abs(a / want - 1.0).max() <= TOLERANCE, (s, np.abs(a / want - 1.0).max())
