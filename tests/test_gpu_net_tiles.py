"""The BF16 network's tensor-core convolutions where their tiling can go
wrong: images that are not whole tiles, channel counts that are not whole
16s or 8s, one level (no decoder), inputs of more channels than fit in shared
memory at once, tiles too few or many for the GPU.  Against the FP64
reference; tolerances are those of the full-width BF16 tests (8 significant
bits per stored activation and gradient)."""
import numpy as np
import pytest

from oracle import nn
from paper_2012_14707_gb300 import build as lbm_build
from paper_2012_14707_gb300 import lbm

pytestmark = pytest.mark.gpu

SHAPES = [  # base, levels, H, W, batch
    (8, 1, 5, 3, 1), (8, 1, 16, 8, 2), (5, 2, 10, 34, 3), (12, 3, 20, 44, 1), (20, 2, 34, 18, 2),
    (512, 1, 6, 10, 1), (32, 2, 66, 130, 1), (48, 3, 24, 40, 1), (64, 4, 16, 24, 1), (8, 3, 256, 260, 2),
]


def bf(v):
    """v rounded to BF16 (nearest even), as float64."""
    u = np.asarray(v, np.float32).view(np.uint32).astype(np.uint64)
    u = (u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000
    return u.astype(np.uint32).view(np.float32).astype(np.float64)


def network_bf16(p, x, t, levels, switch=0.0):
    """(y, gradients) with BF16 storage, p in FP32; in the backward pass a
    ReLU is open where its input exceeds `switch` times the layer's r.m.s."""
    w = {k: bf(v) if k.endswith(".w") else v for k, v in p.items()}
    conv = {}

    def layer(name, h, first=nn.conv3x3):
        z = first(h, w[name + ".w"], w[name + ".b"])
        conv[name] = (h, z > switch * np.sqrt((z * z).mean()))
        return bf(np.maximum(z, 0.0))

    h, skips = bf(x), []
    for l in range(levels):
        if l:
            h = bf(nn.pool2(h))
        h = layer(f"e{l}b", layer(f"e{l}a", h))
        skips.append(h)
    for l in range(levels - 2, -1, -1):
        h = layer(f"d{l}b", layer(f"d{l}a", np.concatenate([nn.up2(h), skips[l]], axis=3)))
    y = bf(nn.conv1x1(h, w["head.w"], w["head.b"]))

    g = {}

    def back(name, gz):
        gx, g[name + ".w"], g[name + ".b"] = nn.conv3x3_backward(conv[name][0], w[name + ".w"], gz)
        return bf(gx)

    gy = bf(2.0 * (y - t) / y.size)
    gx, g["head.w"], g["head.b"] = nn.conv1x1_backward(h, w["head.w"], gy)
    top = "d0b" if levels > 1 else "e0b"
    gh = bf(gx) * conv[top][1]
    gskip = {}
    for l in range(levels - 1):
        ga = back(f"d{l}b", gh) * conv[f"d{l}a"][1]
        gc = back(f"d{l}a", ga)
        cu = gc.shape[3] - skips[l].shape[3]
        gskip[l] = gc[..., cu:]
        below = f"d{l + 1}b" if l + 1 <= levels - 2 else f"e{levels - 1}b"
        gh = bf(nn.up2_backward(gc[..., :cu])) * conv[below][1]
    for l in range(levels - 1, -1, -1):
        if l < levels - 1:
            gh = bf(nn.pool2_backward(gp) + gskip[l]) * conv[f"e{l}b"][1]
        ga = back(f"e{l}b", gh) * conv[f"e{l}a"][1]
        gp = back(f"e{l}a", ga)
    return y, g


@pytest.mark.parametrize("base,levels,H,W,N", SHAPES)
def test_bf16_network_of_awkward_shape_matches_reference(base, levels, H, W, N):
    import torch

    lbm_build.build()
    torch.cuda.set_device(0)
    rng = np.random.default_rng(base * 1000 + H)
    p = nn.init_params(7, base=base, levels=levels)
    for k in p:
        if k.endswith(".b"):
            p[k] = rng.standard_normal(p[k].shape) * 0.05
        p[k] = p[k].astype(np.float32).astype(np.float64)
    x = rng.standard_normal((N, H, W, 3)).astype(np.float32).astype(np.float64)
    t = rng.standard_normal((N, H, W, 3)).astype(np.float32).astype(np.float64)
    y_ref, g_ref = network_bf16(p, x, t, levels)
    g_hi, g_lo = (network_bf16(p, x, t, levels, d)[1] for d in (1.1e-3, -1.1e-3))
    names = [(n + s) for n, *_ in nn.layer_shapes(3, 3, base, levels) for s in (".w", ".b")]
    net = lbm.Net(H, W, base=base, levels=levels, precision="bf16", max_batch=N + 1)
    net.set_params(np.concatenate([p[n].reshape(-1) for n in names]))
    xd = torch.tensor(x, dtype=torch.float32, device="cuda")
    td = torch.tensor(t, dtype=torch.float32, device="cuda")
    yd = torch.empty((N, H, W, 3), dtype=torch.float32, device="cuda")
    net.forward(xd.data_ptr(), N, yd.data_ptr())
    y = yd.cpu().numpy()
    assert np.linalg.norm(y - y_ref) <= 1e-2 * np.linalg.norm(y_ref)
    g, loss = net.gradients(xd.data_ptr(), td.data_ptr(), N)
    g2, _ = net.gradients(xd.data_ptr(), td.data_ptr(), N)
    assert np.array_equal(g, g2)  # sums in a fixed order
    assert loss == pytest.approx(nn.mse(y_ref, t), rel=1e-2)
    off = 0
    for n in names:
        b = g_ref[n].reshape(-1)
        a = g[off:off + b.size]
        off += b.size
        switches = np.linalg.norm(g_hi[n] - g_lo[n])
        assert np.linalg.norm(a - b) <= 1e-2 * np.linalg.norm(b) + switches + 1e-12, n
    net.close()


def test_weights_are_packed_again_after_they_change():
    import torch

    lbm_build.build()
    torch.cuda.set_device(0)
    H, W = 16, 24
    rng = np.random.default_rng(3)
    xd = torch.tensor(rng.standard_normal((1, H, W, 3)), dtype=torch.float32, device="cuda")
    td = torch.tensor(rng.standard_normal((1, H, W, 3)), dtype=torch.float32, device="cuda")
    ys = []
    net = lbm.Net(H, W, base=8, levels=2, precision="bf16", max_batch=1, seed=1)
    fresh = lbm.Net(H, W, base=8, levels=2, precision="bf16", max_batch=1, seed=2)
    for step in range(3):
        y = torch.empty((1, H, W, 3), device="cuda")
        z = torch.empty((1, H, W, 3), device="cuda")
        net.forward(xd.data_ptr(), 1, y.data_ptr())
        fresh.set_params(net.get_params())
        fresh.forward(xd.data_ptr(), 1, z.data_ptr())
        assert torch.equal(y, z)
        ys.append(y)
        net.train_step(xd.data_ptr(), td.data_ptr(), 1, 1e-2)
    assert not torch.equal(ys[0], ys[1]) and not torch.equal(ys[1], ys[2])
