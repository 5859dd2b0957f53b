"""Steps launched as a chain (each step's launch overlaps its predecessor's
tail) give bitwise the state of the same steps taken one at a time with a
synchronisation between them."""
import numpy as np
import pytest

from paper_2012_14707_gb300 import build as lbm_build
from paper_2012_14707_gb300 import cases, lbm

pytestmark = pytest.mark.gpu

CASES2 = {
    "channel_4x32": lambda: cases.config_poiseuille(),
    "lid_37x9": lambda: cases.channel(37, 9, 0.2, 0.85, Kn=0.05, ax=1e-6, u_top=0.01),
    "cylinders_300x150": lambda: cases.cylinder_array(300, 150, 1),
    "box_70x45": lambda: cases.periodic_box(70, 45, ax=1e-5),
}
CASES3 = {
    "lid_3d": lambda: cases.channel3d(13, 10, 9, 0.35, 0.8, 0.05, u_top=0.01),
    "spheres_3d": lambda: cases.sphere_array3d(20, 4),
}


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16", "fp16"])
@pytest.mark.parametrize("name", sorted(CASES2))
def test_chained_steps_are_the_single_steps(name, precision):
    import torch

    lbm_build.build()
    torch.cuda.set_device(0)
    c = CASES2[name]()
    f = cases.random_populations(c.nx, c.ny, 3)
    got = []
    for chunks in ([64], [1] * 64):
        s = lbm.Solver(c, precision=precision)
        s.set_f(f)
        for n in chunks:
            s.step(n)
            if n == 1:
                torch.cuda.synchronize()
        got.append(s.get_f())
        s.close()
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("name", sorted(CASES3))
def test_chained_steps_are_the_single_steps_3d(name, precision):
    import torch

    lbm_build.build()
    torch.cuda.set_device(0)
    c = CASES3[name]()
    got = []
    for chunks in ([48], [1] * 48):
        s = lbm.Solver3D(c, precision=precision)
        for n in chunks:
            s.step(n)
            if n == 1:
                torch.cuda.synchronize()
        got.append(s.get_f())
        s.close()
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_captured_steps_replay(precision):
    """Two steps captured in a caller's CUDA graph and replayed three times
    are six steps."""
    import torch

    lbm_build.build()
    torch.cuda.set_device(0)
    c = CASES2["cylinders_300x150"]()
    f = cases.random_populations(c.nx, c.ny, 3)
    st = torch.cuda.Stream()
    s = lbm.Solver(c, precision=precision, stream=st.cuda_stream)
    s.set_f(f)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        s.step(2)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    got = s.get_f()
    s.close()
    s = lbm.Solver(c, precision=precision)
    s.set_f(f)
    s.step(6)
    assert np.array_equal(got, s.get_f())
    s.close()
