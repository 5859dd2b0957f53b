"""Density and velocity as the library forms them (FP32 and 16-bit storage: in
double-FP32) against FP64 sums over the populations it returns.  Every
stored population is an FP32 (or 16-bit) number, so both sides sum the same
values; double-FP32 keeps about 2^-46 of the largest term (here below 1, so
1.5e-14), the populations come back as FP64 numbers near 1 (9 or 19
roundings of 1.1e-16), and u divides by rho near 1: 1e-13 covers both."""
import numpy as np
import pytest

from paper_2012_14707_gb300 import build as lbm_build
from paper_2012_14707_gb300 import cases, lbm

pytestmark = pytest.mark.gpu

C2 = np.array([[0, 0], [1, 0], [0, 1], [-1, 0], [0, -1], [1, 1], [-1, 1], [-1, -1], [1, -1]])


def macro(f, c, a, solid):
    rho = f.sum(0)
    u = [(np.tensordot(c[:, k].astype(float), f, 1) + 0.5 * rho * a[k]) / rho for k in range(len(a))]
    fl = solid == 0
    return [np.where(fl, v, 0.0) for v in [rho, *u]]


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16", "fp16"])
def test_fields_are_the_moments_of_the_populations(precision):
    import torch

    lbm_build.build()
    torch.cuda.set_device(0)
    for c in (cases.cylinder_array(131, 77, 2), cases.periodic_box(33, 1, ax=1e-3, ay=-2e-3)):
        s = lbm.Solver(c, precision=precision)
        s.set_f(cases.random_populations(c.nx, c.ny, 5, amp=3e-2))
        s.step(3)
        want = macro(s.get_f(), C2, (c.ax, c.ay), c.solid)
        for got, w in zip(s.fields(), want):
            assert np.abs(got - w).max() <= 1e-13
        s.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_fields_are_the_moments_of_the_populations_3d(precision):
    import torch

    lbm_build.build()
    torch.cuda.set_device(0)
    for c in (cases.sphere_array3d(20, 4), cases.channel3d(9, 5, 6, 0.35, 0.8, 0.05, u_top=0.02)):
        s = lbm.Solver3D(c, precision=precision)
        s.step(7)
        want = macro(s.get_f(), cases.C3, c.a, c.solid)
        for got, w in zip(s.fields(), want):
            assert np.abs(got - w).max() <= 1e-13
        s.close()
