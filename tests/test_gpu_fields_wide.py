"""Density and velocity of FP32 and 16-bit states at FP64 accuracy, and of
states with infinities or near the largest numbers as FP64 sums and quotients
give them.

The populations are set, read back and compared without a step.  A stored
deviation is an FP32 number (or shorter) of magnitude 2^-12 to 2^-5, so its sum
over a node is exact in FP64, and float32(f - w) recovers it from the returned
population f = w + d (rounded by at most 2^-54, below half a unit in d's last
place).  From there each side takes at most four roundings (rho, the force
term, its sum with j, the quotient), each of at most 2^-53 of the term it
rounds: 8 in all, 2^-50 of (|j| + rho |a| / 2) / rho."""
import numpy as np
import pytest

from paper_2012_14707_gb300 import build as lbm_build
from paper_2012_14707_gb300 import cases, lbm

pytestmark = pytest.mark.gpu

C2 = np.array([[0, 0], [1, 0], [0, 1], [-1, 0], [0, -1], [1, 1], [-1, 1], [-1, -1], [1, -1]])
W2 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
W3 = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


def wide(d, c, a):
    """rho, u and the size of u's terms from deviations d, in FP64."""
    with np.errstate(all="ignore"):
        rho = 1.0 + d.sum(0)
        u, size = [], []
        for k in range(len(a)):
            j = sum(c[q, k] * d[q] for q in range(len(c)) if c[q, k])
            force = 0.5 * rho * a[k]
            u.append((j + force) / rho)
            size.append((np.abs(j) + np.abs(force)) / rho)
    return rho, u, size


def stored(s, w):
    """The deviations a solver holds."""
    f = s.get_f()
    return (f - w.reshape(-1, *[1] * (f.ndim - 1))).astype(np.float32).astype(np.float64)


def deviations(shape, seed):
    rng = np.random.default_rng(seed)
    d = np.exp2(rng.uniform(-12, -5, shape)) * rng.choice([-1.0, 1.0], shape)
    return d.astype(np.float32).astype(np.float64)


def check(s, w, c, a, solid):
    rho, u, size = wide(stored(s, w), c, a)
    fl = solid == 0
    got = s.fields()
    assert np.abs(got[0] - rho)[fl].max() <= 2.0 ** -52
    for g, v, z in zip(got[1:], u, size):
        assert (np.abs(g - v) <= 2.0 ** -50 * z)[fl].all()


@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp16"])
def test_fields_at_fp64_accuracy(precision):
    lbm_build.build()
    for c in (cases.cylinder_array(131, 77, 2), cases.periodic_box(33, 1, ax=1e-3, ay=-2e-3)):
        s = lbm.Solver(c, precision=precision)
        s.set_f(W2.reshape(9, 1, 1) + deviations((9, c.ny, c.nx), 3))
        check(s, W2, C2, (c.ax, c.ay), c.solid)
        s.close()


def test_fields_at_fp64_accuracy_3d():
    lbm_build.build()
    for c in (cases.sphere_array3d(20, 4), cases.channel3d(9, 5, 6, 0.35, 0.8, 0.05, u_top=0.02)):
        s = lbm.Solver3D(c, precision="fp32")
        s.set_f(W3.reshape(19, 1, 1, 1) + deviations((19, c.nz, c.ny, c.nx), 4))
        check(s, W3, cases.C3, c.a, c.solid)
        s.close()


def _extremes(q, shape):
    """Deviations with, node by node: one infinity; all of the largest size; two
    opposite infinities; sums beyond FP32 that cancel; the smallest steps of f;
    exponents far apart."""
    big = 3.0e38
    d = np.zeros((q, int(np.prod(shape))))
    kinds = np.arange(d.shape[1]) % 6
    d[1, kinds == 0] = np.inf
    d[:, kinds == 1] = big
    d[1, kinds == 2], d[3, kinds == 2] = np.inf, -np.inf
    d[1:3, kinds == 3], d[5:7, kinds == 3] = big, -big
    d[:, kinds == 4] = 2.0 ** -50
    d[:, kinds == 5] = (10.0 ** -np.arange(q))[:, None]
    return d.reshape(q, *shape)


def _same(got, want):
    """Equal infinities and NaN; else within 2^-48 of the value: no sum here
    cancels but exactly, and the reference rounds at most 19 + 4 times."""
    got, want = got.ravel(), want.ravel()
    fin = np.isfinite(want)
    np.testing.assert_array_equal(got[~fin], want[~fin])
    assert (np.abs(got[fin] - want[fin]) <= 2.0 ** -48 * np.abs(want[fin])).all()


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_fields_of_extreme_states(precision):
    lbm_build.build()
    c = cases.periodic_box(37, 11)
    s = lbm.Solver(c, precision=precision)
    s.set_f(W2.reshape(9, 1, 1) + _extremes(9, (c.ny, c.nx)))
    rho, u, _ = wide(stored(s, W2), C2, (c.ax, c.ay))
    for g, w in zip(s.fields(), [rho, *u]):
        _same(g, w)
    s.close()


def test_fields_of_extreme_states_3d():
    lbm_build.build()
    c = cases.periodic_box3d(7, 6, 5)
    s = lbm.Solver3D(c, precision="fp32")
    s.set_f(W3.reshape(19, 1, 1, 1) + _extremes(19, (c.nz, c.ny, c.nx)))
    rho, u, _ = wide(stored(s, W3), cases.C3, c.a)
    for g, w in zip(s.fields(), [rho, *u]):
        _same(g, w)
    s.close()
