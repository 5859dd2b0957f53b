"""Several threads reading and setting the fields of one batch's cases: each
gets its own case's data (the binding drops the interpreter lock during a
call, so the calls overlap)."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

from paper_2012_14707_gb300 import build as lbm_build
from paper_2012_14707_gb300 import cases, lbm

pytestmark = pytest.mark.gpu


def _batch():
    cl = cases.batch_cases(6, seed=9, nx_range=(64, 300), ny_range=(64, 260), kn_range=(0.02, 0.1))
    return cl, lbm.Batch(cl, precision="fp32")


def test_threads_read_their_own_case():
    lbm_build.build()
    cl, b = _batch()
    b.run_to(0.0, 100, check_every=50)
    want = [b.fields(k) for k in range(len(cl))]

    def read(k):
        return all(np.array_equal(a, w)
                   for _ in range(40) for a, w in zip(b.fields(k), want[k]))

    with ThreadPoolExecutor(len(cl)) as pool:
        assert all(pool.map(read, range(len(cl))))
    b.close()


def test_threads_set_their_own_case():
    lbm_build.build()
    cl, b = _batch()
    rng = np.random.default_rng(4)
    start = [[1.0 + 1e-3 * rng.standard_normal((c.ny, c.nx)),
              *(1e-3 * rng.standard_normal((2, c.ny, c.nx)))] for c in cl]
    for k in range(len(cl)):
        b.set_fields(k, *start[k])
    want = [b.fields(k) for k in range(len(cl))]
    b.reset()

    def put(k):
        for _ in range(40):
            b.set_fields(k, *start[k])

    with ThreadPoolExecutor(len(cl)) as pool:
        list(pool.map(put, range(len(cl))))
    for k in range(len(cl)):
        for a, w in zip(b.fields(k), want[k]):
            np.testing.assert_array_equal(a, w)
    b.close()
