"""Batches whose FP64 planes take the split step, as a handle of their size does."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2510_14712_gb300")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_14712_gb300 import build
    build.build()
    P.load()


def test_fp64_planes_that_split_and_planes_that_do_not():
    """A 2-D FP64 batch with planes on either side of 2^20 nodes, shock capturing on two."""
    cases = [inputs.couette(2, (x, y), Ma=0.5, seed=x, rel=1e-2) for x, y in ((1024, 1024), (1023, 1024), (1300, 807))]
    b = P.Batch(cases, precision="fp64")
    try:
        for k in (0, 1):
            b.set_shock_capturing(0.1, 0.05, 0.1, k=k)
        b.init().step(5)
        got = [b.fields(k) for k in range(3)]
    finally:
        b.close()
    for k, c in enumerate(cases):
        s = P.Solver(c, precision="fp64")
        try:
            if k < 2:
                P.lbm_set_shock_capturing(s.h, 0.1, 0.05, 0.1)
            want = s.init().step(5).fields()
        finally:
            s.close()
        for q in ("rho", "u", "T"):
            if k == 1:                               # tiles of another shape than the handle's
                assert np.abs(got[k][q] - want[q]).max() <= 1e-12 * np.abs(want[q]).max(), (k, q)
            else:
                assert np.array_equal(got[k][q], want[q]), (k, q)
