"""A layout change whose allocation fails (injected with lbm_debug_fail_alloc) leaves a
handle without buffers: it refuses to step, and the next lbm_init or
lbm_set_populations allocates again."""
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


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])          # two populations, scratch, staging, shock capturing
@pytest.mark.parametrize("again", ["init", "populations"])
def test_failed_layout_is_refused_then_recovers(k, again):
    c = inputs.add_noise(inputs.tgv(shape=(16, 8, 6)), 1)
    ref, s = P.Solver(c, precision="fp32"), P.Solver(c, precision="fp32")
    try:
        for x in (ref, s):
            P.lbm_set_shock_capturing(x.h, 0.1, 0.0, 0.1)
        P.lbm_set_boundary(ref.h, P.LBM_FACE_XLO, P.LBM_BC_OUTFLOW)
        ref.init()
        state = P.lbm_get_populations(ref.h)
        want = ref.step(3).fields()
        s.init().step(2)
        P.lbm_debug_fail_alloc(k)
        try:
            with pytest.raises(P.LbmError) as ei:
                P.lbm_set_boundary(s.h, P.LBM_FACE_XLO, P.LBM_BC_OUTFLOW)
        finally:
            P.lbm_debug_fail_alloc(0)
        assert ei.value.code == P.LBM_ENOMEM
        for call in (lambda: s.step(1), s.fields, lambda: P.lbm_get_populations(s.h)):
            with pytest.raises(P.LbmError) as ei:
                call()
            assert ei.value.code == P.LBM_ESTATE
        if again == "init":
            s.init()
        else:
            P.lbm_set_populations(s.h, state)
        got = s.step(3).fields()
        for q in ("rho", "u", "T"):
            assert np.array_equal(got[q], want[q]), q
    finally:
        ref.close()
        s.close()
