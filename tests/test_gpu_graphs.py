"""Step graphs (lbm_set_graphs) against plain launches, bit for bit: after changes of
the layout, and over the forms of the 3-D and 2-D steps."""
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


def same(a, b):
    for k in ("rho", "u", "T"):
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("shape", [(40, 12, 9), (64, 33)])
def test_graphs_after_the_layout_changed_and_came_back(shape):
    """periodic -> outflow -> periodic gives byte-identical parameters, and the allocator may
    return the old population addresses with the scratch planes elsewhere (another handle
    takes their place here): graphs captured before must not be replayed."""
    c = inputs.add_noise(inputs.tgv(shape=shape) if len(shape) == 3 else inputs.riemann(Nx=shape[0], Ny=shape[1]), 3)
    c.x_low = c.x_high = "periodic"
    plain = P.Solver(c, precision="fp32")
    s = P.Solver(c, precision="fp32")
    others = []
    try:
        want = plain.init().step(6).fields()
        P.lbm_set_graphs(s.h, True)
        same(s.init().step(6).fields(), want)
        for _ in range(3):
            P.lbm_set_boundary(s.h, P.LBM_FACE_XLO, P.LBM_BC_OUTFLOW)
            s.init().step(2)
            others.append(P.Solver(c, precision="fp32"))        # takes freed blocks of the periodic layout
            P.lbm_set_boundary(s.h, P.LBM_FACE_XLO, P.LBM_BC_PERIODIC)
            same(s.init().step(6).fields(), want)
    finally:
        for o in others + [plain, s]:
            o.close()
