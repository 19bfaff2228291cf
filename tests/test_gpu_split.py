"""GPU parity of the 3-D step's passes at the sizes where their tilings can go
wrong: row segments of 128 nodes and their 16-byte side units (multiples of the
unit, one more, one less, narrower than a unit), odd and even pairs, one- and
two-node extents, inflow / outflow and wall ends, in every storage form.

Three steps from a noisy drifting state against the FP64 oracle.  Tolerances:
FP64 1e-12 and FP32 1e-5 (the suite's bounds; three FP32 steps of about 50
roundings of 6e-8 each stay below it), FP16-deviation 1e-3 on rho and T.
"""
import numpy as np
import pytest

import inputs
from parity_util import oracle_run, rel_l2

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2510_14712_gb300")

TOL = {"fp64": 1e-12, "fp32": 1e-5, "fp16dev": 1e-3}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_14712_gb300 import build
    build.build()
    P.load()


def _box(shape, faces):
    sc = inputs.scenario("tgv_d3q27")
    c = inputs.Case(name="tgv_d3q27", D=3, shape=shape, eos=dict(sc["eos"]), tau=0.15, Pr=0.71, cv=sc["cv"])
    arr, n = tuple(reversed(shape)), int(np.prod(shape))
    drift = (0.07, -0.05, 0.04)
    c.rho = sc["rho0"] * (1 + 0.01 * inputs.uniform(1, n).reshape(arr))
    c.T = sc["T0"] * (1 + 0.01 * inputs.uniform(2, n).reshape(arr))
    c.u = [drift[a] + 0.01 * inputs.uniform(3 + a, n).reshape(arr) for a in range(3)]
    if faces == "tube":
        c.x_low, c.x_high = ("inflow", (1.02 * sc["rho0"], list(drift), sc["T0"])), "outflow"
    elif faces == "walls":
        c.x_low, c.x_high = ("wall", ([0.0, -0.05, 0.04], sc["T0"])), ("wall", ([0.0, -0.03, 0.02], sc["T0"]))
        c.u[0] = 0.01 * inputs.uniform(3, n).reshape(arr)
    elif faces == "mixed":
        c.x_low, c.x_high = ("wall", ([0.0, -0.05, 0.04], sc["T0"])), "outflow"
        c.u[0] = 0.01 * inputs.uniform(3, n).reshape(arr)
    return c


CASES = (
    [(s, "periodic", "fp32") for s in ((1, 4, 3), (2, 3, 3), (4, 3, 2), (8, 5, 1), (33, 7, 5), (127, 2, 3), (128, 3, 2),
                                       (132, 2, 3), (260, 1, 2), (64, 19, 6))]
    + [(s, "periodic", "fp16dev") for s in ((4, 3, 2), (7, 3, 2), (8, 4, 3), (20, 5, 3), (136, 3, 2))]
    + [(s, "periodic", "fp64") for s in ((1, 3, 2), (33, 5, 4), (40, 9, 3))]
    + [(s, "tube", "fp32") for s in ((5, 3, 2), (123, 2, 2), (124, 3, 2), (125, 3, 3), (128, 4, 3), (251, 2, 2))]
    + [(s, "tube", "fp16dev") for s in ((6, 3, 2), (124, 2, 2), (129, 3, 2))]
    + [(s, "walls", "fp32") for s in ((4, 3, 2), (124, 3, 2), (129, 2, 3))]
    + [((30, 5, 4), "walls", "fp64"), ((37, 4, 3), "mixed", "fp32"), ((29, 3, 4), "mixed", "fp64")]
)


@pytest.mark.parametrize("shape,faces,precision", CASES, ids=["x".join(map(str, c[0])) + "-%s-%s" % c[1:] for c in CASES])
def test_split_step_matches_oracle(shape, faces, precision):
    c = _box(shape, faces)
    want = oracle_run(c, 3)
    s = P.Solver(c, precision=precision)
    try:
        got = s.init().step(3).fields()
    finally:
        s.close()
    for k in ("rho", "T") + (() if precision == "fp16dev" else ("u",)):
        err = rel_l2(got[k], want[k])
        assert err <= TOL[precision], "%s: relative L2 %.2e" % (k, err)
