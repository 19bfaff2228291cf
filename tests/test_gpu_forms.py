"""GPU parity of the forms that the dispatch of the 3-D collision can reach, at the sizes
where the choice falls (row segments of 128 nodes 9/16, 3/16 or 1/4 full) and in the
combinations of closure, storage and x faces that no other test runs; with the largest
error of a single node bounded, so that one wrong column cannot hide in a norm.

Two steps from a state with 1% noise at every node against the FP64 oracle.  Bounds, per
node in units of the field's rms (u: of the drift): FP64 2e-11 and FP32 5e-4 as
parity_util (20 and 50 times the relative-L2 bounds 1e-12 and 1e-5).  FP16 deviations: the
drift makes deviations of about 0.2 of the populations, each stored to 2^-12 / sqrt(3) of
itself; in quadrature over the weights (0.35 for rho, 0.11 for j_a) one store leaves 1e-5
of rho and 3e-6 in u, three stores 2e-5 and 5e-6 (1e-4 of the drift).  T has about 1.5
times rho's.  Ten times these are allowed: 3e-4 in rho and T, 1.5e-3 in u."""
import numpy as np
import pytest

import inputs
from parity_util import node_err, oracle_run

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2510_14712_gb300")

NODE = {"fp64": (2e-11, 2e-11), "fp32": (5e-4, 5e-4), "fp16dev": (3e-4, 1.5e-3)}       # rho and T, u


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_14712_gb300 import build
    build.build()
    P.load()


def _case(shape, faces, fluid="vdw"):
    sc = inputs.scenario("tgv_d3q27" if fluid == "vdw" else "tgv_pr_d3q27")
    D = len(shape)
    c = inputs.Case(name="tgv_d3q27", D=D, shape=shape, eos=dict(sc["eos"]), tau=0.15, Pr=0.71, cv=sc["cv"])
    arr, n = tuple(reversed(shape)), int(np.prod(shape))
    drift = (0.07, -0.05, 0.04)[:D]
    c.rho = sc["rho0"] * (1 + 0.01 * inputs.uniform(1, n).reshape(arr))
    c.T = sc["T0"] * (1 + 0.01 * inputs.uniform(2, n).reshape(arr))
    c.u = [drift[a] + 0.01 * inputs.uniform(3 + a, n).reshape(arr) for a in range(D)]
    if faces == "tube":
        c.x_low, c.x_high = ("inflow", (1.02 * sc["rho0"], list(drift), sc["T0"])), "outflow"
    elif faces == "walls":
        c.x_low, c.x_high = ("wall", ([0.0, -0.05, 0.04][:D], sc["T0"])), ("wall", ([0.0, -0.03, 0.02][:D], sc["T0"]))
        c.u[0] = 0.01 * inputs.uniform(3, n).reshape(arr)
    return c


def worst(got, want, precision):
    lim, ulim = NODE[precision]
    errs = {"rho": (node_err(got["rho"], want["rho"])[0], lim), "T": (node_err(got["T"], want["T"])[0], lim)}
    for a in range(len(want["u"])):
        errs["u%d" % a] = (node_err(got["u"][a], want["u"][a])[0], ulim)
    return {k: v for k, v in errs.items() if not v[0] <= v[1]}


def run(c, precision, steps=2, step_kernel=0, sc=None):
    s = P.Solver(c, precision=precision, step_kernel=step_kernel)
    try:
        if sc:
            P.lbm_set_shock_capturing(s.h, *sc)
        return s.init().step(steps).fields()
    finally:
        s.close()


CASES = (
    # rows and pairs on either side of the line
    [((x, 3, 2), "periodic", "fp32", "vdw") for x in (4, 8, 68, 72, 76, 140, 144, 148, 276, 284)]
    + [((x, 3, 2), "periodic", "fp16dev", "vdw") for x in (8, 16, 64, 72, 80, 136, 144, 152)]
    + [((x, 3, 2), "tube", "fp32", "vdw") for x in (8, 22, 23, 24, 25, 26, 129, 130)]
    + [((x, 3, 2), "tube", "fp16dev", "vdw") for x in (5, 6, 30, 31, 32, 33, 124, 125)]
    # bounded rows of which there are more than a round of segments: pairs below the line, rows above
    # (no wall channel of 14400 nodes: a wall-normal velocity within FP32 rounding of zero, of
    # which so large a channel has some, flips the side of the upwind difference there)
    + [((x, 30, 20), "tube", "fp32", "vdw") for x in (6, 15, 23, 24)]
    + [((x, 30, 20), "walls", "fp32", "vdw") for x in (6, 15)]
    + [((x, 30, 20), "tube", "fp16dev", "vdw") for x in (6, 15, 31, 32)]
    + [((x, 30, 20), f, "fp32", "pr") for x in (7, 14) for f in ("tube", "walls")]
    # Peng-Robinson: P and c_s^2 handed on, in rows, even and odd pairs, bounded x
    + [((x, 3, 2), "periodic", p, "pr") for x in (5, 6, 35, 38, 72, 132) for p in ("fp32", "fp64")]
    + [((x, 4, 3), f, p, "pr") for x in (21, 26) for f in ("tube", "walls") for p in ("fp32", "fp64")]
)


@pytest.mark.parametrize("shape,faces,precision,fluid", CASES, ids=["x".join(map(str, c[0])) + "-%s-%s-%s" % c[1:] for c in CASES])
def test_collision_forms_match_oracle(shape, faces, precision, fluid):
    c = _case(shape, faces, fluid)
    bad = worst(run(c, precision), oracle_run(c, 2), precision)
    assert not bad, bad


def test_one_population_pulled_from_the_wrong_node_is_seen():
    """The FP16-deviation bound is tight enough: the oracle's result with one face population
    (2/27 of the density) of the first column taken from the node right of it fails."""
    c = _case((136, 3, 2), "periodic")
    want = oracle_run(c, 2)
    got = {k: np.array(want[k]) for k in ("rho", "u", "T")}
    got["rho"][..., 0] += 2.0 / 27.0 * (c.rho[..., 1] - c.rho[..., 0])
    assert not worst(want, want, "fp16dev")
    assert worst(got, want, "fp16dev")


SC_FP16 = [((x, 9, 5), "periodic") for x in (33, 72)] + [((x, 5, 6), "tube") for x in (30, 67)] + [((70, 17), "periodic"), ((61, 9), "tube")]


@pytest.mark.parametrize("shape,faces", SC_FP16, ids=["x".join(map(str, c[0])) + "-" + c[1] for c in SC_FP16])
def test_shock_capturing_with_fp16_deviations(shape, faces):
    """Shock capturing on FP16-deviation handles.  The coefficients multiply differences of
    rounded fields, so the bound is the storage's alone times four."""
    from oracle import lbm as olbm
    c = _case(shape, faces)
    coef = (0.1, 0.05, 0.1)
    m = olbm.Model(c.D, c.shape, c.eos, c.tau, c.Pr, c.cv, c.x_low, c.x_high)
    m.shock_capturing = coef
    want = olbm.Sim(m, c.rho, c.u, c.T).step(3).fields()
    got = run(c, "fp16dev", 3, sc=coef)
    lim, ulim = NODE["fp16dev"]
    assert node_err(got["rho"], want["rho"])[0] <= 4 * lim
    assert node_err(got["T"], want["T"])[0] <= 4 * lim
    for a in range(c.D):
        assert node_err(got["u"][a], want["u"][a])[0] <= 4 * ulim


PLANES = [((x, 1024), f, fl, sc) for x in (1023, 1024) for f in ("periodic", "walls") for fl in ("vdw", "pr") for sc in (None, (0.3, 0.1, 0.2))]


@pytest.mark.parametrize("shape,faces,fluid,coef", PLANES, ids=["%s-%s-%s-%s" % (c[0][0], c[1], c[2], "sc" if c[3] else "") for c in PLANES])
def test_fp64_planes_on_either_side_of_the_split_step(shape, faces, fluid, coef):
    """FP64 planes of 2^20 nodes and more take the three passes: one node column less or more
    against the multi-pass step and, in the default form, every tile shape."""
    c = _case(shape, faces, fluid)
    want = run(c, "fp64", 3, step_kernel=P.LBM_STEP_MULTIPASS, sc=coef)
    s = P.Solver(c, precision="fp64")
    try:
        if coef:
            P.lbm_set_shock_capturing(s.h, *coef)
        for k in range(min(P.lbm_tile_count(s.h), 3)):
            s.init()
            P.lbm_set_tile(s.h, k)
            bad = worst(s.step(3).fields(), want, "fp64")
            assert not bad, (k, bad)
    finally:
        s.close()
