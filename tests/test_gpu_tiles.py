"""GPU parity of the 2-D tile step at the sizes where a tile can go wrong: planes
narrower than a tile's halo, one node more or less than a tile, odd widths (a
pair of nodes across the edge), one- and two-row planes, inflow / outflow and
wall ends, in every storage form and with every tile shape; and 3-D batches
(one graph branch per group of instances) against single handles.

Three steps from a noisy drifting state against the FP64 oracle, with the
suite's tolerances: FP64 1e-12, FP32 1e-5, FP16-deviation 1e-3 on rho and T.
"""
import math

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


def _plane(shape, faces, seed=1):
    sc = inputs.scenario("tgv_d3q27")
    D = len(shape)
    c = inputs.Case(name="tgv_d3q27", D=D, shape=shape, eos=dict(sc["eos"]), tau=0.15, Pr=0.71, cv=sc["cv"])
    arr, n = tuple(reversed(shape)), int(np.prod(shape))
    drift = (0.07, -0.05, 0.04)[:D]
    c.rho = sc["rho0"] * (1 + 0.01 * inputs.uniform(seed, n).reshape(arr))
    c.T = sc["T0"] * (1 + 0.01 * inputs.uniform(seed + 1, n).reshape(arr))
    c.u = [drift[a] + 0.01 * inputs.uniform(seed + 2 + a, n).reshape(arr) for a in range(D)]
    wall = ("wall", (([0.0, -0.05, 0.04])[:D], sc["T0"]))
    if faces == "tube":
        c.x_low, c.x_high = ("inflow", (1.02 * sc["rho0"], list(drift), sc["T0"])), "outflow"
    elif faces in ("walls", "mixed"):
        c.x_low, c.x_high = wall, (wall if faces == "walls" else "outflow")
        c.u[0] = 0.01 * inputs.uniform(seed + 2, n).reshape(arr)
    return c


CASES = (
    [(s, "periodic", "fp32") for s in ((1, 1), (2, 3), (3, 2), (6, 4), (15, 9), (16, 8), (33, 7), (63, 17), (64, 8), (65, 16),
                                       (130, 5))]
    + [(s, "periodic", "fp16dev") for s in ((5, 3), (32, 9), (67, 8))]
    + [(s, "periodic", "fp64") for s in ((1, 2), (9, 5), (33, 9))]
    + [(s, "tube", "fp32") for s in ((5, 1), (60, 4), (63, 9), (64, 8), (65, 3), (128, 17))]
    + [(s, "tube", p) for s in ((31, 5), (66, 8)) for p in ("fp16dev", "fp64")]
    + [(s, "walls", p) for s in ((4, 1), (61, 3), (64, 9), (66, 2)) for p in ("fp32", "fp64")]
    + [((63, 5), "mixed", "fp32"), ((40, 9), "mixed", "fp64")]
)


@pytest.mark.parametrize("shape,faces,precision", CASES, ids=["x".join(map(str, c[0])) + "-%s-%s" % c[1:] for c in CASES])
def test_tile_step_matches_oracle(shape, faces, precision):
    c = _plane(shape, faces)
    want = oracle_run(c, 3)
    s = P.Solver(c, precision=precision)
    try:
        for k in range(P.lbm_tile_count(s.h)):
            s.init()
            P.lbm_set_tile(s.h, k)
            got = s.step(3).fields()
            for q in ("rho", "T") + (() if precision == "fp16dev" else ("u",)):
                err = rel_l2(got[q], want[q])
                assert err <= TOL[precision], "tile %d %s: relative L2 %.2e" % (k, q, err)
    finally:
        s.close()


def test_batch_3d_matches_single_handles():
    """A 3-D batch (periodic and tube instances, shock capturing on one) steps each
    instance as a single handle does."""
    cases = [_plane((24, 9, 5), "periodic", 11), _plane((40, 6, 7), "tube", 21), _plane((13, 5, 4), "periodic", 31),
             _plane((130, 3, 2), "tube", 41), _plane((16, 8, 8), "periodic", 51)]
    b = P.Batch(cases, precision="fp32")
    try:
        b.set_shock_capturing(0.1, 0.0, 0.1, k=1)
        b.init().step(7)
        got = [b.fields(k) for k in range(len(cases))]
    finally:
        b.close()
    for k, c in enumerate(cases):
        s = P.Solver(c, precision="fp32")
        try:
            if k == 1:
                P.lbm_set_shock_capturing(s.h, 0.1, 0.0, 0.1)
            want = s.init().step(7).fields()
        finally:
            s.close()
        for q in ("rho", "u", "T"):
            assert np.array_equal(got[k][q], want[q]), (k, q)


SC_TOL = {"fp64": 1e-12, "fp32": 5e-5}            # the suite's bounds with shock capturing
SC_CASES = ([(s, "periodic") for s in ((1, 1), (3, 2), (7, 5), (63, 17), (64, 16), (65, 33), (130, 3))]
            + [(s, "tube") for s in ((4, 1), (61, 15), (64, 17), (66, 4), (129, 18))] + [((62, 5), "walls")])


@pytest.mark.parametrize("step_kernel", [0, 1])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("shape,faces", SC_CASES, ids=["x".join(map(str, c[0])) + "-" + c[1] for c in SC_CASES])
def test_shock_capturing_tiles_match_oracle(shape, faces, precision, step_kernel):
    """The coefficient tiles (64 x 16 nodes, four-node halo, wrapped or clamped) at their
    edges, after the tile step and after the multi-pass step."""
    from oracle import lbm as olbm
    c = _plane(shape, faces)
    coef = (0.5, 0.2, 0.4)
    m = olbm.Model(c.D, c.shape, c.eos, c.tau, c.Pr, c.cv, c.x_low, c.x_high)
    m.shock_capturing = coef
    want = olbm.Sim(m, c.rho, c.u, c.T).step(4).fields()
    s = P.Solver(c, precision=precision, step_kernel=step_kernel)
    try:
        P.lbm_set_shock_capturing(s.h, *coef)
        got = s.init().step(4).fields()
    finally:
        s.close()
    for q, w in (("rho", want["rho"]), ("u", np.stack(want["u"])), ("T", want["T"])):
        err = rel_l2(got[q], w)
        assert err <= SC_TOL[precision], "%s: relative L2 %.2e" % (q, err)


SC3_CASES = ([(s, "periodic") for s in ((1, 1, 1), (3, 2, 5), (7, 9, 3), (33, 8, 6), (64, 5, 9), (66, 17, 4), (9, 8, 37))]
             + [(s, "tube") for s in ((4, 1, 2), (61, 9, 5), (64, 8, 7), (67, 3, 11))] + [((34, 6, 5), "walls")])


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("shape,faces", SC3_CASES, ids=["x".join(map(str, c[0])) + "-" + c[1] for c in SC3_CASES])
def test_shock_capturing_columns_match_oracle(shape, faces, precision):
    """The 3-D coefficient columns (64 or 32 x 8 nodes marching z, four-node halo, wrapped
    or clamped) at the edges of the columns and of their z-segments."""
    from oracle import lbm as olbm
    c = _plane(shape, faces)
    coef = (0.5, 0.2, 0.4)
    m = olbm.Model(c.D, c.shape, c.eos, c.tau, c.Pr, c.cv, c.x_low, c.x_high)
    m.shock_capturing = coef
    want = olbm.Sim(m, c.rho, c.u, c.T).step(4).fields()
    s = P.Solver(c, precision=precision)
    try:
        P.lbm_set_shock_capturing(s.h, *coef)
        got = s.init().step(4).fields()
    finally:
        s.close()
    for q, w in (("rho", want["rho"]), ("u", np.stack(want["u"])), ("T", want["T"])):
        err = rel_l2(got[q], w)
        assert err <= SC_TOL[precision], "%s: relative L2 %.2e" % (q, err)


@pytest.mark.parametrize("shape,faces", [((70, 9), "periodic"), ((61, 5), "tube"), ((33, 7, 5), "periodic"), ((40, 3, 6), "tube"),
                                         ((1, 1), "periodic")])
def test_initial_populations_round_the_fp64_equilibria(shape, faces):
    """FP32 handles evaluate the initial equilibria in double-float arithmetic (2^-45 relative): every
    stored value is the FP64 handle's rounded to FP32, at most one ulp off where it lies that close to
    the middle of two FP32 numbers (2^-20 of all values; 1e-4 allowed)."""
    c = _plane(shape, faces)
    c.rho = c.rho * (1 + 0.3 * np.sin(np.arange(c.rho.size)).reshape(c.rho.shape))
    pops = {}
    for prec, dt in (("fp64", np.float64), ("fp32", np.float32)):
        s = P.Solver(c, precision=prec)
        try:
            s.init()
            pops[prec] = P.lbm_get_populations(s.h).view(dt).copy()
        finally:
            s.close()
    want = pops["fp64"].astype(np.float32)
    off = pops["fp32"] != want
    assert off.mean() <= 1e-4
    assert np.all(np.abs(pops["fp32"] - want) <= np.spacing(np.abs(want)))


@pytest.mark.parametrize("precision", ["fp32", "fp16dev", "fp64"])
@pytest.mark.parametrize("shape,faces", [((1, 1), "periodic"), ((70, 9), "periodic"), ((61, 5), "tube"), ((33, 7, 5), "periodic"),
                                         ((40, 3, 6), "tube"), ((515, 300), "periodic")])
def test_totals_are_the_sums_of_the_fields(shape, faces, precision):
    """lbm_totals by groups of four nodes (rows of any length, ghost columns left out): the
    mass is the sum of the reported rho up to FP64's rounding; momentum and energy are the
    sums of rho u and rho (c_v T - a rho + u^2 / 2) up to the fields' FP32 rounding (6e-8
    each, a few of them per term)."""
    c = _plane(shape, faces)
    s = P.Solver(c, precision=precision)
    try:
        f = s.init().step(2).fields()
    finally:
        s.close()
    rho, u, T, tot = f["rho"], f["u"], f["T"], f["totals"]
    assert abs(tot[0] - math.fsum(rho.ravel())) <= 1e-14 * np.abs(rho).sum()
    tol = 1e-12 if precision == "fp64" else 2e-6
    for a in range(c.D):
        assert abs(tot[1 + a] - (rho * u[a]).sum()) <= tol * np.abs(rho * u[a]).sum() + 1e-300
    e = [rho * c.cv * T, -c.eos["a"] * rho * rho, 0.5 * rho * (u * u).sum(0)]
    assert abs(tot[1 + c.D] - sum(x.sum() for x in e)) <= tol * sum(np.abs(x).sum() for x in e)
