"""3-D batches: every pass of the step is one launch over the blocks of all instances of a
kind.  Instances of every kind (row segments with periodic and bounded x, pairs of even
and odd rows, walls, shock capturing, extents of one node) in one batch step bit for bit
as single handles do, in every storage form."""
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


def _box(shape, faces, seed):
    sc = inputs.scenario("tgv_d3q27")
    c = inputs.Case(name="tgv_d3q27", D=3, shape=shape, eos=dict(sc["eos"]), tau=0.15, Pr=0.71, cv=sc["cv"])
    arr, n = tuple(reversed(shape)), int(np.prod(shape))
    drift = (0.07, -0.05, 0.04)
    c.rho = sc["rho0"] * (1 + 0.01 * inputs.uniform(seed, n).reshape(arr))
    c.T = sc["T0"] * (1 + 0.01 * inputs.uniform(seed + 1, n).reshape(arr))
    c.u = [drift[a] + 0.01 * inputs.uniform(seed + 2 + a, n).reshape(arr) for a in range(3)]
    if faces == "tube":
        c.x_low, c.x_high = ("inflow", (1.02 * sc["rho0"], list(drift), sc["T0"])), "outflow"
    elif faces in ("walls", "mixed"):
        wall = ("wall", ([0.0, -0.05, 0.04], sc["T0"]))
        c.x_low, c.x_high = wall, (wall if faces == "walls" else "outflow")
        c.u[0] = 0.01 * inputs.uniform(seed + 2, n).reshape(arr)
    return c


# shape, faces, shock capturing
MIXED = [((128, 3, 4), "periodic", True), ((72, 9, 5), "periodic", False), ((24, 9, 17), "periodic", True),
         ((13, 5, 4), "periodic", True), ((4, 1, 2), "periodic", False), ((130, 3, 2), "tube", True), ((21, 4, 9), "tube", True),
         ((7, 2, 3), "tube", False), ((40, 3, 6), "walls", True), ((9, 4, 3), "mixed", False), ((1, 1, 1), "periodic", False),
         ((64, 8, 7), "periodic", True)]
SETS = {"mixed": MIXED, "one kind": [((16, 8, 8), "periodic", False)] * 5, "pairs only": [((13, 5, 4), "periodic", True)] * 3,
        "no wall": MIXED[:8], "single": MIXED[5:6],
        "one large": [((64, 60, 54), "tube", True)] + MIXED[2:6]}


@pytest.mark.parametrize("precision", ["fp32", "fp16dev", "fp64"])
@pytest.mark.parametrize("name", sorted(SETS))
def test_batch_of_every_kind_matches_single_handles(name, precision):
    kinds = SETS[name]
    cases = [_box(s, f, 10 * k + 1) for k, (s, f, _) in enumerate(kinds)]
    coef = (0.1, 0.05, 0.1)
    b = P.Batch(cases, precision=precision)
    try:
        for k, (_, _, on) in enumerate(kinds):
            if on:
                b.set_shock_capturing(*coef, k=k)
        b.init().step(4)
        b.autotune(1)                                # leaves the state alone
        b.step(3)
        got = [b.fields(k) for k in range(len(cases))]
        flags = [b.flags(k) for k in range(len(cases))]
    finally:
        b.close()
    for k, c in enumerate(cases):
        s = P.Solver(c, precision=precision)
        try:
            if kinds[k][2]:
                P.lbm_set_shock_capturing(s.h, *coef)
            want = s.init().step(7).fields()
            assert flags[k] == P.lbm_get_flags(s.h)
        finally:
            s.close()
        for q in ("rho", "u", "T"):
            assert np.array_equal(got[k][q], want[q]), (k, kinds[k], q)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_walls_of_a_2d_batch_match_single_handles(precision):
    cases = [inputs.couette(2, (60 + 9 * k, 3 + k), Ma=0.5, seed=k, rel=1e-2) for k in range(3)]
    b = P.Batch(cases, precision=precision)
    try:
        b.init().step(9)
        got = [b.fields(k) for k in range(3)]
    finally:
        b.close()
    for k, c in enumerate(cases):
        s = P.Solver(c, precision=precision)
        try:
            n = P.lbm_tile_count(s.h)
            fits = []
            for t in range(n):                       # the batch's tile shape is one of the handle's
                s.init()
                P.lbm_set_tile(s.h, t)
                want = s.step(9).fields()
                fits.append(all(np.array_equal(got[k][q], want[q]) for q in ("rho", "u", "T")))
        finally:
            s.close()
        assert any(fits), k
