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


# lattice, precision, closure of the step -> indices that lbm_set_tile has taken
INDICES = [((40, 6, 5), "fp32", 5), ((40, 6, 5), "fp16dev", 5), ((40, 6, 5), "fp64", 1), ((64, 9), "fp32", 9), ((64, 9), "fp16dev", 9),
           ((64, 9), "fp64", 5)]


@pytest.mark.parametrize("shape,precision,count", INDICES, ids=["%dd-%s" % (len(i[0]), i[1]) for i in INDICES])
def test_form_indices_that_were_valid_stay_valid(shape, precision, count):
    """Every index up to the count of earlier versions is taken and steps alike; autotuning
    reports a time for each and chooses one of them."""
    c = inputs.add_noise(inputs.tgv(shape=shape) if len(shape) == 3 else inputs.riemann(Nx=shape[0], Ny=shape[1]), 3)
    s = P.Solver(c, precision=precision)
    tol = 1e-12 if precision == "fp64" else 1e-5
    try:
        assert P.lbm_tile_count(s.h) >= count
        want = s.init().step(3).fields()
        for k in range(count):
            s.init()
            P.lbm_set_tile(s.h, k)
            got = s.step(3).fields()
            assert np.abs(got["rho"] - want["rho"]).max() <= tol * np.abs(want["rho"]).max()
        chosen, _ = P.lbm_autotune(s.h, 1)
        times = P.lbm_autotune_times(s.h)
        assert len(times) == P.lbm_tile_count(s.h) and min(times) > 0 and times[chosen] == min(times)
    finally:
        s.close()


def _tube(c, D):
    sc = inputs.scenario("tgv_d3q27")
    c.x_low, c.x_high = ("inflow", (1.02 * sc["rho0"], [0.05] * D, sc["T0"])), "outflow"
    c.u = [u + 0.05 for u in c.u]
    return c


def _walls(c, D):
    T0 = inputs.scenario("tgv_d3q27")["T0"]
    c.x_low, c.x_high = ("wall", ([0.0, -0.05, 0.04][:D], T0)), ("wall", ([0.0, -0.03, 0.02][:D], T0))
    c.u = [0.2 * u for u in c.u]
    return c


def _box(shape, faces):
    sc = inputs.scenario("tgv_d3q27")
    D, n = len(shape), int(np.prod(shape))
    c = inputs.Case(name="tgv_d3q27", D=D, shape=shape, eos=dict(sc["eos"]), tau=0.15, Pr=0.71, cv=sc["cv"])
    arr = tuple(reversed(shape))
    c.rho = sc["rho0"] * (1 + 0.01 * inputs.uniform(1, n).reshape(arr))
    c.T = sc["T0"] * (1 + 0.01 * inputs.uniform(2, n).reshape(arr))
    c.u = [0.02 * inputs.uniform(3 + a, n).reshape(arr) for a in range(D)]
    return _tube(c, D) if faces == "tube" else (_walls(c, D) if faces == "walls" else c)


REPLAY = ([((x, 7, 5), f, p) for x in (21, 72) for f in ("periodic", "tube", "walls") for p in ("fp32", "fp16dev", "fp64")]
          + [((61, 9), f, p) for f in ("periodic", "tube", "walls") for p in ("fp32", "fp16dev", "fp64")])


@pytest.mark.parametrize("capture", [False, True], ids=["", "sc"])
@pytest.mark.parametrize("shape,faces,precision", REPLAY, ids=["x".join(map(str, c[0])) + "-%s-%s" % c[1:] for c in REPLAY])
def test_replayed_steps_are_the_plain_steps(shape, faces, precision, capture):
    """Plain launches against graph replay, bit for bit, an odd number of steps, and against
    the FP64 oracle (FP64 1e-12, FP32 5e-5 and FP16 deviations 1e-3 on rho and T, the suite's
    bounds with shock capturing)."""
    from oracle import lbm as olbm
    c = _box(shape, faces)
    coef = (0.1, 0.05, 0.1)
    m = olbm.Model(c.D, c.shape, c.eos, c.tau, c.Pr, c.cv, c.x_low, c.x_high)
    if capture:
        m.shock_capturing = coef
    want = olbm.Sim(m, c.rho, c.u, c.T).step(5).fields()
    tol = {"fp64": 1e-12, "fp32": 5e-5, "fp16dev": 1e-3}[precision]
    out = []
    for graphs in (False, True):
        s = P.Solver(c, precision=precision)
        try:
            if capture:
                P.lbm_set_shock_capturing(s.h, *coef)
            P.lbm_set_graphs(s.h, graphs)
            out.append(s.init().step(5).fields())
        finally:
            s.close()
    same(out[1], out[0])
    for q in ("rho", "T"):
        assert np.linalg.norm(out[0][q] - want[q]) <= tol * np.linalg.norm(want[q]), q
