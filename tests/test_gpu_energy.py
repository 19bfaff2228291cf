"""Conservation of the total energy in FP32 handles: the drift against the FP64 handle
over 200 steps of a periodic noisy box stays unbiased.

Bound per step, relative to the total energy: 2.5e-9, one 24th of half an FP32 ulp.
Independent roundings of about 2e-8 per node and step leave 2e-8 / sqrt(nodes x steps)
= 1e-11 of it; what passes the bound is a bias that every node has in every step."""
import numpy as np
import pytest

import inputs

pytestmark = pytest.mark.gpu

P = pytest.importorskip("paper_2510_14712_gb300")

STEPS, BOUND = 200, 2.5e-9


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_14712_gb300 import build
    build.build()
    P.load()


def vdw(U2, rho, T):
    return dict(eos=dict(a=3.0 / U2, b=1.0 / 3.0, R=8.0 / 3.0, kappa=0.01, eta_over_mu=1.0, rho_ref=rho, T_ref=T), cv=8.0,
                rho=rho, T=T, u=(0.015 if U2 > 10 else 0.05))


# the fluids and states of the scenarios: Taylor-Green, Riemann, shock-liquid column
FLUIDS = {"a3_7": vdw(7.0, 0.6, 0.15), "a3_10": vdw(10.0, 0.65, 0.115), "a3_10_light": vdw(10.0, 0.3, 0.11),
          "a3_35_vapour": vdw(35.0, 0.7385, 0.0326), "a3_35_liquid": vdw(35.0, 1.657, 0.9 / 35.0)}

# Peng-Robinson: h and P handed from the closure to the collision
PR_EOS = dict(kind="pr", a=0.4032248593772784, b=0.2530765865415995, R=3.253076586541602, kappa=0.01, eta_over_mu=0.0,
              rho_ref=0.4, T_ref=0.0875, Tc=1.0 / 12.0, m=0.43163854590719997)
for _r in (0.3, 0.4, 0.45):
    FLUIDS["pr_%g" % _r] = dict(eos=PR_EOS, cv=8.132691466354006, rho=_r, T=0.0875 if _r < 0.45 else 0.09, u=0.05)


def box(fluid, shape):
    f = FLUIDS[fluid]
    c = inputs.Case(name="tgv_d3q27", D=len(shape), shape=shape, eos=dict(f["eos"]), tau=0.1, Pr=0.71, cv=f["cv"])
    arr, n = tuple(reversed(shape)), int(np.prod(shape))
    rel = 0.003 if f["rho"] > 1.5 else 0.01
    c.rho = f["rho"] * (1 + rel * inputs.uniform(1, n).reshape(arr))
    c.T = f["T"] * (1 + 0.3 * rel * inputs.uniform(2, n).reshape(arr))
    c.u = [f["u"] * ((0.4, 0.3, 0.2)[a] + inputs.uniform(3 + a, n).reshape(arr)) for a in range(c.D)]
    return c


def energies(c, precision, step_kernel=0, t_fp64=None):
    s = P.Solver(c, precision=precision, step_kernel=step_kernel, t_fp64=t_fp64)
    try:
        e0 = s.init().fields()["totals"][-1]
        return e0, s.step(STEPS).fields()["totals"][-1]
    finally:
        s.close()


def drift(c, **form):
    r0, r1 = energies(c, "fp64")
    e0, e1 = energies(c, "fp32", **form)
    return (e1 / r1 - e0 / r0) / STEPS


@pytest.mark.parametrize("step_kernel,t_fp64", [(0, None), (1, None), (0, True), (1, True)])
@pytest.mark.parametrize("shape", [(64, 40, 24), (45, 31, 20), (200, 100)], ids=str)
@pytest.mark.parametrize("fluid", sorted(FLUIDS))
def test_total_energy_does_not_drift(fluid, shape, step_kernel, t_fp64):
    d = drift(box(fluid, shape), step_kernel=step_kernel, t_fp64=t_fp64)
    assert abs(d) <= BOUND, "%.2e of the total energy per step" % d
