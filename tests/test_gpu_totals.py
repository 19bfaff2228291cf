"""Totals of FP32 fields: to FP64's rounding for any mixture of magnitudes, and with
infinities and sums beyond FP32's range as sums in FP64 give them."""
import math

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


def _handle(shape):
    c = inputs.tgv(shape=shape) if len(shape) == 3 else inputs.riemann(Nx=shape[0], Ny=shape[1])
    c.x_low = c.x_high = "periodic"
    return c, P.Solver(c, precision="fp32")


@pytest.mark.parametrize("shape", [(4, 1, 1), (3, 1, 1), (4, 1), (2, 1)], ids=str)
def test_mass_of_one_group_to_fp64_rounding(shape):
    """The nodes of one group, densities from 1 to 1e-9 with all their bits: the sum is
    exact but for two FP64 roundings of a number of its size (sums of the errors in FP32
    alone leave up to 2^-48)."""
    c, s = _handle(shape)
    n = int(np.prod(shape))
    try:
        for seed in range(40):
            x = inputs.uniform(100 * seed, 2 * n)
            rho = (1.0 + 0.4 * x[:n]) * 10.0 ** (-9.0 * (0.5 + 0.5 * x[n:]) * (np.arange(n) % 2 == seed % 2))
            arr = tuple(reversed(shape))
            f = s.init(rho=rho.reshape(arr), u=[np.zeros(arr)] * c.D, T=np.full(arr, 0.2)).fields()
            want = math.fsum(f["rho"].ravel())
            assert abs(f["totals"][0] - want) <= 2.0 ** -52 * want, (seed, f["totals"][0] - want)
    finally:
        s.close()


@pytest.mark.parametrize("shape", [(8, 3, 2), (9, 3)], ids=str)
@pytest.mark.parametrize("value,node", [(math.inf, 5), (-math.inf, 0), (math.nan, 7), (3.0e38, None)])
def test_mass_with_infinities_and_beyond_fp32(shape, value, node):
    """The rest population of one node (or of all) set to `value`."""
    c, s = _handle(shape)
    Q, rest = (27, 13) if c.D == 3 else (9, 4)
    try:
        s.init()
        pops = P.lbm_get_populations(s.h).view(np.float32).copy()
        rows = pops.reshape(2 * Q, int(np.prod(shape[1:])), -1)
        if node is None:
            rows[:Q, :, :shape[0]] = 0
            rows[rest, :, :shape[0]] = value
        else:
            rows[rest, node // shape[0], node % shape[0]] = value
        P.lbm_set_populations(s.h, pops.view(np.uint8))
        f = s.fields()
    finally:
        s.close()
    with np.errstate(over="ignore", invalid="ignore"):
        want = f["rho"].sum()
    if math.isnan(value):
        assert math.isnan(f["totals"][0])
    elif node is None:
        assert abs(f["totals"][0] - want) <= 1e-14 * want and want > 3.5e38
    else:
        assert f["totals"][0] == value
