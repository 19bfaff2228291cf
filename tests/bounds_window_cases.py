"""Cases of the bounds-check test with a window of the population buffers declared
outside (tests/test_gpu_bounds_window.py), run on the bounds-check build of the library.

Every access into the window must be counted and skipped, a load giving 0 and a store
dropped.  So one step with the window hidden is, outside the window, bit for bit the step
from populations that hold zeros there: an access that is not checked, a wider range than
the one checked or a load that gives something else shows as a difference."""
import ctypes
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import inputs  # noqa: E402
import paper_2510_14712_gb300 as P  # noqa: E402

G = 4
DT = {"fp64": np.float64, "fp32": np.float32, "fp16dev": np.float16}


def case(shape, faces, seed=1):
    sc = inputs.scenario("tgv_d3q27")
    D, n = len(shape), int(np.prod(shape))
    c = inputs.Case(name="tgv_d3q27", D=D, shape=shape, eos=dict(sc["eos"]), tau=0.15, Pr=0.71, cv=sc["cv"])
    arr = tuple(reversed(shape))
    c.rho = sc["rho0"] * (1 + 0.01 * inputs.uniform(seed, n).reshape(arr))
    c.T = sc["T0"] * (1 + 0.01 * inputs.uniform(seed + 1, n).reshape(arr))
    c.u = [0.05 + 0.01 * inputs.uniform(seed + 2 + a, n).reshape(arr) for a in range(D)]
    if faces == "tube":
        c.x_low, c.x_high = ("inflow", (1.02 * sc["rho0"], [0.05] * D, sc["T0"])), "outflow"
    elif faces == "walls":
        wall = ("wall", ([0.0, -0.05, 0.04][:D], sc["T0"]))
        c.x_low = c.x_high = wall
    return c


# shape, faces, precision, step kernel, first columns (padded x) of windows of 8 elements
CASES = [
    ((72, 3, 2), "periodic", "fp32", 0, (0, 32, 64)),            # rows: both seam units
    ((264, 2, 2), "periodic", "fp32", 0, (120, 128, 256)),       # rows: side units between segments
    ((144, 3, 2), "periodic", "fp16dev", 0, (0, 120, 128, 136)),
    ((37, 3, 2), "periodic", "fp32", 0, (0, 16, 32)),            # pairs, odd
    ((38, 3, 2), "periodic", "fp16dev", 0, (0, 16, 32)),
    ((60, 3, 2), "tube", "fp32", 0, (16, 64)),                   # bounded rows: interior, ghosts right of the last node
    ((124, 2, 2), "tube", "fp32", 0, (64, 128)),
    ((140, 2, 2), "tube", "fp32", 0, (120, 128)),                # side unit of the second segment
    ((140, 2, 2), "tube", "fp16dev", 0, (120, 128)),
    ((45, 3, 2), "walls", "fp32", 0, (16, 32)),
    ((21, 3, 2), "periodic", "fp64", 0, (0, 8, 16)),
    ((130, 17), "periodic", "fp32", 0, (0, 56, 64, 120, 128)),   # 2-D tiles: halos, wrapped pulls, odd tail of the row
    ((67, 9), "periodic", "fp16dev", 0, (0, 56, 64)),
    ((70, 9), "periodic", "fp64", 0, (0, 24, 32, 64)),
    ((61, 9), "tube", "fp32", 0, (16, 56)),
    ((61, 9), "tube", "fp64", 0, (16, 32)),
    ((62, 9), "walls", "fp32", 0, (16, 40)),
    ((72, 9), "periodic", "fp32", 1, (0, 32, 64)),               # 2-D multi-pass: rows
]


def run_case(lib, shape, faces, precision, kernel, columns):
    c = case(shape, faces)
    Q = 9 if c.D == 2 else 27
    rows = int(np.prod(shape[1:]))
    hidden, zeroed = P.Solver(c, precision=precision, step_kernel=kernel), P.Solver(c, precision=precision, step_kernel=kernel)
    bad = []
    try:
        hidden.init()
        state = P.lbm_get_populations(hidden.h).view(DT[precision]).copy()
        plane = state.size // (2 * Q)
        pitch = plane // rows
        zeroed.init()
        # directions with c_x = -1, 0, +1, f and g, the rest population left alone
        third = Q // 3
        for n, i in enumerate((1, third + 2, 2 * third + 1, Q + 2, Q + third + 2, Q + 2 * third + 2)):
            for col in columns:
                lo = i * plane + ((n + col // 8) % rows) * pitch + col
                if faces != "periodic" and col <= G < col + 8:
                    continue                                     # a face's own node: its ghosts are copies
                z = state.copy()
                z[lo:lo + 8] = 0
                # both handles start from buffers that hold the same everywhere
                for s, v in ((hidden, state), (zeroed, z)):
                    P.lbm_set_populations(s.h, v.view(np.uint8).ravel())
                before = P.lbm_debug_bounds_violations()
                lib.lbm_debug_hide_populations(hidden.h, lo, lo + 8)
                P._check(lib.lbm_step_async(hidden.h, 1))
                lib.lbm_debug_hide_populations(hidden.h, 0, 0)
                counted = P.lbm_debug_bounds_violations() - before
                P._check(lib.lbm_step_async(zeroed.h, 1))
                assert P.lbm_debug_bounds_violations() == before + counted
                a = P.lbm_get_populations(hidden.h).view(DT[precision]).copy()
                b = P.lbm_get_populations(zeroed.h).view(DT[precision]).copy()
                a[lo:lo + 8] = b[lo:lo + 8] = 0                  # stores there were dropped
                # nodes past the row's nodes are never read: what is stored there may differ
                width = shape[0] + (0 if faces == "periodic" else 2 * G)
                diff = (a.view(np.uint8).reshape(-1, pitch, a.itemsize) != b.view(np.uint8).reshape(-1, pitch, b.itemsize))[:, :width].any()
                if diff or counted <= 0:
                    bad.append((i, col, counted, bool(diff)))
    finally:
        hidden.close()
        zeroed.close()
    return bad


def main():
    lib = P.load()
    lib.lbm_debug_hide_populations.argtypes = [ctypes.c_void_p, ctypes.c_longlong, ctypes.c_longlong]
    failed = 0
    for k in CASES:
        bad = run_case(lib, *k)
        if bad:
            failed += 1
            print("FAILED", k, bad)
    print("windows: %d of %d cases failed" % (failed, len(CASES)))


if __name__ == "__main__":
    main()
