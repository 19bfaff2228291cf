"""Cases of tests/test_gpu_incomplete.py, run on the bounds-check build of the library
(LBM_LIBRARY): its debug entries raise status bits as a kernel would."""
import ctypes
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import inputs  # noqa: E402
import paper_2510_14712_gb300 as P  # noqa: E402


def code(call):
    try:
        call()
    except P.LbmError as e:
        return e.code
    return P.LBM_OK


def single(lib, enqueue):
    c = inputs.tgv(shape=(12, 8, 6))
    s = P.Solver(c, precision="fp32")
    try:
        s.init()
        enqueue(s, 2)
        assert lib.lbm_debug_raise_flags(s.h, ctypes.c_uint(P.LBM_FLAG_INCOMPLETE)) == P.LBM_OK
        if enqueue is sync_step:                              # the flag of the step is read with it
            assert code(lambda: s.step(1)) == P.LBM_ECUDA
        for _ in range(2):                                    # the state stays refused
            assert code(s.fields) == P.LBM_ECUDA
            assert code(lambda: P.lbm_get_populations(s.h)) == P.LBM_ECUDA
            assert code(lambda: s.step(1)) == P.LBM_ESTATE
        assert P.lbm_get_flags(s.h) & P.LBM_FLAG_INCOMPLETE
        s.init().step(2)                                      # until it is given anew
        s.fields()
        state = P.lbm_get_populations(s.h)
        lib.lbm_debug_raise_flags(s.h, ctypes.c_uint(P.LBM_FLAG_INCOMPLETE))
        assert code(lambda: P.lbm_sync(s.h)) == P.LBM_ECUDA
        P.lbm_set_populations(s.h, state)
        assert code(s.fields) == P.LBM_OK and code(lambda: s.step(1)) == P.LBM_OK
        # other flags do not refuse the fields
        lib.lbm_debug_raise_flags(s.h, ctypes.c_uint(P.LBM_FLAG_NONFINITE))
        P._check(P.load().lbm_step_async(s.h, 1))
        assert code(s.fields) == P.LBM_OK and code(lambda: P.lbm_sync(s.h)) == P.LBM_EUNSTABLE
        assert code(s.fields) == P.LBM_OK
    finally:
        s.close()


def sync_step(s, n):
    s.step(n)


def async_step(s, n):
    P._check(P.load().lbm_step_async(s.h, n))


def batch(lib):
    cases = [inputs.add_noise(inputs.tgv(shape=(12, 8, 6)), k) for k in range(3)]
    b = P.Batch(cases, precision="fp32")
    try:
        b.init().step_async(2)
        assert lib.lbm_debug_raise_batch_flags(b.b, 1, ctypes.c_uint(P.LBM_FLAG_INCOMPLETE)) == P.LBM_OK
        assert code(lambda: b.fields(0)) == P.LBM_OK
        assert code(lambda: b.fields(1)) == P.LBM_ECUDA
        assert code(lambda: b.autotune(1)) == P.LBM_ECUDA
        assert code(b.sync) == P.LBM_ECUDA
        assert code(lambda: b.step(1)) == P.LBM_ESTATE
        assert b.flags(1) & P.LBM_FLAG_INCOMPLETE and not b.flags(2) & P.LBM_FLAG_INCOMPLETE
        c = cases[1]
        u = np.stack(c.u)
        P._bcheck(P.load().lbm_batch_init(b.b, 1, P._ptr(np.ascontiguousarray(c.rho)), P._ptr(u), P._ptr(np.ascontiguousarray(c.T))))
        assert code(lambda: b.step(2)) == P.LBM_OK
        for k in range(3):
            assert code(lambda: b.fields(k)) == P.LBM_OK
    finally:
        b.close()


def main():
    lib = P.load()
    lib.lbm_debug_raise_flags.argtypes = [ctypes.c_void_p, ctypes.c_uint]
    lib.lbm_debug_raise_batch_flags.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_uint]
    single(lib, sync_step)
    single(lib, async_step)
    batch(lib)
    print("incomplete ok")


if __name__ == "__main__":
    main()
