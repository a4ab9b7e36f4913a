"""gpsoc_apply_h_noalloc refuses what it refuses before it touches the device: no launch is left running by a call that
returns an error (host code only, no GPU needed)."""
import ctypes as C

import pytest


@pytest.fixture(scope="module")
def call():
    from paper_2602_17950_gb300 import build
    from paper_2602_17950_gb300 import gpsoc as g
    build.build()

    def run(n, pars):
        grid = g.Grid(len(n), (C.c_int * 3)(*(list(n) + [1] * (3 - len(n)))), (C.c_double * 3)(5.0, 5.0, 5.0))
        trap = g.Trap(0, (C.c_double * 3)(1, 1, 1), 0.0, 0.0, None)
        arr = (g.Params * len(pars))(*[g.Params(*p) for p in pars])
        # device pointers that are never read: every call here ends in a host check
        return g.library().gpsoc_apply_h_noalloc(C.byref(grid), C.byref(trap), arr, len(pars), C.c_void_p(256),
                                                 C.c_void_p(256), None, None)
    return run


@pytest.mark.parametrize("batch,at", [(1, 0), (64, 63), (65, 64), (200, 130)])
def test_parameters_are_checked_before_the_first_launch(call, batch, at):
    for bad in (float("nan"), float("inf")):
        pars = [(0.1, 0.2, 3.0, 1.0)] * batch
        pars[at] = (0.1, 0.2, bad, 1.0)
        assert call((8, 8), pars) == 1          # EINVAL


def test_budget_comes_first(call):
    assert call((256, 256), [(0.1, 0.2, float("nan"), 1.0)] * 3) == 8      # EBUDGET, as before
