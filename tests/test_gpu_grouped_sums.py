"""GPU tests of the grid sums of passes with more than 1024 blocks per solve, whose partial sums are added
in groups of 64 blocks first: against the same calls at the rule's tiles (one partial per block)."""
import numpy as np
import pytest

import seeded_inputs as si

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2602_17950_gb300 import Problem  # noqa: E402

N, L = (64, 64, 32), (7.0, 7.0, 6.0)
PARS = [(0.4, 0.7, 60.0, -2.0), (0.2, 0.3, 150.0, 3.0)]
TRAP = {"kind": 1, "g": (1.0, 1.2, 0.8), "quad": 0.1, "quart": 0.02}


def _run(p, psi, prec, one_line):
    for axis in range(3):
        p.tuning_set(axis, 1 if one_line else 0, 4 if one_line else 0, precision=prec)
    assert p.tile_shape(0, precision=prec)[0] == 1 or not one_line     # 2048 row and column blocks per solve
    p.set_initial(psi)
    _, obs = p.apply_h(precision=1 if prec else 0)
    p.set_initial(psi)
    # every pass of an iteration: update (stop1: max |dPhi| too), residual maximum, beta, step sums
    res = p.iterate(3, precision=prec, stop=1)
    return obs, res, p.psi()


# two FP64 orders of the same sums: 1e-13 of the sums, which three iterations carry into the state;
# FP32 passes add FP32 terms in double words in either order, so the totals agree to 2^-40 or so of their
# terms and the states to FP32 rounding of what scales with them
@pytest.mark.parametrize("prec,rel,arr", [(0, 1e-13, 1e-11), (1, 1e-10, 1e-5)])
def test_grouped_sums_equal_ungrouped(prec, rel, arr):
    psi = np.stack([si.smooth_random_state(N, L, 40 + k, width=2.0) for k in range(2)])
    with Problem(N, L, PARS, trap=TRAP) as p:
        try:
            a, ra, pa = _run(p, psi, prec, False)
            b, rb, pb = _run(p, psi, prec, True)
        finally:
            for axis in range(3):
                p.tuning_set(axis, 0, 0, precision=prec)
    np.testing.assert_allclose(b, a, rtol=rel if prec == 0 else 1e-6)
    assert np.max(np.abs(pb - pa)) <= arr * np.max(np.abs(pa))
    for x, y in zip(ra, rb):
        assert y["res_inf"] == pytest.approx(x["res_inf"], rel=1e-9 if prec == 0 else 1e-3)
        assert y["energy"] == pytest.approx(x["energy"], rel=1e-12 if prec == 0 else 1e-6)


def test_grouped_hybrid_opening_pass():
    # 128^3: 2128 blocks of the opening pass (the last group has 16), 4096 row and 2048 column blocks
    n, box = (128, 128, 128), (8.0, 8.0, 8.0)
    psi = si.smooth_random_state(n, box, 5, width=2.0)[None]
    with Problem(n, box, PARS[:1], trap=TRAP) as p:
        p.set_initial(psi)
        h = p.iterate(2, precision=2, stop=1)[0]
        E, mu, m = p.observables()
        p.set_initial(psi)
        d = p.iterate(2, precision=0, stop=1)[0]
        E2, mu2, m2 = p.observables()
    assert E[0] == pytest.approx(E2[0], rel=1e-6) and mu[0] == pytest.approx(mu2[0], rel=1e-6)
    np.testing.assert_allclose(m, m2, rtol=1e-5)
    assert h["energy"] == pytest.approx(d["energy"], rel=1e-6) and h["res_inf"] == pytest.approx(d["res_inf"], rel=1e-4)
