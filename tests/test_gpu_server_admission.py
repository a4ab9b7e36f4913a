"""A request whose bucket cannot be made ends a server step's admission with its error; the requests admitted
before it run once, and it and those behind it stay queued."""
import pytest

import seeded_inputs as si

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2602_17950_gb300 import GpsocError, Problem, Server  # noqa: E402

TRAP = {"kind": 0, "g": (1.0, 1.1)}
N, L, PAR = (32, 32), (6.0, 6.0), (0.3, 0.5, 60.0, -1.0)
OPTS = dict(tol=1e-12, res_tol=1e-9)


@pytest.mark.parametrize("precision", [0, 2])
def test_requests_admitted_before_an_error_run_once(precision):
    psi = si.gaussian_guess(N, L, 470)
    with Server(hbm_budget_bytes=2e9, slots_per_bucket=4, precision=precision, iters_per_step=8) as sv:
        first = [sv.submit(N, L, PAR, psi, trap=TRAP, **OPTS) for _ in range(2)]
        bad = sv.submit(N, (6.0, -6.0), PAR, psi, trap=TRAP, **OPTS)      # no problem can be made of this box
        behind = sv.submit(N, L, PAR, psi, trap=TRAP, **OPTS)
        for _ in range(2):
            with pytest.raises(GpsocError, match="EINVAL"):
                sv.step()
            assert sv.stats()["queued"] == 2
        sv.cancel(bad)
        assert sv.step() == 3                          # three requests, each in one slot
        got = [sv.poll(t, timeout_ms=-1)[0] for t in first + [behind]]
    with Problem(N, L, [PAR], trap=TRAP) as p:
        p.set_initial(psi[None])
        alone = p.solve(precision=precision, **OPTS)[0]
    for r in got:
        assert r["status"] == "OK" and r["energy"] == pytest.approx(alone["energy"], rel=1e-10)
