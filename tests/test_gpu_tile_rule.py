"""FP32 passes at the ends of the documented range, where the tile rule is held to what the kernels run: columns of
1024 points, and many columns of 8.  MIXED and HYBRID iterations against FP64 ones at the bars of the other
trajectory tests (states 1e-4, energies 1e-6: the directions carry FP32 rounding), with the same grid spacing."""
import numpy as np
import pytest

import seeded_inputs as si

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2602_17950_gb300 import Problem  # noqa: E402

PAR = (0.3, 0.4, 40.0, 2.0)


@pytest.mark.parametrize("n,L,batch", [((16, 1024), (4.0, 64.0), 1), ((8, 1024), (3.0, 64.0), 3),
                                       ((1024, 1024), (64.0, 64.0), 1), ((16, 8, 1024), (4.0, 3.0, 64.0), 1),
                                       ((256, 256, 8), (24.0, 24.0, 3.0), 8), ((256, 8, 256), (24.0, 3.0, 24.0), 8)])
def test_fp32_iterations_at_the_ends_of_the_range(n, L, batch):
    trap = {"kind": 0, "g": (1.0, 1.1, 1.2)[:len(n)]}
    one = si.gaussian_guess(n, L, 60)
    psi = np.stack([one * np.exp(0.3j * k) for k in range(batch)])
    with Problem(n, L, [PAR] * batch, trap=trap) as p:
        got = {}
        for prec in (0, 1, 2):
            p.set_initial(psi)
            res = p.iterate(3, precision=prec)
            got[prec] = res, p.psi()
        for axis in range(1, len(n)):
            lines, ept, threads = p.tile_shape(axis, precision=1)
            assert (lines, ept) in p.tile_candidates(axis, precision=1) and threads <= 384
    res64, psi64 = got[0]
    for prec in (1, 2):
        res, out = got[prec]
        assert np.max(np.abs(out - psi64)) < 1e-4 * np.max(np.abs(psi64)), prec
        for a, b in zip(res, res64):
            assert a["iters"] == 3
            assert a["energy"] == pytest.approx(b["energy"], rel=1e-6)
