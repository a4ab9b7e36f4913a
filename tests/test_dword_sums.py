"""Running double-word sums (csrc/dword.cuh: dwa_*), the short split and the integer narrowing, on their
host build against exact rational arithmetic."""
import ctypes as C
import os
import subprocess
from fractions import Fraction as F

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2602_17950_gb300", "csrc")
U = F(1, 2 ** 24)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("dwa") / "dwacc_check.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I", CSRC,
                    os.path.join(HERE, "native", "dwacc_check.cpp"), "-o", so], check=True)
    lb = C.CDLL(so)
    lb.dwa_run.argtypes = [C.c_int, C.c_int, C.c_int, C.c_void_p, C.c_void_p, C.c_void_p]
    lb.dwa_narrow.argtypes, lb.dwa_narrow.restype = [C.c_double], C.c_float
    lb.dwa_split.argtypes = [C.c_double, C.c_void_p, C.c_void_p]
    return lb


def _words(rng, n, spread):
    x = rng.uniform(-1, 1, n) * 2.0 ** rng.integers(-spread, spread + 1, n)
    hi = x.astype(np.float32)
    lo = (x - hi.astype(np.float64)).astype(np.float32)
    return np.ascontiguousarray(np.stack([hi, lo], axis=1))


@pytest.mark.parametrize("kind,opens", [(0, 0), (0, 1), (1, 0), (2, 0), (2, 1), (3, 0), (4, 0), (5, 0)])
@pytest.mark.parametrize("n", [1, 2, 5, 12])
def test_sums(lib, kind, opens, n):
    """A term's error: 3 roundings of at most u times its low part (2u of its modulus) and the product of
    the low words, 7 u^2; the low word of the sum, at most (n + 4) u of the moduli, is rounded twice a term;
    and once more, u^2, where the sum is normalised."""
    rng = np.random.default_rng(100 * kind + n)
    for spread in (0, 4, 20):
        for _ in range(40):
            a, b, out = _words(rng, n, spread), _words(rng, n, spread), np.zeros(2, np.float32)
            lib.dwa_run(kind, opens, n, a.ctypes.data, b.ctypes.data, out.ctypes.data)
            x = [F(float(p)) + F(float(q)) for p, q in a]
            y = [F(float(p)) + F(float(q)) for p, q in b]
            terms = {0: [p * q for p, q in zip(x, y)], 1: [-p * q for p, q in zip(x, y)], 2: [p * p for p in x],
                     3: [p * F(float(q[0])) for p, q in zip(x, b)], 4: [F(float(p[0])) ** 2 for p in a], 5: x}[kind]
            got = F(float(out[0])) + F(float(out[1]))
            moduli = sum(abs(t) for t in terms)
            assert abs(got - sum(terms)) <= (8 + 2 * n * (n + 4)) * U * U * moduli
            assert abs(float(out[1])) <= np.spacing(abs(out[0]))      # normalised


def test_short_split_is_the_long_one(lib):
    rng = np.random.default_rng(3)
    f, g = np.zeros(2, np.float32), np.zeros(2, np.float32)
    xs = list(rng.uniform(-2, 2, 2000) * 2.0 ** rng.integers(-200, 200, 2000))
    xs += [0.0, -0.0, 2.0 ** -80, 2.0 ** -81, np.nextafter(2.0 ** 128, 0), 2.0 ** 127, 2.0 ** 128, 1.0, -1.0, 5e-324,
           np.inf, -np.inf, 1 + 2.0 ** -24, 1 + 2.0 ** -24 - 2.0 ** -52, 2 - 2.0 ** -52]
    for x in xs:
        lib.dwa_split(float(x), f.ctypes.data, g.ctypes.data)
        assert f.tobytes() == g.tobytes(), x
    lib.dwa_split(float("nan"), f.ctypes.data, g.ctypes.data)
    assert np.isnan(f[0]) and np.isnan(g[0])


def test_narrowing(lib):
    rng = np.random.default_rng(4)
    for x in rng.uniform(-2, 2, 2000) * 2.0 ** rng.integers(-120, 120, 2000):
        assert abs(F(lib.dwa_narrow(float(x))) - F(float(x))) <= U * abs(F(float(x)))     # half an ulp
    assert lib.dwa_narrow(0.0) == 0.0 and lib.dwa_narrow(1e-60) == 0.0
    assert lib.dwa_narrow(1e60) == np.inf and lib.dwa_narrow(-np.inf) == -np.inf and np.isnan(lib.dwa_narrow(np.nan))
