"""Fixed-point transforms of the FP64 passes (csrc/fixfft.cuh), on their host build: against
transforms in more than 53 bits, their error compared with FP64 butterflies of the same passes."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2602_17950_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fx") / "fixfft_check.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", CSRC,
                    os.path.join(HERE, "native", "fixfft_check.cpp"), "-o", so], check=True)
    lb = C.CDLL(so)
    lb.fx_line.argtypes = [C.c_void_p, C.c_int, C.c_int, C.c_int]
    lb.fx_table.argtypes = [C.c_int, C.c_void_p]
    lb.fx_round_trip.argtypes = [C.c_double, C.c_int, C.c_int]
    lb.fx_round_trip.restype = C.c_double
    lb.fx_widen.argtypes = [C.c_longlong, C.c_int]
    lb.fx_widen.restype = C.c_double
    return lb


def _line(lib, x, e, inverse=False):
    y = np.ascontiguousarray(x, dtype=np.complex128).copy()
    lib.fx_line(y.ctypes.data, len(y), e, int(inverse))
    return y


def _exact(x, inverse=False):
    """The transform with long double arithmetic (at least 64 bits): direct sums."""
    n = len(x)
    k = np.arange(n)
    # the angle 2 pi m / n of m = j k mod n, from the octant's values in long double
    pi = np.longdouble("3.14159265358979323846264338327950288")
    m = k.astype(np.longdouble) * (2 * pi / n)
    re, im = np.cos(m), np.sin(m) * (1 if inverse else -1)
    at = np.outer(k, k) % n
    a, b = x.real.astype(np.longdouble), x.imag.astype(np.longdouble)
    return re[at] @ a - im[at] @ b, re[at] @ b + im[at] @ a


def _fp64(x, e, inverse=False):
    """FP64 Stockham passes in the order of the transforms tested."""
    n, L, le = len(x), int(np.log2(len(x))), {2: 1, 4: 2, 8: 3}[e]
    rem, y, ns = L % le, x.astype(np.complex128), 1
    sgn = 1 if inverse else -1
    radices = ([2 ** rem] if rem else []) + [e] * (L // le)
    for r in radices:
        g = np.arange(n // r)
        k = g % ns
        v = [y[g + q * (n // r)] * np.exp(sgn * 2j * np.pi * q * k / (ns * r)) for q in range(r)]
        out = np.empty_like(y)
        d = _fp64_dft(v, sgn)
        for q in range(r):
            out[(g // ns) * ns * r + k + q * ns] = d[q]
        y, ns = out, ns * r
    return y


def _fp64_dft(v, sgn):
    if len(v) == 1:
        return v
    ev, od = _fp64_dft(v[::2], sgn), _fp64_dft(v[1::2], sgn)
    h = len(v) // 2
    w = [{0: 1, 1: sgn * 1j}.get(4 * q / len(v), np.exp(sgn * 2j * np.pi * q / len(v))) for q in range(h)]
    return [ev[q] + w[q] * od[q] for q in range(h)] + [ev[q] - w[q] * od[q] for q in range(h)]


def _inputs(n, seed):
    """Lines the passes meet: condensates, their spectra, noise; and the peaked ones, where one
    exponent per line is at its worst."""
    rng = np.random.default_rng(seed)
    x = np.linspace(-1, 1, n, endpoint=False)
    noise = rng.uniform(-1, 1, n) + 1j * rng.uniform(-1, 1, n)
    bump = np.exp(-(x - 0.1) ** 2 / 0.02) * np.exp(5j * x)
    return {"gaussian": bump, "vortex": bump * (x + 0.2j), "spectrum": np.fft.fft(bump), "noise": noise,
            "noisy bump": bump * noise, "narrow": np.exp(-(x / (8.0 / n)) ** 2) * noise,
            "tiny": noise * 1e-280, "huge": noise * 1e280}


def _error(y, exact):
    re, im = exact
    d = (y.real - re) ** 2 + (y.imag - im) ** 2
    return float(np.sqrt(np.sum(d) / np.sum(re ** 2 + im ** 2)))


def test_twiddle_table(lib):
    pi = np.longdouble("3.14159265358979323846264338327950288")
    w = (C.c_longlong * 2)()
    for k in range(1024):
        lib.fx_table(k, w)
        a = 2 * pi * np.longdouble(k) / 1024
        for got, want in ((w[0], np.cos(a)), (w[1], -np.sin(a))):
            # 26 rounded terms of half a unit each, and long double's own 2^-63
            assert abs(np.longdouble(got) - want * np.longdouble(2) ** 62) <= 16
    for k, want in ((0, (1, 0)), (256, (0, -1)), (512, (-1, 0)), (768, (0, 1))):
        lib.fx_table(k, w)
        assert (w[0], w[1]) == (want[0] << 62, want[1] << 62)


def test_conversions(lib):
    rng = np.random.default_rng(1)
    d = rng.choice([-1.0, 1.0], 4000) * rng.uniform(1, 2, 4000) * 2.0 ** rng.integers(-8, 1, 4000)
    for f in (59, 60, 61):
        for v in d:     # exponent 0 of 53 bits above 2^(1 - f): nothing is dropped within f - 53 bits
            assert abs(lib.fx_round_trip(v, 1023, f) - v) <= 2.0 ** (1 - f)
    assert lib.fx_round_trip(1.75, 1023, 59) == 1.75 and lib.fx_round_trip(-0.0, 1023, 59) == 0.0
    assert lib.fx_round_trip(1e-300, 1023, 59) == 0.0
    for v, s in ((1, 0), (-1, 0), (3, -2), ((1 << 62) + 1, 0), (-(1 << 62) - 513, 5), ((1 << 54) - 1, -60),
                 ((1 << 53) + 1, 0), (2 ** 63 - 1, 0)):
        assert abs(int(lib.fx_widen(v, 0)) - v) <= abs(v) >> 53
        assert lib.fx_widen(v, s) == np.ldexp(lib.fx_widen(v, 0), s)
    assert lib.fx_widen(1 << 40, 1000) == np.inf and lib.fx_widen(-(1 << 40), -1200) == 0.0


# 2 elements per thread: lines of up to 64 points only
@pytest.mark.parametrize("n,e", [(n, e) for e in (4, 8) for n in (8, 16, 32, 64, 128, 256, 512, 1024)]
                         + [(n, 2) for n in (8, 16, 32, 64)])
def test_lines_no_less_exact_than_fp64(lib, n, e):
    for inverse in (False, True):
        for name, x in _inputs(n, n + e).items():
            ref = _exact(x, inverse)
            fx, fp = _error(_line(lib, x, e, inverse), ref), _error(_fp64(x, e, inverse), ref)
            # outputs are rounded to FP64 in either case: half an ulp each, 2^-53 / sqrt(3) at most
            assert fx <= max(fp, 2.0 ** -53), (name, inverse, fx, fp)


@pytest.mark.parametrize("n", [8, 64, 1024])
def test_extreme_lines(lib, n):
    full = np.full(n, 1.9999999999999998 * (1 + 1j))         # the largest sums a line can have
    for inverse in (False, True):
        y = _line(lib, full, 8, inverse)
        assert abs(y[0] - n * full[0]) <= 1e-15 * abs(n * full[0]) and np.max(np.abs(y[1:])) <= 1e-15 * n
        alt = full * np.where(np.arange(n) % 2, -1, 1)
        y = _line(lib, alt, 8, inverse)
        assert abs(y[n // 2] - n * full[0]) <= 1e-15 * abs(n * full[0])
    assert np.all(_line(lib, np.zeros(n), 8) == 0)
    for bad in (np.nan, np.inf):
        x = full.copy()
        x[n // 3] = bad
        assert np.all(np.isnan(_line(lib, x, 8)))
    one = np.zeros(n, dtype=complex)                          # a single mode comes back exactly
    one[0] = 1.0
    assert np.array_equal(_line(lib, one, 8), np.ones(n))
