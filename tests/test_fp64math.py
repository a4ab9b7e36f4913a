"""The short FP64 functions (csrc/fp64math.cuh), host build: their errors within the bounds their comments derive, which
are the library's or less (1/sqrt: 1 ulp, sine and cosine: 2 ulp, division: 1/2 ulp and 2^-60 relative)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2602_17950_gb300", "csrc")
SLACK = 2.0 ** -7      # what is left out of a series, 2^-60 relative, in ulp of at least 2^-53


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fm") / "fp64math_check.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I", CSRC,
                    os.path.join(HERE, "native", "fp64math_check.cpp"), "-o", so], check=True)
    lb = C.CDLL(so)
    for name, args in (("fm_rsqrt", [C.c_double, C.c_int]), ("fm_divide", [C.c_double, C.c_double]),
                       ("fm_rsqrt1", [C.c_double]), ("fm_taylor", [C.c_double, C.c_int])):
        getattr(lb, name).argtypes, getattr(lb, name).restype = args, C.c_double
    return lb


def test_rsqrt(lib):
    rng = np.random.default_rng(1)
    xs = list(rng.uniform(1, 4, 4000)) + list(rng.uniform(1, 4, 1500) * 2.0 ** rng.integers(-110, 108, 1500))
    xs += [1.0, np.nextafter(1, 0), np.nextafter(1, 2), 4 - 2.0 ** -50, 2.0 ** -111, np.nextafter(2.0 ** 112, 0)]
    for x in xs:
        for off in (-2, 0, 2):       # the start may be off by 2 FP32 ulp
            e = lib.fm_rsqrt(float(x), off)
            assert 0 <= e <= 1 + SLACK, (x, off)
    for x in (0.0, -1.0, 5e-324, 2.0 ** -112, 2.0 ** 112, np.inf, -np.inf, np.nan):     # left to the library
        assert lib.fm_rsqrt(float(x), 0) == -1


def test_division_by_a_norm(lib):
    rng = np.random.default_rng(2)
    for d in np.concatenate([rng.choice([-1, 1], 3000) * 2.0 ** rng.uniform(-52, -8, 3000),
                             [0.0, 2.0 ** -30, -2.0 ** -30, 2.0 ** -30 * (1 - 2.0 ** -20), 2.0 ** -53]]):
        a = rng.uniform(1, 2) * 2.0 ** rng.integers(-60, 10)
        assert lib.fm_divide(float(a), 1.0 - float(d)) <= 0.5 + SLACK, d


def test_normalisation(lib):
    rng = np.random.default_rng(3)
    for d in np.concatenate([rng.choice([-1, 1], 3000) * 2.0 ** rng.uniform(-60, -20, 3000),
                             [0.0, 2.0 ** -20 * (1 - 2.0 ** -30), -2.0 ** -20 * (1 - 2.0 ** -30)]]):
        # the sum is rounded, and the correction before it, 2^-53 of at most 2^-21
        assert 0 <= lib.fm_rsqrt1(float(d)) <= 0.5 + SLACK, d
    assert lib.fm_rsqrt1(2.0 ** -20) == -1 and lib.fm_rsqrt1(float("nan")) == -1


@pytest.mark.parametrize("odd,bound", [(1, 1.0), (0, 2.0)])
def test_sine_and_cosine(lib, odd, bound):
    rng = np.random.default_rng(4)
    xs = list(rng.uniform(0, 0.7999, 6000)) + list(2.0 ** rng.uniform(-60, -1, 2000))
    xs += [0.5, np.nextafter(0.5, 0), 0.79999, 2.0 ** -27] + ([] if odd else [0.0])
    for x in xs:
        assert 0 <= lib.fm_taylor(float(x), odd) <= bound + SLACK, x
    for x in (-1e-3, 0.8, 1.0, np.inf, np.nan, -0.0):          # left to the library
        assert lib.fm_taylor(float(x), odd) == -1, x
