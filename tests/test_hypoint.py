"""The double-word arithmetic of the hybrid opening pass (csrc/hypoint.cuh), host build: its error is no larger than
with an accurate sum and a normalised product for every term, for each quantity it stores or sums."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2602_17950_gb300", "csrc")
NAMES = ["phi", "hlin", "mass1", "rho", "spin a", "spin z", "H(Phi)", "<H_lin Phi, Phi>", "rho^2", "|F|^2", "mass"]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("hp") / "hypoint_check.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I", CSRC,
                    os.path.join(HERE, "native", "hypoint_check.cpp"), "-o", so], check=True)
    return C.CDLL(so)


# points a thread takes: one (small grids) to many (large batches)
@pytest.mark.parametrize("threads,points", [(60000, 1), (20000, 4), (6000, 16)])
def test_error_no_larger_than_term_by_term(lib, threads, points):
    """The two rms differ by chance by 1/sqrt(2 n) each at most (n errors of about normal size; here n >= 6000, and far
    less as both see the same points): 2% is twice that."""
    rms, most = np.zeros((2, 11)), np.zeros((2, 11))
    assert lib.hp_errors(7, threads, points, rms.ctypes.data_as(C.c_void_p), most.ctypes.data_as(C.c_void_p)) == 11
    for k, name in enumerate(NAMES):
        assert rms[0, k] <= 1.02 * rms[1, k], (name, rms[:, k])
        # products within 7 u^2, a sum's rounding within 3 u^2, five levels of them at most, of values that are themselves
        # products of such (H(Phi), rho^2, |F|^2: three factors)
        assert most[0, k] <= 3 * (7 + 5 * 3), (name, most[:, k])


@pytest.mark.parametrize("n", [1, 3, 24, 96])
def test_radial_part_and_norm_are_fp64_sums(lib, n):
    """FP64 products and sums: of the 2n terms each is rounded, and each sum of at most their moduli, 2^-53 each."""
    rng = np.random.default_rng(n)
    for _ in range(200):
        phi = rng.normal(size=2 * n) * np.exp(-4 * rng.uniform())
        p = (rng.normal(size=2 * n) * np.exp(-8 * rng.uniform())).astype(np.float32)
        got, err, mod = np.zeros(2), np.zeros(2), np.zeros(2)
        lib.hp_radial(n, *(C.c_void_p(a.ctypes.data) for a in (phi, p, got, err, mod)))
        assert np.all(np.abs(err) <= (2 * n + 1) * 2.0 ** -53 * mod)


def test_fp32_values_are_of_the_fp64_state(lib):
    """|r|^2 of the FP64 residual: two roundings of u each, and u times the cross terms (2u of it each) and the low words'
    squares; the density is a double word's high word: half an ulp (u) and what the low word is off by, some u^2."""
    most = np.zeros(2)
    lib.hp_fp32(5, 200000, C.c_void_p(most.ctypes.data))
    u = 2.0 ** -24
    assert most[0] <= 2 + 8 * u and most[1] <= 1 + 64 * u
