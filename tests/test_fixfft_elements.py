"""Fixed-point transforms as the kernels run them (csrc/fixfft.cuh, host build): element by element, also where the
line's values differ by many powers of two; inverse transforms as forward ones read at index -j; and the
largest lines for 2, 4 and 8 elements per thread, each with its own scaling."""
import numpy as np
import pytest

from tests.test_fixfft import _exact, _inputs, _line, lib  # noqa: F401

SHAPES = [(n, e) for e in (4, 8) for n in (8, 16, 32, 64, 128, 256, 512, 1024)] + [(n, 2) for n in (8, 16, 32, 64)]


def _bound(x, out):
    """Units are at most 2^(m - 59), 2^m <= 2 max (parts of x).  Every pass rounds each value within 3 of its units, which a
    later pass cannot enlarge relative to what it adds up: 3 passes and the inputs' own truncation are n (9 + 1.5)
    2^(m - 59); tabled twiddles are within 2^-58 of theirs, 3 passes: n max 2^-56.  Below n max 2^-54 together; and
    each output is rounded to FP64."""
    largest = max(np.max(np.abs(x.real)), np.max(np.abs(x.imag)))
    return len(x) * largest * 2.0 ** -54 + np.abs(out) * 2.0 ** -53


def _wide(n, seed):
    """Lines whose values span many powers of two: one large among small ones, a decaying tail, one small real part."""
    rng = np.random.default_rng(seed)
    noise = rng.uniform(-1, 1, n) + 1j * rng.uniform(-1, 1, n)
    one = noise * 2.0 ** -20
    one[n // 3] = 1.5
    return {"one large": one, "tail": noise * 2.0 ** -np.linspace(0, 60, n), "small real": noise.imag * 1j + noise.real * 2.0 ** -40}


@pytest.mark.parametrize("n,e", SHAPES)
def test_every_element(lib, n, e):  # noqa: F811
    for name, x in {**_inputs(n, n + e), **_wide(n, n + e)}.items():
        y = _line(lib, x, e)
        back = y[-np.arange(n) % n]                      # the inverse transform, unnormalised
        for got, (re, im) in ((y, _exact(x)), (back, _exact(x, inverse=True))):
            err = np.hypot((got.real - re).astype(float), (got.imag - im).astype(float))
            assert np.all(err <= _bound(x, got)), (name, np.max(err / _bound(x, got)))


@pytest.mark.parametrize("n,e", SHAPES)
def test_largest_lines(lib, n, e):  # noqa: F811
    full = np.full(n, 1.9999999999999998 * (1 + 1j))     # the largest sums a line can have
    for sign, at in ((np.ones(n), 0), (np.where(np.arange(n) % 2, -1, 1), n // 2)):
        y = _line(lib, full * sign, e)
        want = np.zeros(n, dtype=complex)
        want[at] = n * full[0]
        assert np.all(np.abs(y - want) <= _bound(full, want))
    assert np.all(_line(lib, np.zeros(n), e) == 0)
    for bad in (np.nan, np.inf, -np.inf):
        x = full.copy()
        x[n // 3] = bad
        assert np.all(np.isnan(_line(lib, x, e)))
    for scale in (2.0 ** -1070, 2.0 ** 1010):            # subnormal, and near the largest
        y = _line(lib, np.full(n, scale + 0j), e)
        assert y[0] == n * scale and np.all(y[1:] == 0)
