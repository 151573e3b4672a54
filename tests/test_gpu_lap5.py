"""The integer-pipe five-point sum against exact rational arithmetic: the rounding of the
result (2^-53 of it) plus 5 x 2^-59 of the largest value before it, plus the units that
complemented negative values are off (8 x 2^-59).  Infinities, NaN, overflow and tiny
magnitudes take the FP64 form and equal it."""
import ctypes
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def apply(f):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_2643_gb300 import mpfc
    lib = mpfc.load()
    lib.mpfc_probe_lap5.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    d = torch.from_numpy(np.ascontiguousarray(f)).cuda()
    out = torch.empty(len(f), dtype=torch.float64, device="cuda")
    assert lib.mpfc_probe_lap5(d.data_ptr(), out.data_ptr(), len(f), None) == 0
    torch.cuda.synchronize()
    return out.cpu().numpy()


def groups(kind, rng, n=3000):
    u = rng.uniform(-1, 1, (n, 5))
    if kind == "noise":
        return u
    if kind == "smooth":          # five nearby values: everything cancels
        return 0.3 + 1e-9 * u
    if kind == "spread":          # exponents far apart, sums of one or two of the values
        return u * 2.0 ** rng.integers(-80, 80, (n, 5))
    if kind == "zeros":
        return u * rng.integers(0, 2, (n, 5)) * np.where(rng.random((n, 5)) < 0.5, -1.0, 1.0)
    if kind == "constant":
        return np.repeat(u[:, :1] * 2.0 ** rng.integers(-300, 300, (n, 1)), 5, axis=1)
    return np.where(u < 0, -1, 1) * (2.0 ** rng.integers(-3, 3, (n, 5))) * (1 + rng.integers(-1, 2, (n, 5)) * 2.0 ** -52)


@pytest.mark.parametrize("kind", ["noise", "smooth", "spread", "zeros", "constant", "powers"])
def test_error_bound(kind):
    f = groups(kind, np.random.default_rng(7))
    got = apply(f)
    for row, g in zip(f, got):
        want = sum(Fraction(x) for x in row[:4]) - 4 * Fraction(row[4])
        bound = abs(want) / 2 ** 53 + Fraction(float(np.abs(row).max())) * 13 / 2 ** 59
        assert abs(Fraction(float(g)) - want) <= bound, (row, g, float(want))
    if kind == "constant":
        assert np.all(got == 0.0)


def test_values_outside_the_integer_range_take_the_fp64_form():
    big = 1.7e308
    f = np.array([[np.nan, 1, 1, 1, 1], [np.inf, 1, 1, 1, 1], [1, 1, 1, 1, -np.inf], [np.inf, -np.inf, 0, 0, 0],
                  [big, big, 1, 1, 1], [1, 1, 1, 1, big], [0, 0, 0, 0, 0], [-0.0, 0, 0, 0, 0], [5e-324, 0, 0, 0, 5e-324],
                  [1e-280, -1e-280, 2e-280, 0, 1e-281], [1e307, 1e307, 1e307, 1e307, 1e307]])
    with np.errstate(all="ignore"):
        want = (f[:, 0] + f[:, 1]) + (f[:, 2] + f[:, 3]) - 4.0 * f[:, 4]
    got = apply(f)
    assert np.array_equal(np.isnan(got), np.isnan(want))
    ok = ~np.isnan(want)
    assert np.allclose(got[ok], want[ok], rtol=2e-16, atol=0.0)
