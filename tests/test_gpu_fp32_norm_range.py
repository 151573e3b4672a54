"""The mixed form's residual norm on fields whose residual is far outside the binary32 range of
its squares.  Fields of 2^-30 and below are linear to FP64 rounding (phi^2 <= 2^-60 beside gam
near 1), so the step on a field scaled by a power of two is the scaled step, residuals included.

Tolerance: the scaled residuals differ by the cubic term (2^-60 relative, in the solution) and
by binary32 rounding where the scaled inner cycles meet subnormals (2^-149 beside residuals of at
least 2^-120): 1e-3 covers both a thousandfold, and a lost norm is off by all of itself."""
import numpy as np
import pytest

from paper_1208_2643_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_2643_gb300 import mpfc
    mpfc.load()
    return mpfc


def run(mp, scheme, exponent, cycles, mode, tol=0.0, max_cycles=100):
    m, n = 96, 64
    g = mp.Solver(mp.default_params(m=m, n=n, h=0.5, dt=0.05, precision=mp.MPFC_FP32_INNER, tol=tol, max_cycles=max_cycles))
    g.set_launch_mode(mode)
    g.set_state(2.0 ** exponent * inputs.noise_field(m, n, 0.5, 0.4, 6))
    if cycles:
        return g.step_cycles(scheme, cycles)
    rc, infos = g.step(scheme, 1, raise_on_error=False)
    return dict(infos[0], rc=rc)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("scheme", [1, 2])
@pytest.mark.parametrize("exponent", [-66, -99])   # fields near 1e-20 and 1e-30
def test_small_fields(mp, scheme, exponent, mode):
    for cycles in (1, 2):
        ref, got = run(mp, scheme, -30, cycles, mode), run(mp, scheme, exponent, cycles, mode)
        scale = 2.0 ** (exponent + 30)
        assert got["status"] == 0 and got["cycles"] == cycles
        for key in ("res0", "res"):
            assert abs(got[key] - scale * ref[key]) <= 1e-3 * scale * ref[key], (cycles, key, got[key], scale * ref[key])


@pytest.mark.parametrize("exponent", [-30, -99])
def test_a_tolerance_below_the_rounding_floor_is_not_met(mp, exponent):
    got = run(mp, 1, exponent, 0, 0, tol=2.0 ** (exponent - 80), max_cycles=6)
    assert got["rc"] == mp.MPFC_ERR_NOT_CONVERGED and got["cycles"] == 6 and got["res"] > 0.0
