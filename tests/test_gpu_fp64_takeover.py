"""Scheme 2 steps whose values or residuals leave the correction form's range: the FP64 V-cycle
takes the step over and restricts phi^k onto the coarse levels again (its planes share memory
with the correction form's).  Tolerance: the bar of every whole-step test, 1e-10 of the largest
value after each step taken with the oracle's number of V-cycles."""
import numpy as np
import pytest

from paper_1208_2643_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("amp,s", [(2.0 ** 21, 1e-5), (1e-20, 0.05)])
def test_scheme2_takeover(oracle_mod, mode, amp, s):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_2643_gb300 import mpfc as mp
    mp.load()
    m, n = 96, 64
    phi0 = amp * (1.0 + 0.01 * inputs.noise_field(m, n, 0.0, 1.0, 6))
    g = mp.Solver(mp.default_params(m=m, n=n, h=0.5, dt=s, tol=1e-10 if amp > 1 else 1e-40))
    g.set_launch_mode(mode)
    g.set_state(phi0)
    o = oracle_mod.Solver(oracle_mod.Params(m=m, n=n, h=0.5, s=s))
    o.set_state(phi0)
    for _ in range(2):
        assert o.step(2, fixed_cycles=3, guess=1)["status"] == 0
        assert g.step_cycles(2, 3)["status"] == 0
        pg, po = g.get_state()[0], o.get_state()[0]
        assert np.abs(pg - po).max() <= 1e-10 * np.abs(po).max()
