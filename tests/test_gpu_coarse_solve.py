"""The coarsest solve of the correction form (an inverse of the Jacobian by the whole CTA,
updates by one warp) at the edges of its range, against the oracle's Newton iteration: 4 cells,
32 (one a lane, all lanes), 36 and 64 (two a lane), both schemes, with the fields of order one where
the Jacobian moves most during the solve, in the coarse tail and launched by itself.

Tolerance: the bar of every whole-step test, 1e-10 of the largest value after each step taken
with the oracle's number of V-cycles."""
import numpy as np
import pytest

from paper_1208_2643_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("m,n,coarsest", [(16, 16, 2), (64, 32, 4), (48, 48, 4), (128, 32, 4)])
@pytest.mark.parametrize("scheme", [1, 2])
@pytest.mark.parametrize("tail_cells", [0, 1024])
def test_coarsest_solve(oracle_mod, m, n, coarsest, scheme, tail_cells):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_2643_gb300 import mpfc as mp
    mp.load()
    phi0 = inputs.noise_field(m, n, 0.2, 1.0, 9)
    g = mp.Solver(mp.default_params(m=m, n=n, h=0.5, dt=0.05, coarsest=coarsest))
    g.set_launch_shape(4, 0, 608, tail_cells, 1)
    g.set_state(phi0)
    o = oracle_mod.Solver(oracle_mod.Params(m=m, n=n, h=0.5, s=0.05, coarse_cells=coarsest))
    o.set_state(phi0)
    for _ in range(2):
        ro = o.step(scheme, fixed_cycles=6, guess=1)
        rg = g.step_cycles(scheme, 6)
        assert ro["status"] == 0 and rg["status"] == 0
        pg, po = g.get_state()[0], o.get_state()[0]
        assert np.abs(pg - po).max() <= 1e-10 * np.abs(po).max()


# the mixed form's bar against the oracle solved to 1e-13 (tests/test_gpu_fp32_inner.py)
BOUND = 1e-8


@pytest.mark.parametrize("m,n,coarsest", [(16, 16, 2), (64, 32, 4), (128, 32, 4)])
@pytest.mark.parametrize("tail_cells", [0, 1024])
def test_fp32_coarsest_solve(oracle_mod, m, n, coarsest, tail_cells):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_2643_gb300 import mpfc as mp
    mp.load()
    phi0 = inputs.noise_field(m, n, 0.07, 0.05, 9)
    g = mp.Solver(mp.default_params(m=m, n=n, h=0.5, dt=0.05, coarsest=coarsest, precision=mp.MPFC_FP32_INNER))
    g.set_launch_shape(4, 0, 608, tail_cells, 1)
    g.set_state(phi0)
    o = oracle_mod.Solver(oracle_mod.Params(m=m, n=n, h=0.5, s=0.05, coarse_cells=coarsest))
    o.set_state(phi0)
    for _ in range(2):
        info = g.step(2, 1)[0]
        assert info["status"] == 0 and info["res"] <= 1e-10
        assert o.step(2, tol=1e-13, guess=1)["status"] == 0
        pg, po = g.get_state()[0], o.get_state()[0]
        assert np.abs(pg - po).max() <= BOUND * np.abs(po).max()
