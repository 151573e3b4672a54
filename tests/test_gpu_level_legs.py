"""A level's way down or up of the correction-form V-cycle as one launch (tiles of 16 x 16 cells
with a halo in shared memory) against the same cycle with every level in the single-CTA tail,
whose sweeps have no halo: the same cell functions on the same values, so the same bits.
Grids whose tiles are ragged, narrower than a tile, or wrap around; one to three sweeps; Neumann
rows at the first and last tile row; the pinning weight in the halo."""
import numpy as np
import pytest

from paper_1208_2643_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("m,n", [(160, 96), (64, 256), (256, 64), (96, 96), (256, 256)])
@pytest.mark.parametrize("scheme,bc,pinned,nu1,nu2", [(1, 0, 0, 2, 2), (2, 1, 0, 2, 2), (2, 0, 1, 2, 2), (2, 1, 1, 1, 3),
                                                      (1, 1, 0, 3, 1)])
def test_leg_is_bitwise_the_tail(m, n, scheme, bc, pinned, nu1, nu2):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_2643_gb300 import mpfc as mp
    mp.load()
    phi0 = inputs.noise_field(m, n, 0.07, 0.05, 11)
    runs = []
    for tail_cells in (0, 1 << 20):
        g = mp.Solver(mp.default_params(m=m, n=n, h=0.5, dt=0.05, bc=bc, pinning=pinned, nu1=nu1, nu2=nu2))
        if pinned:
            W = np.zeros((n, m))
            W[: max(1, n // 5)] = 2.0
            W[:, m // 2] += 1.0
            g.set_pinning(W, inputs.noise_field(m, n, 0.1, 0.05, 4))
        g.set_launch_shape(4, 0, 608, tail_cells, 1)
        g.set_state(phi0)
        st = g.step_cycles(scheme, 3)
        assert st["status"] == 0
        runs.append(g.get_state())
    for a, b in zip(*runs):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("m,n", [(160, 96), (64, 256), (384, 256), (512, 128)])
@pytest.mark.parametrize("scheme,bc,pinned,nu1,nu2", [(1, 0, 0, 2, 2), (2, 1, 1, 2, 2), (2, 1, 0, 1, 2), (1, 0, 0, 2, 1)])
def test_fp32_leg_is_bitwise_the_one_launch_sweeps(m, n, scheme, bc, pinned, nu1, nu2):
    """The FP32 inner cycles' legs against per-level launches (mpfc_set_fp32_sweep), 16 x 16 tiles
    and 32 x 32, whole steps."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_2643_gb300 import mpfc as mp
    mp.load()
    phi0 = inputs.noise_field(m, n, 0.07, 0.05, 12)
    runs = []
    for tiled in (False, True):
        g = mp.Solver(mp.default_params(m=m, n=n, h=0.5, dt=0.05, bc=bc, pinning=pinned, nu1=nu1, nu2=nu2,
                                        precision=mp.MPFC_FP32_INNER))
        if pinned:
            W = np.zeros((n, m))
            W[: max(1, n // 5)] = 2.0
            g.set_pinning(W, inputs.noise_field(m, n, 0.1, 0.05, 4))
        g.set_launch_shape(4, 0, 608, 0, 1)
        if tiled:
            g.set_fp32_sweep(8, 0)
        g.set_state(phi0)
        infos = g.step(scheme, 2)
        assert all(i["status"] == 0 for i in infos)
        runs.append(([i["cycles"] for i in infos], g.get_state()))
    assert runs[0][0] == runs[1][0]
    for a, b in zip(runs[0][1], runs[1][1]):
        assert np.array_equal(a, b)
