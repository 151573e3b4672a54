"""The -1 norm's Poisson solve through mpfc_energy at the edges of its levels and right-hand
sides, against the oracle's energies (FFT, or the cosine basis under the Neumann rule).

Tolerance: the solve stops at a relative residual of 1e-13, which bounds the relative error of
the -1 norm's square by about 2e-13 times the ratio of the largest to the relevant wavelength
squared; 1e-10 as in the existing energy test, 1e-9 on the longest grid (16:1)."""
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


# one level; two; all tail; one level above the tail; ragged halves; 64-cell coarsest grids
@pytest.mark.parametrize("m,n", [(4, 4), (8, 8), (12, 20), (64, 64), (128, 64), (96, 160), (128, 32), (256, 64), (192, 320)])
@pytest.mark.parametrize("scale", [1.0, 1e-25, 1e60])
@pytest.mark.parametrize("precision", [0, 1])
def test_minus_one_norm(mp, m, n, scale, precision):
    from oracle import energy
    h = 0.5
    g = mp.Solver(mp.default_params(m=m, n=n, h=h, dt=0.05, precision=precision))
    phi = inputs.noise_field(m, n, 0.07, 0.05, 1)
    psi = inputs.noise_field(m, n, 0.0, 1.0, 2)
    psi = (psi - psi.mean()) * scale
    g.set_state(phi, phi, psi)
    e = g.energy()
    got = e["pseudoF"] - e["F"]
    want = energy.pseudo_F(phi, psi, h, 0.025, 1.0) - energy.F(phi, h, 0.025)
    if scale < 1:   # far below F's rounding: the sum must be F itself
        assert abs(got) <= 1e-14 * abs(e["F"])
    else:
        slack = 1e-14 * abs(e["F"]) if scale == 1.0 else 0.0
        assert abs(got - want) <= 1e-10 * abs(want) + slack, (got, want)


def test_zero_and_nonfinite_velocity(mp):
    g = mp.Solver(mp.default_params(m=64, n=96))
    phi = inputs.noise_field(64, 96, 0.07, 0.05, 1)
    g.set_state(phi)
    e = g.energy()
    assert e["pseudoF"] == e["F"]
    psi = np.zeros((96, 64))
    psi[3, 4] = np.nan
    g.set_state(phi, phi, psi)
    with pytest.raises(mp.MPFCError):
        g.energy()
    g.set_state(phi, phi, inputs.noise_field(64, 96, 0.0, 0.1, 3))
    assert g.energy()["pseudoF"] > e["F"]
    assert g.step(1, 2)[1]["status"] == 0    # the solve's scratch is rewritten by the next step
