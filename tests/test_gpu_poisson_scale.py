"""The -1 norm's Poisson solve where h^2 psi is far from 1, on phi = 0, so that F = 0 and pseudoF
is the norm's square itself, against the oracle's (FFT, or the cosine basis under the Neumann
rule).  Tolerance: the solve stops at a relative residual of 1e-13, which bounds the relative
error of the square by about 2e-13 times the ratio of the largest to the relevant wavelength
squared; 1e-10 as in the other energy tests."""
import numpy as np
import pytest

from paper_1208_2643_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("m,n", [(8, 8), (96, 160)])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("h,scale", [(0.5, 1.0), (0.5, 1e-25), (0.5, 1e60), (1e-18, 1.0), (1e-13, 1.0), (1e16, 1.0),
                                     (1e-60, 1e120), (1e-30, 1e40), (1e40, 1e-80)])
def test_minus_one_norm_of_any_scale(m, n, bc, h, scale):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import energy
    from paper_1208_2643_gb300 import mpfc as mp
    mp.load()
    g = mp.Solver(mp.default_params(m=m, n=n, h=h, dt=0.05, bc=bc))
    psi = inputs.noise_field(m, n, 0.0, 1.0, 2)
    psi = psi - psi.mean()
    zero = np.zeros((n, m))
    g.set_state(zero, zero, psi * scale)
    # pseudoF = h^2 sum psi x / (2 M) with -Delta_h x = psi: h^4 scale^2 times its value at h = 1
    want = energy.pseudo_F(zero, psi, 1.0, 0.025, 1.0, ny_neumann=bool(bc))
    got = g.energy()["pseudoF"]
    assert abs(got / (h * h * scale) / (h * h * scale) - want) <= 1e-10 * want, (got, want)
