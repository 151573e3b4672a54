"""Single V-cycles of the correction form against the oracle's FAS cycle, where a lost low part is
seen (whole steps converge whatever a cycle's rounding), and its coarsest solve's fallback.

Tolerance of a cycle: a cell update's corrections are off by a few 2^-44 (the reciprocal's bound)
of its residual's terms, the other operations by 2^-46 of theirs; with a cancellation of up to a
hundred between those terms, 1e-11 (160 x 2^-44) of the change that the cycle makes.  A cycle in
binary32 would be off by at least 2^-24 = 6e-8 of it."""
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


# 64 x 64: launches of their own for the producers' work; 96 x 160: one-launch ways; 512 x 384: levels of
# per-level launches above them
@pytest.mark.parametrize("m,n", [(64, 64), (96, 160), (512, 384)])
@pytest.mark.parametrize("scheme,neumann,pinned", [(1, 0, 0), (2, 0, 0), (1, 1, 0), (2, 1, 1)])
@pytest.mark.parametrize("s", [0.05, 1.0])
def test_one_cycle(mp, oracle_mod, m, n, scheme, neumann, pinned, s):
    phi0 = inputs.noise_field(m, n, 0.07, 0.05, 5)
    o = oracle_mod.Solver(oracle_mod.Params(m=m, n=n, h=0.5, s=s, ny_neumann=neumann))
    g = mp.Solver(mp.default_params(m=m, n=n, h=0.5, dt=s, bc=neumann, pinning=pinned))
    if pinned:
        W = np.zeros((n, m))
        W[:8] = 2.0
        target = inputs.noise_field(m, n, 0.1, 0.05, 4)
        o.set_pinning(W, target)
        g.set_pinning(W, target)
    o.set_state(phi0)
    g.set_state(phi0)
    assert o.step(scheme, fixed_cycles=1, guess=1)["status"] == 0
    assert g.step_cycles(scheme, 1)["status"] == 0
    pg, po = g.get_state()[0], o.get_state()[0]
    change = np.abs(po - phi0).max()
    assert np.abs(pg - po).max() <= 1e-11 * change, (np.abs(pg - po).max() / change)


def small_pivot(oracle_mod, m, n, h, s, phi0):
    """A weight on the cells of one coarsest cell for which the Jacobian's first pivot there is 0.01,
    below the 0.05 that the elimination without pivoting accepts (gam + W + g' < 0: only negative
    weights get there)."""
    p = oracle_mod.Params(m=m, n=n, h=h, s=s)
    f = 2 ** (oracle_mod.num_levels(m, n) - 1)
    c, gam, theta = oracle_mod.scheme_consts(p, 2)
    pc = phi0
    for _ in range(f.bit_length() - 1):
        pc = oracle_mod.restrict(pc)
    mc, nc = m // f, n // f
    unit = np.zeros((nc, mc))
    unit[0, 0] = 1.0
    L3 = unit
    for _ in range(3):
        L3 = oracle_mod.laplacian(L3, h * f)
    diag = oracle_mod.laplacian(unit, h * f)[0, 0]
    W = np.zeros((n, m))
    W[:f, :f] = (0.01 - (1.0 - c * theta * L3[0, 0])) / (-c * diag) - gam - 1.5 * pc[0, 0] ** 2
    return W


@pytest.mark.parametrize("m,n", [(8, 8), (8, 12), (12, 20)])   # coarsest grids of 16, 24 and 60 cells
@pytest.mark.parametrize("tail_cells", [0, 256])               # the coarsest solve alone and in the tail
def test_coarsest_solve_with_a_small_pivot(mp, oracle_mod, m, n, tail_cells):
    """Tolerance: the bar of every whole-step test."""
    h, s = 1.0, 10.0
    phi0 = inputs.noise_field(m, n, 0.07, 0.05, 5)
    W, target = small_pivot(oracle_mod, m, n, h, s, phi0), np.full((n, m), 0.07)
    o = oracle_mod.Solver(oracle_mod.Params(m=m, n=n, h=h, s=s))
    g = mp.Solver(mp.default_params(m=m, n=n, h=h, dt=s, pinning=1))
    g.set_launch_shape(4, 0, 608, tail_cells, 1)
    for x in (o, g):
        x.set_pinning(W, target)
        x.set_state(phi0)
    assert o.step(2, fixed_cycles=6, guess=1)["status"] == 0
    assert g.step_cycles(2, 6)["status"] == 0
    pg, po = g.get_state()[0], o.get_state()[0]
    assert np.abs(pg - po).max() <= 1e-10 * np.abs(po).max()


@pytest.mark.parametrize("m,n", [(8, 8), (8, 12), (12, 20)])
@pytest.mark.parametrize("tail_cells", [0, 256])
def test_fp32_coarsest_solve_with_a_small_pivot(mp, oracle_mod, m, n, tail_cells):
    """A converged step of the mixed form.  Tolerance: both residuals are at most 1e-10; the step's
    Jacobian has no eigenvalue below 0.1 there, and mu and kappa enter phi with c / h^2 < 40:
    1e-7 of a field near 0.1."""
    h, s = 1.0, 10.0
    phi0 = inputs.noise_field(m, n, 0.07, 0.05, 5)
    W, target = small_pivot(oracle_mod, m, n, h, s, phi0), np.full((n, m), 0.07)
    o = oracle_mod.Solver(oracle_mod.Params(m=m, n=n, h=h, s=s))
    g = mp.Solver(mp.default_params(m=m, n=n, h=h, dt=s, pinning=1, precision=mp.MPFC_FP32_INNER, max_cycles=400))
    g.set_launch_shape(4, 0, 608, tail_cells, 1)
    for x in (o, g):
        x.set_pinning(W, target)
        x.set_state(phi0)
    assert o.step(2, tol=1e-10, max_cycles=400, guess=1)["status"] == 0
    assert g.step(2, 1)[0]["status"] == 0
    pg, po = g.get_state()[0], o.get_state()[0]
    assert np.abs(pg - po).max() <= 1e-8
