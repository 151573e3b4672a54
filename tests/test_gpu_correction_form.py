"""The V-cycle in correction form (float-float corrections around an FP64 iterate) against
the oracle's FAS cycle where its branches and edges differ: sweep counts with and without the
producers' first half sweep and the last half sweeps' update, each coarsest-solve path, grids
that are all tail, and the routes to the FP64 V-cycle (values, residuals and coefficients
outside the form's range).

Tolerance: the bar of every whole-step test, 1e-10 of the largest value after each step
taken with the oracle's number of V-cycles; a cycle's corrections carry 2^-46 of the change
it makes, so the form itself is far below it."""
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


def lockstep(mp, oracle_mod, m, n, scheme, cycles, steps=2, phi0=None, h=0.5, s=0.05, shape=None, mode=0, neumann=0,
             okw=None, **kw):
    okw = okw or {}
    phi0 = inputs.noise_field(m, n, 0.07, 0.05, 5) if phi0 is None else phi0
    g = mp.Solver(mp.default_params(m=m, n=n, h=h, dt=s, bc=neumann, **kw))
    if shape:
        g.set_launch_shape(*shape)
    g.set_launch_mode(mode)
    g.set_state(phi0)
    o = oracle_mod.Solver(oracle_mod.Params(m=m, n=n, h=h, s=s, ny_neumann=neumann, **okw))
    o.set_state(phi0)
    for k in range(steps):
        ro = o.step(scheme, fixed_cycles=cycles, guess=1)
        rg = g.step_cycles(scheme, cycles)
        assert ro["status"] == 0 and rg["status"] == 0 and rg["cycles"] == cycles
        pg, po = g.get_state()[0], o.get_state()[0]
        assert np.abs(pg - po).max() <= 1e-10 * np.abs(po).max(), (k, np.abs(pg - po).max(), np.abs(po).max())
    return g


@pytest.mark.parametrize("nu1,nu2", [(1, 1), (0, 2), (2, 0), (3, 2)])
@pytest.mark.parametrize("m,n,scheme", [(64, 64, 1), (128, 96, 2)])
def test_sweep_counts(mp, oracle_mod, nu1, nu2, m, n, scheme):
    lockstep(mp, oracle_mod, m, n, scheme, 4, nu1=nu1, nu2=nu2, okw=dict(nu1=nu1, nu2=nu2))


# coarsest grids of 16 (chord), 24 (register columns), 36, 60 and 64 cells (shared memory); widths whose half
# rows are not a multiple of a warp; grids of two levels
@pytest.mark.parametrize("m,n", [(8, 8), (128, 192), (96, 160), (96, 96), (128, 32), (12, 20), (20, 12), (512, 128)])
@pytest.mark.parametrize("neumann", [0, 1])
def test_grids(mp, oracle_mod, m, n, neumann):
    lockstep(mp, oracle_mod, m, n, 2, 4, neumann=neumann)


@pytest.mark.parametrize("m,n", [(64, 64), (128, 96)])
@pytest.mark.parametrize("tail_cells", [0, 1 << 20])
def test_no_tail_and_all_tail_on_the_stream(mp, oracle_mod, m, n, tail_cells):
    """Launched one by one, without a tail and with every level in it."""
    lockstep(mp, oracle_mod, m, n, 1, 3, shape=(4, 0, 608, tail_cells, 1), mode=mp.MPFC_LAUNCH_STREAM)


@pytest.mark.parametrize("mode", [0, 1])
def test_values_outside_the_range_take_the_fp64_cycle(mp, oracle_mod, mode):
    """|phi| of 2^21 (mu near 1e19) and fields of 1e-20: the FP64 loop takes the step over,
    in the graph and on the stream."""
    m, n = 96, 64
    for amp, tol in ((2.0 ** 21, 1e-10), (1e-20, 1e-40)):
        phi0 = amp * (1.0 + 0.01 * inputs.noise_field(m, n, 0.0, 1.0, 6))
        lockstep(mp, oracle_mod, m, n, 1, 3, phi0=phi0, s=1e-5 if amp > 1 else 0.05, tol=tol, mode=mode)


def test_coefficients_outside_the_range_take_the_fp64_cycle(mp, oracle_mod):
    """h = 1e-5: (4/h^2)^2 = 1.6e21; every level keeps its 11 FP64 launches.  After eight
    cycles the oracle itself is within 1.6e-13 of its run in extended precision."""
    g = lockstep(mp, oracle_mod, 128, 64, 1, 8, h=1e-5, s=1e-10)
    assert g.launch_counts(1)[1] == 3 * 11 + 2


def _follow_singles(mp, cfgs, scheme, steps=2, **kw):
    ps = [mp.default_params(h=0.5, m=m, n=n, dt=s, **kw) for m, n, s, _ in cfgs]
    b = mp.BatchSolver(ps)
    singles = []
    for i, (p, (m, n, s, amp)) in enumerate(zip(ps, cfgs)):
        phi0 = inputs.noise_field(m, n, 0.07, 0.05, 30 + i)
        if amp > 1:
            phi0 = amp * (1.0 + 0.01 * inputs.noise_field(m, n, 0.0, 1.0, 30 + i))
        b.set_state(i, phi0)
        g = mp.Solver(p)
        g.set_state(phi0)
        singles.append(g)
    for step in range(steps):
        rc, st = b.step_cycles(scheme, 4)
        assert rc == 0
        for i, g in enumerate(singles):
            g.step_cycles(scheme, 4)
            a, ref = b.get_state(i)[0], g.get_state()[0]
            assert np.abs(a - ref).max() <= 1e-12 * np.abs(ref).max(), (step, i)


# 1e-12: the bar of the batch against single instances (tests/test_gpu_batch.py)
@pytest.mark.parametrize("scheme", [1, 2])
@pytest.mark.parametrize("nu1,nu2", [(2, 2), (0, 2), (2, 0), (1, 3)])
def test_batches_of_uneven_depth(mp, scheme, nu1, nu2):
    """Instances of two levels (all of them in the tail) beside deeper ones, with each coarsest
    grid's size; without the small ones, a tail of four levels; and a single-level instance,
    with which the whole batch keeps the FP64 V-cycle."""
    small = [(8, 8, 0.05, 1.0), (12, 20, 0.05, 1.0)]
    large = [(128, 192, 0.05, 1.0), (96, 160, 0.02, 1.0), (128, 32, 0.05, 1.0)]
    for cfgs in (small + large, large, large[1:] + [(8, 6, 0.05, 1.0)]):
        _follow_singles(mp, cfgs, scheme, nu1=nu1, nu2=nu2)


def test_batch_instance_outside_the_range(mp):
    """One instance of |phi| near 2^21 takes the FP64 loop (the oracle's run of it converges)."""
    _follow_singles(mp, [(64, 64, 0.05, 1.0), (96, 64, 1e-5, 2.0 ** 21), (128, 128, 0.05, 1.0)], 1)


@pytest.mark.parametrize("tx,ty", [(1024, 1), (1, 1024), (64, 16), (32, 2)])
def test_batch_tiles_larger_than_a_block(mp, tx, ty):
    ps = [mp.default_params(h=0.5, m=m, n=n, dt=0.05) for m, n in ((128, 192), (96, 160))]
    out = []
    for tile in (None, (tx, ty)):
        b = mp.BatchSolver(ps)
        for i, p in enumerate(ps):
            b.set_state(i, inputs.noise_field(p.m, p.n, 0.07, 0.05, i))
        if tile:
            for level in range(b.levels - 1):
                b.set_tile(level, *tile)
        assert b.step(2, 2)[0] == 0
        out.append([b.get_state(i)[0] for i in range(2)])
    for x, y in zip(*out):
        assert np.array_equal(x, y)
