"""Steps that leave the correction form for the FP64 V-cycle: at once (values or residuals outside
its range after the guess) and after cycles of it (residuals falling below 2^-56), under both
boundary rules, with pinning, for both models and schemes, in the graph and on the stream, and
in batches.  The FP64 V-cycle's coarse planes share memory with the correction form's.

Tolerance: the bar of every whole-step test, 1e-10 of the largest value after each step taken
with the oracle's number of V-cycles; 1e-12 for batches against single instances."""
import numpy as np
import pytest

from paper_1208_2643_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

M, N = 96, 64
LEAVES = 2.0 ** -56   # residual norms below this leave the form


@pytest.fixture(scope="module")
def mp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_2643_gb300 import mpfc
    mpfc.load()
    return mpfc


def weight():
    W = np.zeros((N, M))
    W[:8] = 2.0
    W[:, 40] += 1.0
    return W


# fields of 2e-15: two to five cycles in correction form, then FP64; of 1e-20: FP64 from the start
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("amp", [2e-15, 1e-20])
@pytest.mark.parametrize("scheme,neumann,pinned,model", [(1, 0, 0, 0), (2, 0, 0, 0), (1, 1, 0, 0), (2, 1, 0, 0), (2, 0, 1, 0),
                                                         (2, 1, 1, 0), (1, 1, 0, 1), (2, 0, 0, 1)])
def test_small_fields(mp, oracle_mod, scheme, neumann, pinned, model, amp, mode):
    phi0 = amp * inputs.noise_field(M, N, 0.5, 0.4, 6)
    target = amp * inputs.noise_field(M, N, 0.1, 0.05, 4)
    o = oracle_mod.Solver(oracle_mod.Params(m=M, n=N, h=0.5, s=0.05, ny_neumann=neumann, model=model))
    g = mp.Solver(mp.default_params(m=M, n=N, h=0.5, dt=0.05, bc=neumann, model=model, pinning=pinned, tol=1e-40))
    g.set_launch_mode(mode)
    if pinned:
        o.set_pinning(weight(), target)
        g.set_pinning(weight(), target)
    o.set_state(phi0)
    g.set_state(phi0)
    for _ in range(2):
        ro = o.step(scheme, fixed_cycles=7, guess=1)
        rg = g.step_cycles(scheme, 7)
        assert ro["status"] == 0 and rg["status"] == 0 and rg["cycles"] == 7
        if amp > 1e-16:   # cycles of both kinds ran
            assert ro["res0"] > 2 * LEAVES and ro["hist"][0] > 2 * LEAVES and ro["hist"][-2] < 0.5 * LEAVES, ro
        else:
            assert ro["res0"] < 0.5 * LEAVES
        pg, po = g.get_state()[0], o.get_state()[0]
        assert np.abs(pg - po).max() <= 1e-10 * np.abs(po).max()


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("scheme,neumann,pinned", [(1, 1, 0), (2, 1, 0), (2, 0, 1), (2, 1, 1)])
def test_large_fields(mp, oracle_mod, scheme, neumann, pinned, mode):
    amp = 2.0 ** 21
    phi0 = amp * (1.0 + 0.01 * inputs.noise_field(M, N, 0.0, 1.0, 6))
    target = amp * (1.0 + 0.01 * inputs.noise_field(M, N, 0.0, 1.0, 4))
    o = oracle_mod.Solver(oracle_mod.Params(m=M, n=N, h=0.5, s=1e-5, ny_neumann=neumann))
    g = mp.Solver(mp.default_params(m=M, n=N, h=0.5, dt=1e-5, bc=neumann, pinning=pinned))
    g.set_launch_mode(mode)
    if pinned:
        o.set_pinning(weight(), target)
        g.set_pinning(weight(), target)
    o.set_state(phi0)
    g.set_state(phi0)
    for _ in range(2):
        assert o.step(scheme, fixed_cycles=3, guess=1)["status"] == 0
        assert g.step_cycles(scheme, 3)["status"] == 0
        pg, po = g.get_state()[0], o.get_state()[0]
        assert np.abs(pg - po).max() <= 1e-10 * np.abs(po).max()


@pytest.mark.parametrize("scheme", [1, 2])
def test_batch_instances_that_leave_midway(mp, scheme):
    """One instance leaves after some cycles, one at the start, two not at all."""
    cfgs = [(64, 64, 1.0), (96, 64, 2e-15), (128, 192, 1.0), (96, 160, 1e-20)]
    ps = [mp.default_params(m=m, n=n, h=0.5, dt=0.05, tol=1e-40) for m, n, _ in cfgs]
    b, singles = mp.BatchSolver(ps), []
    for i, (p, (m, n, amp)) in enumerate(zip(ps, cfgs)):
        phi0 = amp * inputs.noise_field(m, n, 0.5, 0.4, 30 + i)
        b.set_state(i, phi0)
        singles.append(mp.Solver(p))
        singles[i].set_state(phi0)
    for step in range(2):
        assert b.step_cycles(scheme, 7)[0] == 0
        for i, g in enumerate(singles):
            assert g.step_cycles(scheme, 7)["status"] == 0
            got, want = b.get_state(i)[0], g.get_state()[0]
            assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max(), (step, i)
