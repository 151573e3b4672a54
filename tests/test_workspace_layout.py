"""Workspace sizes of FP64 handles and batches: the correction form's planes are in the layout only
where that form runs, and never make a workspace exceed the device that an FP64 one fits."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def mp():
    from paper_1208_2643_gb300 import build, mpfc
    build.build()
    return mpfc


def batch_bytes(mp, ps):
    return mp.load().mpfc_batch_workspace_bytes(len(ps), (mp.mpfc_params * len(ps))(*ps))


# planes of 8 bytes a cell: 9 on the finest level and 10 on each coarser one (13 1/3 G), two more for the Poisson
# problem of the energies on each level (16 G in all: 2 2/3 more)
def test_handles_that_keep_the_fp64_cycle_have_no_planes_of_the_correction_form(mp):
    G = 1024 * 1024 * 8
    assert mp.workspace_bytes(mp.default_params(m=1024, n=1024, h=1e-6)) < 16.1 * G
    far = mp.default_params(m=1024, n=1024, h=1e-6)
    assert batch_bytes(mp, [far] * 4) < 4 * 13.4 * G
    # an instance of a single level keeps the FP64 V-cycle for the whole batch
    one = [mp.default_params(m=1024, n=1024), mp.default_params(m=8, n=6)]
    assert batch_bytes(mp, one) < 13.4 * G


@pytest.mark.gpu
def test_what_fits_the_device_with_fp64_cycles_still_does(mp):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    total = torch.cuda.get_device_properties(0).total_memory
    G = 1024 * 1024 * 8
    # a batch that takes 93 % of the device with FP64 V-cycles
    count = int(0.93 * total / (13.4 * G))
    need = batch_bytes(mp, [mp.default_params(m=1024, n=1024)] * count)
    assert 0 < need <= total
    # half of it has room for the correction form's planes
    half = batch_bytes(mp, [mp.default_params(m=1024, n=1024)] * (count // 2))
    assert half > count // 2 * 20 * G
    # the largest grid with the learned guess's activations (128 bytes a cell), 2^30 cells
    assert 0 < mp.workspace_bytes(mp.default_params(m=32768, n=32768, guess=mp.MPFC_GUESS_LEARNED)) <= total


@pytest.mark.gpu
@pytest.mark.parametrize("scheme", [1, 2])
def test_batch_in_the_smaller_layout_follows_single_instances(mp, scheme):
    """Coefficients outside the form's range: FP64 V-cycles in both, 1e-12 as in the other
    comparisons of batches with single instances."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import numpy as np
    from paper_1208_2643_gb300 import inputs
    ps = [mp.default_params(m=m, n=n, h=1e-5, dt=1e-10) for m, n in ((128, 64), (96, 160), (8, 8))]
    b, singles = mp.BatchSolver(ps), []
    for i, p in enumerate(ps):
        phi0 = inputs.noise_field(p.m, p.n, 0.07, 0.05, i)
        b.set_state(i, phi0)
        singles.append(mp.Solver(p))
        singles[i].set_state(phi0)
    for _ in range(2):
        assert b.step_cycles(scheme, 4)[0] == 0
        for i, g in enumerate(singles):
            g.step_cycles(scheme, 4)
            got, want = b.get_state(i)[0], g.get_state()[0]
            assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max(), i
