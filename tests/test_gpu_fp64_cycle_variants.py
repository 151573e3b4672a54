"""The FP64 V-cycle's own kernels on handles that keep it (h = 1e-5: coefficients outside the
correction form's range): the coarse tail of one CTA or a cluster, the split grid transfers, block
shapes and the fused residual norm give the bits of the plain per-level cycle, as tuning choices
must.  launch_counts tells that the cycle is the FP64 one (11 launches a level)."""
import numpy as np
import pytest

from paper_1208_2643_gb300 import inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = {"periodic1": (128, 128, 1, 0, 0), "periodic2": (128, 128, 2, 0, 0), "ragged1": (96, 160, 1, 0, 0),
         "ragged2": (96, 160, 2, 0, 0), "neumann2": (128, 128, 2, 1, 0), "pinned2": (128, 128, 2, 0, 1)}


@pytest.fixture(scope="module")
def mp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1208_2643_gb300 import mpfc
    mpfc.load()
    return mpfc


def run(mp, case, shape, split=None, per_level=None):
    m, n, scheme, bc, pinned = CASES[case]
    g = mp.Solver(mp.default_params(m=m, n=n, h=1e-5, dt=1e-10, bc=bc, pinning=pinned))
    if pinned:
        W = np.zeros((n, m))
        W[:10] = 2.0
        W[-10:] = 2.0
        g.set_pinning(W, inputs.noise_field(m, n, 0.1, 0.05, 4))
    if shape is not None:
        g.set_launch_shape(*shape)
    if split is not None:
        g.set_transfer_split(split)
    if per_level is not None:
        assert g.launch_counts(scheme)[1] == 11 * per_level + 2
    g.set_state(inputs.noise_field(m, n, 0.07, 0.05, 3))
    infos = [g.step_cycles(scheme, 3) for _ in range(2)]
    assert all(i["status"] == 0 and i["cycles"] == 3 for i in infos)
    st = g.get_state()
    assert all(np.isfinite(x).all() for x in st)
    return st, [i["res"] for i in infos]


def same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a[0], b[0]))


@pytest.mark.parametrize("ctas", [1, 8, 16])
@pytest.mark.parametrize("case", ["periodic1", "periodic2", "ragged2", "neumann2", "pinned2"])
def test_tail(mp, case, ctas):
    levels = {"ragged2": 5}.get(case, 6)
    ref = run(mp, case, (1, 0, 608, 0, 1), per_level=levels - 1)
    for tail_cells in (16 * 16, 32 * 32, 64 * 64):
        try:
            got = run(mp, case, (1, 0, 608, tail_cells, ctas))
        except mp.MPFCError as e:
            if e.status == mp.MPFC_ERR_INVALID and ctas == 16:
                pytest.skip("this GPU holds no 16-CTA cluster")
            raise
        assert same(got, ref), tail_cells


@pytest.mark.parametrize("case", list(CASES))
def test_transfer_split(mp, case):
    ref = run(mp, case, (1, 0, 16, 0, 1), 0)
    for tail_cells, split in ((0, 1 << 30), (0, 64 * 64), (256, 1 << 30)):
        assert same(run(mp, case, (1, 0, 16, tail_cells, 1), split), ref), (tail_cells, split)


@pytest.mark.parametrize("case", ["ragged1", "ragged2", "pinned2"])
def test_launch_shape(mp, case):
    # the last shape puts every level in the tail: the test is k_resnorm over all cells instead of the
    # last half sweep's residual plus k_resnorm_red, the same norm summed in another order
    ref = run(mp, case, None)
    for shape in ((8, 0, 0, 0, 1), (2, 38912, 0, 1024, 1), (4, 1 << 20, 1 << 20, 256, 8), (1, 0, 608, 64 * 64, 1),
                  (1, 0, 608, 1 << 20, 1)):
        got = run(mp, case, shape)
        assert same(got, ref), shape
        np.testing.assert_allclose(got[1], ref[1], rtol=1e-5)
