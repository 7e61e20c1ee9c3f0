"""Both forms of the two-step launch by name (WP_STENCIL2_SIDE = 1: the planes of 8-plane segments
side by side, 0: marching), whatever form the cost model would take: every output, the imaging
variant's among them, is bitwise that of single steps, on launches of a few blocks and of more
blocks than the device has SMs.  Where the profiler lists the launches, the form asked for must be the
one that ran."""
import numpy as np
import pytest

from paper_2201_06914_gb300.inputs import rademacher_shots
from tests.cases import layered_case
from tests.test_gpu_stencil2 import _run

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("tx", ["128", "256"])
@pytest.mark.parametrize("nx,nz,off_grid", [(17, 3, True), (104, 32, False), (237, 33, True), (512, 201, True)])
def test_both_forms_match_single_steps(monkeypatch, nx, nz, off_grid, tx):
    case = layered_case(ndim=2, nx=nx, nz=nz, nbl=8, nt=37, nshots=2, off_grid=off_grid, zi=0.3, background="const")
    rng = np.random.default_rng(nx)
    case.d_obs = rng.standard_normal((2, case.nt, case.rec.shape[1]))
    Q = rademacher_shots(3, 2, case.nt, 5)
    one = _run(case, Q, {"WP_STENCIL2": "0", "WP_STENCIL_TX": tx}, Tb=16, ncheck=11)
    for side in ("0", "1"):
        monkeypatch.setenv("WP_STENCIL2_SIDE", side)
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CPU,
                                                torch.profiler.ProfilerActivity.CUDA]) as prof:
            two = _run(case, Q, {"WP_STENCIL2": "1", "WP_STENCIL_TX": tx}, Tb=16, ncheck=11)
        ran = {e.key for e in prof.key_averages() if "stencil2" in e.key}
        if ran:
            assert all(("stencil2_tile_kernel" in k) == (side == "1") for k in ran), ran
        for k in one:
            assert np.isfinite(two[k]).all(), k
            np.testing.assert_array_equal(two[k], one[k], err_msg=(side, k))
