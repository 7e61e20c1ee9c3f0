"""Two-step launches at the segment lengths where their index arithmetic has edges: segments of
one plane and of fewer than the unrolled group's four (every entry of the injection tables then
lies in up to nine extended segments), lengths around multiples of four and eight, one segment
for the whole grid, grids whose last float4 of a row is padding or not, receivers on grid points
(one non-zero corner) and between them.  A pair performs the operations of two single steps, so
every output is bitwise that of single-step launches; the environment knobs change launch shapes
only."""
import numpy as np
import pytest

from paper_2201_06914_gb300.inputs import rademacher_shots
from tests.cases import layered_case
from tests.test_gpu_stencil2 import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,off_grid", [(108, 33, False), (237, 40, True), (512, 25, True)])
@pytest.mark.parametrize("tz", [1, 2, 3, 4, 7, 8, 9, 16, 1000])
def test_pairs_match_single_steps(nx, nz, off_grid, tz):
    case = layered_case(ndim=2, nx=nx, nz=nz, nbl=8, nt=37, nshots=2, off_grid=off_grid, zi=0.3, background="const")
    rng = np.random.default_rng(tz)
    case.d_obs = rng.standard_normal((2, case.nt, case.rec.shape[1]))
    Q = rademacher_shots(3, 2, case.nt, 5)
    one = _run(case, Q, {"WP_STENCIL2": "0"}, Tb=16, ncheck=11)
    two = _run(case, Q, {"WP_STENCIL2": "1", "WP_STENCIL2_TZ": str(tz)}, Tb=16, ncheck=11)
    for k in one:
        assert np.isfinite(two[k]).all(), k
        np.testing.assert_array_equal(two[k], one[k], err_msg=k)


@pytest.mark.parametrize("tx", ["128", "256"])
@pytest.mark.parametrize("nx,nz,off_grid", [(104, 31, True), (105, 32, False), (237, 33, True), (17, 3, True)])
def test_side_by_side_planes_match_single_steps(nx, nz, off_grid, tx):
    """Small launches at the library's own choice: 8-plane segments whose planes run side by side,
    grids of a multiple of 8 planes, one less and one more (a last segment of one plane), fewer
    planes than one block holds, rows on and one past a core of 120 columns.  Bitwise as above."""
    case = layered_case(ndim=2, nx=nx, nz=nz, nbl=8, nt=37, nshots=2, off_grid=off_grid, zi=0.3, background="const")
    rng = np.random.default_rng(nx)
    case.d_obs = rng.standard_normal((2, case.nt, case.rec.shape[1]))
    Q = rademacher_shots(3, 2, case.nt, 5)
    one = _run(case, Q, {"WP_STENCIL2": "0", "WP_STENCIL_TX": tx}, Tb=16, ncheck=11)
    two = _run(case, Q, {"WP_STENCIL2": "1", "WP_STENCIL_TX": tx}, Tb=16, ncheck=11)
    for k in one:
        assert np.isfinite(two[k]).all(), k
        np.testing.assert_array_equal(two[k], one[k], err_msg=k)


@pytest.mark.parametrize("nx,ny,nz,tz", [(22, 7, 12, 3), (23, 6, 9, 1), (21, 23, 13, 1000)])
def test_3d_tile_edges(monkeypatch, nx, ny, nz, tz):
    """3-D tiles of 32 x 16 points: rows and y extents on, one below and one past a tile, marches of
    one plane, three planes and the whole depth, against the FP64 oracle (tolerances as in
    test_gpu_parity.py)."""
    from paper_2201_06914_gb300 import wp
    from tests.cases import close
    from tests.test_gpu_parity import GpuRun, _oracle_probed
    monkeypatch.setenv("WP_STENCIL_TZ", str(tz))
    case = layered_case(ndim=3, nx=nx, ny=ny, nz=nz, nbl=5, nt=60, nshots=2, off_grid=True)
    Q = rademacher_shots(6, 2, case.nt, 4)
    ref = _oracle_probed(case, Q, 0.25)
    run = GpuRun(wp, case, case.m0)
    Pu, d = run.forward(Q)
    g, Pv = run.adjoint(ref["res"], Q, ref["Pu"], 0.25)
    for name, a, b, tol in (("d", d, ref["d"], 1e-5), ("Pu", Pu, ref["Pu"], 1e-5), ("Pv", Pv, ref["Pv"], 1e-5),
                            ("g", g, ref["g"].ravel(), 1e-4)):
        ok, err = close(a, b, tol)
        assert ok, (name, err)
