"""TTI passes at the edges of their tiles against the FP64 oracle, with the tolerances of
test_gpu_tti.py (relative L2 1e-5 for data and projections, 1e-4 for the probed gradient): rows one
point past a 128- or 32-point tile and exactly on it, an odd row length (row padding), a y extent
one past and exactly on pass 1's 16-row tile (pass 2's tile has 8 rows), few planes."""
import pytest

from tests.cases import close
from tests.test_gpu_tti import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ndim,nx,ny,nz", [(2, 117, 1, 20), (2, 116, 1, 11), (3, 22, 7, 9), (3, 23, 6, 12), (3, 21, 23, 5)])
def test_tti_tile_edges(ndim, nx, ny, nz):
    nbl = 6 if ndim == 2 else 5
    ref, out = _run(ndim, nx, ny, nz, nbl, 60, 4, 32)
    for k, tol in (("d", 1e-5), ("Pu", 1e-5), ("Pv", 1e-5), ("g", 1e-4)):
        ok, err = close(out[k].reshape(ref[k].shape), ref[k], tol)
        assert ok, (k, err)


@pytest.mark.parametrize("nt,keys", [(40, ("d", "Pu", "Pv", "g")), (150, ("d", "Pu", "Pv", "g", "gx"))])
def test_tti_2d_large_launch(nt, keys):
    """120 shots of a padded 129 x 31 grid: more than two waves of the direct second pass, which
    the small launches above run, so the marching one runs; the odd extents end inside its tile and
    its segments.  Same tolerances.  The exact gradient (the imaging condition in the second pass)
    forms its residual d - d_obs itself, so it is compared where the residual has the size of the
    data (0.29 of it at 150 steps; 1e-5 at 40, where rounding of d to 32 bits is 1 % of it)."""
    ref, out = _run(2, 117, 1, 19, 6, nt, 2, 32, nshots=120)
    for k in keys:
        ok, err = close(out[k].reshape(ref[k].shape), ref[k], 1e-4 if k in ("g", "gx") else 1e-5)
        assert ok, (k, err)
    assert (out["gc"] == out["gx"]).all()
