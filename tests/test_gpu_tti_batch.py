"""A TTI shot gives the same bits alone and in a batch, whichever kernels and march lengths the size
of the launch selects: in 2-D one shot of a padded 129 x 31 grid runs the direct second pass and 120
of them the marching one, in 3-D the z segments differ.  Recorded data and projections of the shot;
the probed and the exact gradient of a batch whose other shots have no residual."""
import numpy as np
import pytest

from paper_2201_06914_gb300.inputs import rademacher_shots
from tests.cases import tti_case

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


class Shots:
    def __init__(self, case, th, sel, Q, r, Tb):
        from paper_2201_06914_gb300 import wp
        self.wp, self.case, self.r, self.Tb, self.n = wp, case, r, Tb, len(sel)
        self.M = wp.Model(case.ndim, case.nx, case.ny, case.nz, case.nbl, case.h, case.h, case.h, case.dt, case.nt,
                          _t(case.m0.ravel()), case.damp_v, eps=_t(th.eps.ravel()), delta=_t(th.delta.ravel()),
                          theta=_t(th.theta.ravel()), phi=_t(th.phi.ravel()))
        self.G = wp.Geometry(case.src[sel], case.rec[sel])
        self.Q, self.wav = _t(Q[sel]), _t(case.wavelet)
        self.ws = wp.workspace(wp.wp_workspace_bytes(self.M.handle, self.G.c, r, Tb, wp.WP_MODE_PROBED))

    def new(self, *shape):
        return torch.full(shape, float("nan"), device="cuda")

    def probed(self, res):
        wp, n, N = self.wp, self.n, self.case.N
        Pu, Pv = self.new(n, 2, self.r, N), self.new(n, 2, self.r, N)
        d, g = self.new(n, self.case.nt, self.G.nrec), self.new(N)
        wp.wp_probe_forward(self.M.handle, self.G.c, self.wav, self.Q, self.r, self.Tb, Pu, d, self.ws)
        wp.wp_adjoint_image(self.M.handle, self.G.c, res, self.Q, self.r, self.Tb, 1.0, Pu, g, Pv, self.ws)
        wp.wp_stream_status(self.ws)
        return {"d": d[0], "Pu": Pu[0], "Pv": Pv[0], "g": g}

    def exact(self, d_obs):
        wp = self.wp
        g, d, J = self.new(self.case.N), self.new(self.n, self.case.nt, self.G.nrec), torch.zeros(1, dtype=torch.float64, device="cuda")
        ws = wp.workspace(wp.wp_workspace_bytes(self.M.handle, self.G.c, 0, 1, wp.WP_MODE_EXACT_FULL))
        wp.wp_exact_gradient(self.M.handle, self.G.c, self.wav, d_obs, g, J, d, wp.WP_MODE_EXACT_FULL, 1, ws)
        wp.wp_stream_status(ws)
        return g, d


@pytest.mark.parametrize("ndim,nx,ny,nz,nbl,nt,S", [(2, 117, 1, 19, 6, 60, 120), (2, 112, 1, 22, 6, 45, 120),
                                                   (3, 33, 20, 24, 5, 40, 40)])
def test_one_shot_alone_and_in_a_batch(ndim, nx, ny, nz, nbl, nt, S):
    r, Tb = 2, 32
    case, th = tti_case(ndim=ndim, nx=nx, ny=ny, nz=nz, nbl=nbl, nt=nt, nshots=S)
    Q = rademacher_shots(0, S, nt, r)
    res = np.zeros((S, nt, case.rec.shape[1]))
    res[0] = np.random.default_rng(3).standard_normal(res.shape[1:])
    one, all_ = (Shots(case, th, sel, Q, r, Tb) for sel in ([0], list(range(S))))
    a, b = one.probed(_t(res[:1])), all_.probed(_t(res))
    _, d = all_.exact(_t(res))
    d_obs = d.clone()
    d_obs[0] += _t(res[0])
    a["gx"], b["gx"] = one.exact(d_obs[:1].contiguous())[0], all_.exact(d_obs)[0]
    for k in a:
        assert torch.isfinite(a[k]).all() and a[k].abs().max() > 0, k
        assert torch.equal(a[k], b[k]), k
