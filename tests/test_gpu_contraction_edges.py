"""Kernels behind the stand-alone calls at the sizes where their index arithmetic has edges, against
FP64 (numpy or torch).  Tolerances: the contraction's bf16 hi/lo split leaves 2^-17 = 7.6e-6 per
product (1e-5 relative L2, as in the parity tests); the residual squares in FP32 and sums in FP64
(5e-7); Q is FP32 (1e-5 on Q^T Q), its sketch reproduced to 1e-4 as in test_gpu_range_finder.py."""
import numpy as np
import pytest

from paper_2201_06914_gb300.inputs import rademacher_shots

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("npoints,cnt,r,t0", [(1, 1, 1, 0), (127, 63, 15, 8), (129, 64, 16, 0), (255, 65, 17, 16),
                                              (1001, 130, 64, 8), (385, 128, 256, 0), (130, 200, 300, 8), (640, 70, 33, 0),
                                              # rows of whole tiles: the pipelined kernel with 4, 3, 2 and 1 stages
                                              (128, 1, 1, 0), (384, 200, 64, 8), (20480, 330, 128, 0), (256, 130, 300, 8)])
@pytest.mark.parametrize("exact_bf16", [True, False])   # without and with the probes' lo part
def test_accumulate_any_row_length(npoints, cnt, r, t0, exact_bf16):
    from paper_2201_06914_gb300 import wp
    rng = np.random.default_rng(npoints + r)
    S, nt = 2, t0 + cnt + 5
    A = rng.standard_normal((S, cnt, npoints)).astype(np.float32)
    Q = rademacher_shots(1, S, nt, r) if exact_bf16 else rng.standard_normal((S, nt, r)).astype(np.float32)
    P0 = rng.standard_normal((S, r, npoints)).astype(np.float32)
    ref = P0 + 0.5 * np.einsum("sti,stx->six", Q[:, t0:t0 + cnt].astype(np.float64), A.astype(np.float64))
    P = _t(P0)
    ws = wp.workspace(wp.wp_probe_accumulate_workspace_bytes(S, nt, r))
    wp.wp_probe_accumulate(_t(A), cnt, npoints, S, _t(Q), nt, t0, r, 0.5, P, ws)
    wp.wp_stream_status(ws)
    assert _rel(P.cpu().numpy(), ref) <= 1e-5
    if r <= 256:
        P = _t(P0)
        wp.wp_probe_accumulate_static(_t(A), cnt, npoints, S, _t(Q), nt, t0, r, 0.5, P)
        wp.wp_static_status()
        assert _rel(P.cpu().numpy(), ref) <= 1e-5


# rows of one CTA: a single one, fewer than 32, more than 512; the rows in shared memory or not (r = 256
# of 1000); more shots than clusters that fit at once
@pytest.mark.parametrize("nt,ncols,r,S", [(9, 12, 9, 2), (70, 64, 33, 3), (1000, 600, 256, 1), (700, 300, 40, 40), (4200, 80, 4, 1)])
def test_range_finder_row_splits(nt, ncols, r, S):
    from paper_2201_06914_gb300 import wp
    rng = np.random.default_rng(nt)
    D = rng.standard_normal((S, nt, ncols)).astype(np.float32)
    Z = rademacher_shots(4, S, nt, r)
    ws = wp.workspace(wp.wp_range_finder_workspace_bytes(nt, ncols, S, False, r))
    Q = torch.full((S, nt, r), float("nan"), device="cuda")
    wp.wp_range_finder(_t(D), nt, ncols, S, False, 1, _t(Z), r, Q, ws)
    wp.wp_stream_status(ws)
    Q = Q.cpu().numpy().astype(np.float64)
    for s in range(S):
        assert np.abs(Q[s].T @ Q[s] - np.eye(r)).max() <= 1e-5
        Y = D[s].astype(np.float64) @ (D[s].astype(np.float64).T @ Z[s])
        R = np.linalg.qr(Y, mode="r")
        R *= np.where(np.diag(R) < 0, -1.0, 1.0)[:, None]
        assert _rel(Q[s] @ R, Y) <= 1e-4


@pytest.mark.parametrize("n", [1, 3, 4, 255, 1023, 262147])
@pytest.mark.parametrize("shift", [0, 1])   # 16-byte aligned records or not
def test_residual_and_misfit(n, shift):
    from paper_2201_06914_gb300 import wp
    g = torch.Generator(device="cuda").manual_seed(n)
    a, b = (torch.randn(n + shift, generator=g, device="cuda")[shift:] for _ in range(2))
    res, J = torch.empty(n, device="cuda"), torch.empty(1, dtype=torch.float64, device="cuda")
    wp.wp_residual(a, b, res, n, J, wp.workspace(wp.wp_residual_workspace_bytes(n)))
    assert torch.equal(res, a - b)
    ref = 0.5 * float((res.double() ** 2).sum())
    assert abs(float(J) - ref) <= 5e-7 * ref


@pytest.mark.parametrize("ndim,nx,ny,nz,tti", [(2, 104, 1, 37, False), (2, 48, 1, 21, True), (3, 28, 19, 17, False)])
def test_dense_rows_written_directly(ndim, nx, ny, nz, tti):
    """Row lengths that are a multiple of 4 (but grids that are no multiple of 128 points): the
    dense projections are the row-aligned ones bit for bit, and so is the image from either."""
    from paper_2201_06914_gb300 import wp
    from tests.cases import layered_case, tti_case
    nbl, nt, r, Tb = 6, 40, 5, 16
    th = None
    if tti:
        case, th = tti_case(ndim=ndim, nx=nx, ny=ny, nz=nz, nbl=nbl, nt=nt, nshots=2)
    else:
        case = layered_case(ndim=ndim, nx=nx, ny=ny, nz=nz, nbl=nbl, nt=nt, nshots=2)
    kw = {k: _t(getattr(th, k).ravel()) for k in ("eps", "delta", "theta", "phi")} if tti else {}
    NZ, NY, NX = (nz + 2 * nbl, ny + 2 * nbl if ndim == 3 else 1, nx + 2 * nbl)
    assert NX % 4 == 0 and (NX * NY * NZ) % 128
    SV = 2 * (2 if tti else 1)
    Q, wav = _t(rademacher_shots(3, 2, nt, r)), _t(case.wavelet)
    res = _t(np.random.default_rng(0).standard_normal((2, nt, case.rec.shape[1])))
    out = {}
    for layout in ("dense", "aligned"):
        M = wp.Model(ndim, nx, ny, nz, nbl, case.h, case.h, case.h, case.dt, nt, _t(case.m0.ravel()), case.damp_v, **kw)
        G = wp.Geometry(case.src, case.rec)
        row = M.use_aligned_probes() if layout == "aligned" else M.N
        ws = wp.workspace(wp.wp_workspace_bytes(M.handle, G.c, r, Tb, wp.WP_MODE_PROBED))
        Pu, Pv = (torch.full((SV, r, row), float("nan"), device="cuda") for _ in range(2))
        g = torch.empty(M.N, device="cuda")
        wp.wp_probe_forward(M.handle, G.c, wav, Q, r, Tb, Pu, None, ws)
        wp.wp_adjoint_image(M.handle, G.c, res, Q, r, Tb, 1.0 / r, Pu, g, Pv, ws)
        g2 = torch.empty(M.N, device="cuda")
        wp.wp_adjoint_image(M.handle, G.c, res, Q, r, Tb, 1.0 / r, Pu, g2, None, ws)   # P_v kept in the workspace
        wp.wp_stream_status(ws)
        assert torch.equal(g, g2)
        out[layout] = [x.cpu() for x in (Pu[..., :M.N], Pv[..., :M.N], g)]
        M.close()
    for a, b in zip(out["dense"], out["aligned"]):
        assert torch.isfinite(a).all() and torch.equal(a, b)
