"""The calls that users of this library make, at the sizes they make them, for timing.

A case is one call (or one loss and its backward) through the public entry points: the C ABI's
Python binding (paper_2201_06914_gb300.wp) and the autograd Function (.autograd).  Kinds:

  misfit        wp_residual: residual and misfit of a batch of shot records
  gradient      autograd.WaveMisfit: the loss of a model and its probed gradient
  forward       wp_probe_forward: propagation with the field projected on r probes
  adjoint       wp_adjoint_image: adjoint propagation, projection and image
  exact         wp_exact_gradient: full history or checkpoints
  offset        wp_offset_image: subsurface-offset volume of stored projections
  range_finder  wp_range_finder: orthonormal probes from the data
  accumulate    wp_probe_accumulate(_static): the contraction alone, on a caller's steps

Models are layered velocities with a smooth perturbation (and a salt body where a true model is
asked for) on interior grids padded by an absorbing layer, as in the package's inputs module, but
drawn on the GPU.  The references in exact() restate the scheme of include/wp.h in FP64 torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

V_MIN, V_MAX, V_CAP = 1500.0, 4500.0, 4725.0   # layered models, 5 % perturbation
EPS_MAX = 0.25                                   # Thomsen epsilon

_FIELD = dict(ny=1, nbl=40, h=12.5, f0=15.0, tti=False, stride=1, layout="aligned")   # of every wave case


def listed():
    return [
        # one two-layer-sized shot record: the smallest call of every gradient
        dict(name="misfit_one_shot", kind="misfit", shots=1, nt=1000, nrec=201),
        # interactive use and tests: one shot on the 201 x 201 grid, 1000 steps, r = 8
        dict(_FIELD, name="gradient_201", kind="gradient", ndim=2, nx=201, nz=201, h=10.0, f0=10.0, nt=1000,
             shots=1, r=8, tb=64),
        # the benchmark's survey (1601 x 401, 1601 receivers, r = 64, blocks of 256 steps), half of
        # its shots and two blocks of its time axis: the forward sweep
        dict(_FIELD, name="forward_salt2d", kind="forward", ndim=2, nx=1601, nz=401, nt=512, shots=32, r=64, tb=256),
        # and the adjoint sweep with the image, keeping P_v as offset volumes need it
        dict(_FIELD, name="adjoint_salt2d", kind="adjoint", ndim=2, nx=1601, nz=401, nt=512, shots=32, r=64, tb=256,
             keep_pv=True),
        # the probe count at which the stacked gradient's error falls below 0.1
        dict(_FIELD, name="forward_salt2d_r448", kind="forward", ndim=2, nx=1601, nz=401, nt=1024, shots=8, r=448, tb=512),
        # the exact baseline of the same survey, in its batches of 16 shots
        dict(_FIELD, name="exact_salt2d", kind="exact", ndim=2, nx=1601, nz=401, nt=256, shots=16, mode="full", ncheck=1),
        # the 3-D isotropic survey (512 x 512 x 256), two blocks of 64 steps, in the default layout
        dict(_FIELD, name="forward_salt3d", kind="forward", ndim=3, nx=512, ny=512, nz=256, h=10.0, f0=12.0, nt=128,
             shots=1, r=32, tb=64, stride=2, layout="dense"),
        # 3-D TTI at a served size, the adjoint sweep
        dict(_FIELD, name="adjoint_tti3d", kind="adjoint", ndim=3, nx=256, ny=256, nz=192, f0=12.0, nt=128, shots=1,
             r=32, tb=64, stride=4, tti=True, keep_pv=False),
        # a served 2-D TTI job (401 x 401, r = 16, blocks of 64 steps), its forward sweep
        dict(_FIELD, name="forward_tti2d", kind="forward", ndim=2, nx=401, nz=401, nt=1000, shots=1, r=16, tb=64, tti=True),
        # common-image gathers: 81 offsets (+-500 m) of 16 shots of the salt survey
        dict(_FIELD, name="offset_salt2d", kind="offset", ndim=2, nx=1601, nz=401, shots=16, r=64, nh=40),
        # data-driven probes for 16 shots
        dict(name="range_finder_data", kind="range_finder", shots=16, nt=2000, ncols=801, r=64, power=1),
        # the contraction of a caller's own time steps on a 201 x 201 grid padded by 40 (odd rows)
        dict(name="accumulate_281", kind="accumulate", shots=16, npoints=281 * 281, nt=1024, t0=256, cnt=256, r=64, static=False),
    ]


# ------------------------------------------------------------------------------------------
# Drawn cases
# ------------------------------------------------------------------------------------------
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(c):
    p = 2 * c["nbl"]
    return (c["nz"] + p, c["ny"] + p if c["ndim"] == 3 else 1, c["nx"] + p)


def _points(c):
    return int(np.prod(_shape(c)))


def _cost(c):
    """A rough cost in bytes moved, to keep drawn cases below the largest listed one."""
    k = c["kind"]
    if k == "misfit":
        return 12.0 * c["shots"] * c["nt"] * c["nrec"]
    if k == "range_finder":
        return 40.0 * c["shots"] * c["nt"] * (c["ncols"] + 8 * c["r"]) * c["power"] + 16.0 * c["shots"] * c["nt"] * c["r"] ** 2
    if k == "accumulate":
        return 4.0 * c["shots"] * c["npoints"] * (c["cnt"] + 3 * c["r"])
    if k == "offset":
        return 8.0 * c["shots"] * c["r"] * _points(c) * (1 + c["nh"] / 16)
    pts = float(_points(c)) * c["shots"] * c["nt"]
    step = (80.0 if c["tti"] else 20.0) * {"forward": 1, "adjoint": 1, "gradient": 2, "exact": 4}[k]
    return pts * step + (16.0 * c.get("r", 0) * pts / c.get("tb", 1) if k != "exact" else 0.0)


def _bytes(c):
    """Device memory of a wave case's state."""
    f = 2 if c["tti"] else 1
    n = float(_points(c)) * c["shots"] * f * 4
    if c["kind"] == "exact":
        return n * ((c["nt"] if c["mode"] == "full" else c["ncheck"] + 2 * c["nt"] / c["ncheck"]) + 12)
    return n * (c["tb"] + (3 if c.get("keep_pv") else 2) * c["r"] + 8)


def _draw(rng):
    kind = rng.choice(["misfit", "gradient", "forward", "forward", "adjoint", "adjoint", "exact", "offset",
                       "range_finder", "accumulate"])
    if kind == "misfit":
        return dict(kind=kind, shots=_log(rng, 1, 32), nt=_log(rng, 200, 4000), nrec=_log(rng, 50, 1601))
    if kind == "range_finder":
        return dict(kind=kind, shots=_log(rng, 1, 16), nt=_log(rng, 300, 2000), ncols=_log(rng, 200, 801),
                    r=_log(rng, 4, 96), power=rng.choice([1, 1, 2]))
    if kind == "accumulate":
        nt = _log(rng, 64, 1024)
        t0 = 8 * rng.randrange(0, nt // 16)
        static = rng.random() < 0.3
        return dict(kind=kind, shots=1 if static else _log(rng, 1, 16), npoints=_log(rng, 1000, 200000), nt=nt, t0=t0,
                    cnt=rng.randint(16, min(512, nt - t0)), r=_log(rng, 4, 256 if static else 512), static=static)
    c = dict(_FIELD, kind=kind, ndim=2 if rng.random() < 0.6 else 3, nbl=rng.choice([20, 40]),
             layout=rng.choice(["aligned", "dense"]))
    if kind in ("gradient", "offset"):
        c["ndim"] = 2
    c["shots"] = 1
    if c["ndim"] == 2:
        c.update(nx=_log(rng, 150, 1601), nz=_log(rng, 100, 401), shots=_log(rng, 1, 32))
    else:
        c.update(nx=_log(rng, 64, 256), ny=_log(rng, 64, 256), nz=_log(rng, 64, 256), stride=4, h=10.0, f0=12.0)
    if kind == "offset":
        c.update(r=_log(rng, 8, 64), nh=rng.randint(0, 64))
        return c
    c["tti"] = rng.random() < 0.35
    c["nt"] = _log(rng, 128, 600) if c["ndim"] == 2 else _log(rng, 48, 128)
    if kind == "exact":
        c["mode"] = "full" if c["ndim"] == 2 and rng.random() < 0.6 else "checkpoint"
        c["ncheck"] = 1 if c["mode"] == "full" else rng.choice([16, 32, 64])
        return c
    c["tb"] = rng.choice([64, 128, 256]) if c["ndim"] == 2 else 64
    c["r"] = _log(rng, 8, 256) if c["ndim"] == 2 else _log(rng, 8, 64)
    if kind == "adjoint":
        c["keep_pv"] = rng.random() < 0.5
    if kind == "gradient":
        c.update(nx=min(c["nx"], 401), shots=min(c["shots"], 4), r=min(c["r"], 64), tb=64)
    return c


def draw(rng):
    top = max(_cost(c) for c in listed())
    while True:
        c = _draw(rng)
        if _cost(c) <= 0.6 * top and (c["kind"] in ("misfit", "range_finder", "accumulate", "offset") or _bytes(c) < 5e10):
            return c


# ------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 2654435761 % (1 << 31))


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device="cuda")


def _smooth(g, nz, ny, nx, cells=16):
    """A smooth random field (nz, ny, nx) with |values| <= 1."""
    low = [max(2, n // cells + 2) if n > 1 else 1 for n in (nz, ny, nx)]
    p = _randn(g, 1, 1, *low)
    if ny == 1:
        p = F.interpolate(p[:, :, :, 0], size=(nz, nx), mode="bilinear", align_corners=True)[0, 0][:, None]
    else:
        p = F.interpolate(p, size=(nz, ny, nx), mode="trilinear", align_corners=True)[0, 0]
    return p / p.abs().max()


def _pad(f, c):
    """Edge values repeated into the absorbing layer."""
    b = c["nbl"]
    if c["ndim"] == 2:
        return F.pad(f[None, :, 0], (b, b, b, b), mode="replicate")[0][:, None].contiguous()
    return F.pad(f[None, None], (b,) * 6, mode="replicate")[0, 0].contiguous()


def _dt(c):
    return 0.4 * c["h"] / (V_CAP * (math.sqrt(1 + 2 * EPS_MAX) if c["tti"] else 1.0))


def _model(c, g):
    """Padded squared slowness of a smooth background model, and the Thomsen fields."""
    nz, ny, nx = c["nz"], c["ny"] if c["ndim"] == 3 else 1, c["nx"]
    z = torch.linspace(0, 1, nz, device="cuda")[:, None, None]
    v = (V_MIN + (V_MAX - V_MIN) * z) * (1 + 0.05 * _smooth(g, nz, ny, nx))
    m = _pad((1.0 / v.double() ** 2).float(), c)
    th = None
    if c["tti"]:
        lim = [EPS_MAX, 0.1, math.radians(40), math.radians(90)]
        th = [_pad(0.5 * hi * (1 + _smooth(g, nz, ny, nx)), c) for hi in lim]
        th[1] = torch.minimum(th[1], th[0])
    return m, th


def _geometry(c):
    """Sources evenly spaced along x one cell deep (3-D: centred in y), receivers on every
    `stride`-th point of the same depth."""
    h, S = c["h"], c["shots"]
    xs = (np.arange(S) + 0.5) * ((c["nx"] - 1) * h / S)
    ys = np.full(S, 0.5 * (c["ny"] - 1) * h if c["ndim"] == 3 else 0.0)
    src = np.stack([xs, ys, np.full(S, h)], 1)[:, None]
    gx = np.arange(0, c["nx"], c["stride"]) * h
    gy = np.arange(0, c["ny"], c["stride"]) * h if c["ndim"] == 3 else np.zeros(1)
    X, Y = np.meshgrid(gx, gy)
    rec = np.stack([X.ravel(), Y.ravel(), np.full(X.size, h)], 1)
    return src, np.broadcast_to(rec, (S,) + rec.shape).copy()


def _ricker(t, f0):
    a = (math.pi * f0 * t) ** 2
    return (1 - 2 * a) * torch.exp(-a)


def _wavelet(c):
    t = torch.arange(c["nt"], device="cuda", dtype=torch.float64) * _dt(c)
    return _ricker(t - 1.5 / c["f0"], c["f0"]).float()


def _records(c, g, src, rec, amp):
    """Shot records (shots, nt, nrec) of six hyperbolic reflections of the wavelet."""
    dt, nt = _dt(c), c["nt"]
    off = torch.from_numpy(np.linalg.norm(rec[:, :, :2] - src[:, :1, :2], axis=2)).cuda().float()
    t = torch.arange(nt, device="cuda").float()[None, :, None] * dt
    par = torch.rand((6, 3), generator=g, device="cuda").tolist()
    out = torch.zeros((c["shots"], nt, rec.shape[1]), device="cuda")
    for a, b, e in par:
        tau = torch.sqrt((nt * dt * (0.05 + 0.8 * a)) ** 2 + (off / (1800.0 + 2700.0 * b)) ** 2)
        out += amp * (2 * e - 1) * _ricker(t - tau[:, None, :], c["f0"])
    return out


def _probes(c, g):
    q = torch.randint(0, 2, (c["shots"], c["nt"], c["r"]), generator=g, device="cuda")
    return (2 * q - 1).float()


def _fields(c):
    return 2 if c["tti"] else 1


def _amp(c):
    """Scale of the modelled data (a point source carries h^ndim of the wavelet)."""
    return 5.0 if c["ndim"] == 2 else 0.1


def _inputs(c, seed):
    """Everything a wave case's call takes, from the seed alone (torch and numpy only)."""
    g = _gen(seed)
    s = {}
    s["m"], s["th"] = _model(c, g)
    s["src"], s["rec"] = _geometry(c)
    s["wavelet"] = _wavelet(c)
    if c["kind"] in ("gradient", "exact"):
        s["d_obs"] = _records(c, g, s["src"], s["rec"], _amp(c))
    if c["kind"] in ("gradient", "forward", "adjoint"):
        s["Q"] = _probes(c, g)
    if c["kind"] == "adjoint":
        s["res"] = _records(c, g, s["src"], s["rec"], _amp(c))
    return s


def _projections(c, g):
    """A stored projection (fields * shots, r, NZ, NY, NX): smooth along x as wavefields are."""
    p = _randn(g, _fields(c) * c["shots"], c["r"], *_shape(c))
    p[..., 1:-1] = 0.5 * p[..., 1:-1] + 0.25 * (p[..., 2:] + p[..., :-2])
    return p


def _layout(c, row_floats, x_pitch):
    """(buffer, view of its points) of projections in the case's layout."""
    rows, (nz, ny, nx) = _fields(c) * c["shots"], _shape(c)
    if c["layout"] == "dense":
        buf = torch.empty((rows, c["r"], nz, ny, nx), device="cuda")
        return buf, buf
    buf = torch.zeros((rows, c["r"], row_floats), device="cuda")
    view = buf[:, :, :nz * ny * x_pitch].unflatten(2, (nz, ny, x_pitch))[..., :nx]
    return buf, view


def _handle(c, s):
    from paper_2201_06914_gb300 import wp
    torch.cuda.current_stream().synchronize()   # the model must be complete before wp_model reads it
    kw = dict(zip(("eps", "delta", "theta", "phi"), s["th"])) if s["th"] else {}
    h = c["h"]
    M = wp.Model(c["ndim"], c["nx"], c["ny"], c["nz"], c["nbl"], h, h, h, _dt(c), c["nt"] if "nt" in c else 1,
                 s["m"], V_CAP, **kw)
    if c["layout"] == "aligned":
        M.use_aligned_probes()
    return M, wp.Geometry(s["src"], s["rec"])


def prepare(case, seed):
    from paper_2201_06914_gb300 import wp
    c, k = case, case["kind"]
    s = {"case": c}
    if k == "misfit":
        g, n = _gen(seed), c["shots"] * c["nt"] * c["nrec"]
        s["d_syn"], s["d_obs"] = _randn(g, n), _randn(g, n)
        s["res"], s["J"] = torch.empty(n, device="cuda"), torch.empty(1, dtype=torch.float64, device="cuda")
        s["ws"] = wp.workspace(wp.wp_residual_workspace_bytes(n))
        return s
    if k == "range_finder":
        s.update(_sketch(c, seed))
        s["Q"] = torch.empty((c["shots"], c["nt"], c["r"]), device="cuda")
        s["ws"] = wp.workspace(wp.wp_range_finder_workspace_bytes(c["nt"], c["ncols"], c["shots"], False, c["r"]))
        return s
    if k == "accumulate":
        s.update(_steps(c, seed))
        s["P"] = torch.empty((c["shots"], c["r"], c["npoints"]), device="cuda")
        if not c["static"]:
            s["ws"] = wp.workspace(wp.wp_probe_accumulate_workspace_bytes(c["shots"], c["nt"], c["r"]))
        return s
    if k == "offset":
        g = _gen(seed)
        s["m"], s["th"] = _model(c, g)
        s["src"], s["rec"] = _geometry(c)
        s["M"], _ = _handle(c, s)
        _, rf, xp = wp.wp_probe_layout(s["M"].handle)
        for n in ("Pu", "Pv"):
            s[n], view = _layout(c, rf, xp)
            view.copy_(_projections(c, g))
        s["out"] = torch.empty((2 * c["nh"] + 1, s["M"].N), device="cuda")
        return s
    s.update(_inputs(c, seed))
    if k == "gradient":
        from paper_2201_06914_gb300.autograd import Problem
        s["m"] = s["m"].requires_grad_()
        s["problem"] = Problem(c["ndim"], c["nx"], c["ny"], c["nz"], c["nbl"], c["h"], _dt(c), c["nt"], s["src"],
                               s["rec"], s["wavelet"], s["d_obs"], s["Q"], Tb=c["tb"], variant="probed",
                               damp_v=V_CAP, thomsen=tuple(s["th"]) if s["th"] else None)
        return s
    s["M"], s["G"] = _handle(c, s)
    M, G = s["M"], s["G"]
    s["g"] = torch.empty(M.N, device="cuda")
    s["d"] = torch.empty((c["shots"], c["nt"], G.nrec), device="cuda")
    if k == "exact":
        s["mode"] = wp.WP_MODE_EXACT_FULL if c["mode"] == "full" else wp.WP_MODE_EXACT_CHECKPOINT
        s["J"] = torch.empty(1, dtype=torch.float64, device="cuda")
        s["ws"] = wp.workspace(wp.wp_workspace_bytes(M.handle, G.c, 0, c["ncheck"], s["mode"]))
        return s
    s["ws"] = wp.workspace(wp.wp_workspace_bytes(M.handle, G.c, c["r"], c["tb"], wp.WP_MODE_PROBED))
    _, rf, xp = wp.wp_probe_layout(M.handle)
    s["Pu"], s["Pu_view"] = _layout(c, rf, xp)
    if k == "adjoint":
        s["Pu_view"].copy_(_projections(c, _gen(seed + 1000003)))
        s["Pv"], s["Pv_view"] = _layout(c, rf, xp) if c["keep_pv"] else (None, None)
    return s


def run(state):
    from paper_2201_06914_gb300 import wp
    s, c = state, state["case"]
    k = c["kind"]
    if k == "misfit":
        wp.wp_residual(s["d_syn"], s["d_obs"], s["res"], s["res"].numel(), s["J"], s["ws"])
        return {"res": s["res"], "J": s["J"]}
    if k == "gradient":
        from paper_2201_06914_gb300.autograd import WaveMisfit
        J = WaveMisfit.apply(s["m"], s["problem"])
        (g,) = torch.autograd.grad(J, s["m"])
        return {"J": J.detach(), "g": g}
    if k == "forward":
        wp.wp_probe_forward(s["M"].handle, s["G"].c, s["wavelet"], s["Q"], c["r"], c["tb"], s["Pu"], s["d"], s["ws"])
        return {"Pu": s["Pu_view"], "d": s["d"]}
    if k == "adjoint":
        wp.wp_adjoint_image(s["M"].handle, s["G"].c, s["res"], s["Q"], c["r"], c["tb"], 1.0 / c["r"], s["Pu"], s["g"],
                            s["Pv"], s["ws"])
        return {"g": s["g"], "Pv": s["Pv_view"]} if c["keep_pv"] else {"g": s["g"]}
    if k == "exact":
        wp.wp_exact_gradient(s["M"].handle, s["G"].c, s["wavelet"], s["d_obs"], s["g"], s["J"], s["d"], s["mode"],
                             c["ncheck"], s["ws"])
        return {"g": s["g"], "J": s["J"].float(), "d": s["d"]}   # the loss at the precision of the model
    if k == "offset":
        wp.wp_offset_image(s["M"].handle, s["Pu"], s["Pv"], c["r"], c["shots"], 1.0 / c["r"], c["nh"], s["out"])
        return {"out": s["out"]}
    if k == "range_finder":
        wp.wp_range_finder(s["D"], c["nt"], c["ncols"], c["shots"], False, c["power"], s["Z"], c["r"], s["Q"], s["ws"])
        return {"Q": s["Q"]}
    s["P"].zero_()   # the first block of a projection
    if c["static"]:
        wp.wp_probe_accumulate_static(s["A"], c["cnt"], c["npoints"], c["shots"], s["Qm"], c["nt"], c["t0"], c["r"], 0.5,
                                      s["P"])
    else:
        wp.wp_probe_accumulate(s["A"], c["cnt"], c["npoints"], c["shots"], s["Qm"], c["nt"], c["t0"], c["r"], 0.5,
                               s["P"], s["ws"])
    return {"P": s["P"]}


def _sketch(c, seed):
    """Shot records of a random reflectivity (band-limited by the wavelet, with noise) and the
    Rademacher sketch of the range finder."""
    g = _gen(seed)
    S, nt, n, r = c["shots"], c["nt"], c["ncols"], c["r"]
    w = _ricker(torch.arange(-20, 21, device="cuda").float() * 1.6e-3, 30.0).double()
    refl = _randn(g, S * n, 1, nt).double()
    D = F.conv1d(refl, w[None, None], padding=20).reshape(S, n, nt).transpose(1, 2)
    D = D + 0.5 * _randn(g, S, nt, n).double()
    Z = (2 * torch.randint(0, 2, (S, nt, r), generator=g, device="cuda") - 1).float()
    return {"D": D.float().contiguous(), "Z": Z}


def _steps(c, seed):
    g = _gen(seed)
    q = 2 * torch.randint(0, 2, (c["shots"], c["nt"], c["r"]), generator=g, device="cuda") - 1
    return {"A": _randn(g, c["shots"], c["cnt"], c["npoints"]), "Qm": q.float()}


# ------------------------------------------------------------------------------------------
# Work
# ------------------------------------------------------------------------------------------
def work(case):
    c, k = case, case["kind"]
    if k == "misfit":
        n = c["shots"] * c["nt"] * c["nrec"]
        return {"bytes": 12 * n, "flops": 3 * n}
    if k == "range_finder":
        S, nt, n, r = c["shots"], c["nt"], c["ncols"], c["r"]
        return {"bytes": 4 * S * (nt * n + 2 * nt * r), "flops": S * c["power"] * (4 * nt * n * r + 2 * nt * r * r)}
    if k == "accumulate":
        S, n = c["shots"], c["npoints"]
        return {"bytes": 4 * S * (n * c["cnt"] + n * c["r"] + c["cnt"] * c["r"]), "flops": 2 * S * n * c["cnt"] * c["r"]}
    N = _points(c)
    if k == "offset":
        n = c["shots"] * c["r"] * N
        return {"bytes": 8 * n + 4 * (2 * c["nh"] + 1) * N, "flops": 2 * (2 * c["nh"] + 1) * n}
    f, S, nt = _fields(c), c["shots"], c["nt"]
    nrec = len(range(0, c["nx"], c["stride"])) * (len(range(0, c["ny"], c["stride"])) if c["ndim"] == 3 else 1)
    step = (40 if c["ndim"] == 2 else 52) if not c["tti"] else (110 if c["ndim"] == 2 else 160)
    sweeps = 2 if k in ("gradient", "exact") else 1
    flops = sweeps * step * N * S * nt
    data = 4 * (N * (1 + (4 if c["tti"] else 0)) + nt)
    rec = 4 * S * nt * nrec
    if k == "exact":
        return {"bytes": data + 2 * rec + 4 * N, "flops": flops + 2 * f * N * S * nt}
    proj, q = 4 * f * S * c["r"] * N, 4 * S * nt * c["r"]
    flops += sweeps * 2 * f * S * N * c["r"] * nt
    if k == "forward":
        return {"bytes": data + q + proj + rec, "flops": flops}
    if k == "adjoint":
        return {"bytes": data + q + (2 if c["keep_pv"] else 1) * proj + rec + 4 * N, "flops": flops + 2 * f * S * N * c["r"]}
    return {"bytes": data + q + rec + 4 * N, "flops": flops + 2 * f * S * N * c["r"]}


# ------------------------------------------------------------------------------------------
# FP64 references
# ------------------------------------------------------------------------------------------
_C2 = (8 / 5, -1 / 5, 8 / 315, -1 / 560)      # second derivative, offsets 1..4
_C1 = (4 / 5, -1 / 5, 4 / 105, -1 / 280)      # first derivative


class _Wave64:
    """The leapfrog scheme in FP64 on fields (shots, NZ, NY, NX), zero beyond the grid."""

    def __init__(self, c, s):
        self.c, self.h, self.dt = c, c["h"], _dt(c)
        self.axes = (1, 3) if c["ndim"] == 2 else (1, 2, 3)
        shape = _shape(c)
        self.b = (self.dt ** 2 / s["m"].detach().double()).reshape((1,) + shape)
        nbl = c["nbl"]
        s0 = 3 * V_CAP * math.log(1000.0) / (2 * nbl * self.h) * self.dt / 2
        sd = torch.zeros((1,) + shape, dtype=torch.float64, device="cuda")
        for ax in self.axes:
            n = shape[ax - 1]
            i = torch.arange(n, device="cuda")
            dist = torch.clamp(torch.maximum(nbl - i, i - (n - nbl - 1)), min=0).double() / nbl
            sd += (s0 * dist ** 2).reshape([n if a == ax else 1 for a in range(4)])
        self.cp, self.cm = 1 + sd, 1 - sd
        if s["th"]:
            eps, delta, theta, phi = (t.double().reshape((1,) + shape) for t in s["th"])
            self.E, self.S = 1 + 2 * eps, torch.sqrt(1 + 2 * delta)
            phi = phi if c["ndim"] == 3 else torch.zeros_like(phi)
            a = {3: torch.sin(theta) * torch.cos(phi), 2: torch.sin(theta) * torch.sin(phi), 1: torch.cos(theta)}
            self.a = {ax: a[ax] for ax in self.axes}

    def lap(self, u):
        out = u * (-2 * sum(_C2) * len(self.axes))
        for ax in self.axes:
            n = u.shape[ax]
            for k, ck in enumerate(_C2, 1):
                if k < n:
                    out.narrow(ax, 0, n - k).add_(u.narrow(ax, k, n - k), alpha=ck)
                    out.narrow(ax, k, n - k).add_(u.narrow(ax, 0, n - k), alpha=ck)
        return out.div_(self.h ** 2)

    def d1(self, u, ax):
        out, n = torch.zeros_like(u), u.shape[ax]
        for k, ck in enumerate(_C1, 1):
            if k < n:
                out.narrow(ax, 0, n - k).add_(u.narrow(ax, k, n - k), alpha=ck / self.h)
                out.narrow(ax, k, n - k).add_(u.narrow(ax, 0, n - k), alpha=-ck / self.h)
        return out

    def hz(self, u):
        t = sum(self.a[ax] * self.d1(u, ax) for ax in self.axes)
        return sum(self.d1(self.a[ax] * t, ax) for ax in self.axes)

    def corners(self, xyz):
        """Flat indices and linear weights (shots, points, corners) of positions in metres."""
        nz, ny, nx = _shape(self.c)
        p = torch.from_numpy(np.ascontiguousarray(xyz)).cuda() / self.h + self.c["nbl"]
        if self.c["ndim"] == 2:
            p[..., 1] = 0
        b = torch.floor(p)
        f, b = p - b, b.long()
        idx, w = [], []
        for cz in (0, 1):
            for cy in (0, 1) if self.c["ndim"] == 3 else (0,):
                for cx in (0, 1):
                    idx.append(((b[..., 2] + cz) * ny + b[..., 1] + cy) * nx + b[..., 0] + cx)
                    t = (f[..., 0] if cx else 1 - f[..., 0]) * (f[..., 2] if cz else 1 - f[..., 2])
                    w.append(t * (f[..., 1] if cy else 1 - f[..., 1]) if self.c["ndim"] == 3 else t)
        return torch.stack(idx, -1), torch.stack(w, -1)

    def sweep(self, points, values, steps, adjoint, each):
        """Marches the fields over `steps`, injecting values(n) (shots, points) at `points`, and
        calls each(n, new increments, old increments, new fields) after every step."""
        S, nf = self.c["shots"], _fields(self.c)
        u = [torch.zeros((S,) + _shape(self.c), dtype=torch.float64, device="cuda") for _ in range(nf)]
        d = [torch.zeros_like(x) for x in u]
        idx, w = self.corners(points)
        idx = idx.reshape(S, -1)
        for n in steps:
            if nf == 1:
                r = [self.lap(u[0])]
            elif not adjoint:
                z0, z1 = self.hz(u[0]), self.hz(u[1])
                h0 = self.lap(u[0]) - z0
                r = [self.E * h0 + self.S * z1, self.S * h0 + z1]
            else:
                e, f = self.E * u[0] + self.S * u[1], self.S * u[0] + u[1]
                r = [self.lap(e) - self.hz(e), self.hz(f)]
            q = (w * values(n)[..., None]).reshape(S, -1)
            for x in r[:1] if adjoint else r:
                x.view(S, -1).scatter_add_(1, idx, q)
            old = d
            d = [x.mul_(self.b).addcmul_(self.cm, y).div_(self.cp) for x, y in zip(r, old)]
            for x, y in zip(u, d):
                x.add_(y)
            each(n, d, old, u)

    def utt(self, new, old):
        return (self.cp * new - self.cm * old) / self.dt ** 2


class _Project:
    """P[field][shot] += sum_n Q[shot][n] a[n], in blocks of 16 steps."""

    def __init__(self, c, Q):
        self.Q, self.S, self.nf = Q.double(), c["shots"], _fields(c)
        self.P = torch.zeros((c["shots"], self.nf, c["r"], _points(c)), dtype=torch.float64, device="cuda")
        self.n, self.a = [], []

    def add(self, n, fields):
        self.n.append(n)
        self.a.append(torch.stack([x.reshape(self.S, -1) for x in fields], 1))
        if len(self.n) == 16:
            self.flush()

    def flush(self):
        if self.n:
            q = self.Q[:, self.n].transpose(1, 2)
            for f in range(self.nf):
                for s in range(self.S):
                    self.P[s, f].addmm_(q[s], torch.stack([x[s, f] for x in self.a]))
        self.n, self.a = [], []
        return self.P


def _forward64(W, c, s, each):
    src = torch.ones((c["shots"], s["src"].shape[1]), dtype=torch.float64, device="cuda")
    wav = s["wavelet"].double()
    ridx, rw = W.corners(s["rec"])
    d = torch.empty((c["shots"], c["nt"], s["rec"].shape[1]), dtype=torch.float64, device="cuda")

    def step(n, new, old, u):
        x = u[0].reshape(c["shots"], -1).gather(1, ridx.reshape(c["shots"], -1)).reshape(rw.shape)
        d[:, n] = (x * rw).sum(-1)
        each(n, new, old)

    W.sweep(s["src"], lambda n: src * wav[n], range(c["nt"]), False, step)
    return d


def exact(case, seed):
    c, k = case, case["kind"]
    if k == "misfit":
        g, n = _gen(seed), c["shots"] * c["nt"] * c["nrec"]
        res = _randn(g, n).double() - _randn(g, n).double()
        return {"res": res, "J": 0.5 * (res * res).sum().reshape(1)}
    if k == "range_finder":
        t = _sketch(c, seed)
        D, Y = t["D"].double(), t["Z"].double()
        for _ in range(c["power"]):
            Y, R = torch.linalg.qr(D @ (D.transpose(1, 2) @ Y))
            Y = Y * torch.sign(torch.diagonal(R, dim1=1, dim2=2))[:, None]
        return {"Q": Y}
    if k == "accumulate":
        t = _steps(c, seed)
        q = t["Qm"][:, c["t0"]:c["t0"] + c["cnt"]].double().transpose(1, 2)
        return {"P": torch.stack([0.5 * (q[i] @ t["A"][i].double()) for i in range(c["shots"])])}
    if k == "offset":
        g, nx, nh = _gen(seed), _shape(c)[2], c["nh"]
        _model(c, g)
        Pu, Pv = _projections(c, g), _projections(c, g)
        out = torch.zeros((2 * nh + 1,) + _shape(c), dtype=torch.float64, device="cuda")
        for s in range(c["shots"]):
            u, v = Pu[s].double(), Pv[s].double()
            for h in range(-nh, nh + 1):
                n = nx - 2 * abs(h)
                if n > 0:
                    i = abs(h)
                    out[h + nh][..., i:i + n] += (u[..., i + h:i + h + n] * v[..., i - h:i - h + n]).sum(0)
        return {"out": out.reshape(2 * nh + 1, -1) / c["r"]}
    s = _inputs(c, seed)
    W, S, nt = _Wave64(c, s), c["shots"], c["nt"]
    rows, shape = _fields(c) * S, _shape(c)
    if k == "forward":
        P = _Project(c, s["Q"])
        d = _forward64(W, c, s, lambda n, new, old: P.add(n, [W.utt(x, y) for x, y in zip(new, old)]))
        return {"Pu": P.flush().reshape((rows, c["r"]) + shape), "d": d}
    if k == "exact":
        hist = []
        if 8.0 * rows * nt * _points(c) > 1.2e11:
            return None
        d = _forward64(W, c, s, lambda n, new, old: hist.append([W.utt(x, y) for x, y in zip(new, old)]))
        res = d - s["d_obs"].double()
        g = torch.zeros(shape, dtype=torch.float64, device="cuda")

        def image(n, new, old, v):
            for a, b in zip(hist[n], v):
                g.add_((a * b).sum(0))

        W.sweep(s["rec"], lambda n: -res[:, n], reversed(range(nt)), True, image)
        return {"g": g.reshape(-1), "J": 0.5 * (res * res).sum().reshape(1), "d": d}
    if k == "gradient":
        P = _Project(c, s["Q"])
        d = _forward64(W, c, s, lambda n, new, old: P.add(n, [W.utt(x, y) for x, y in zip(new, old)]))
        res, Pu = d - s["d_obs"].double(), P.flush().reshape((rows, c["r"], -1))
    else:
        res, Pu = s["res"].double(), _projections(c, _gen(seed + 1000003)).reshape(rows, c["r"], -1)
    P = _Project(c, s["Q"])
    W.sweep(s["rec"], lambda n: -res[:, n], reversed(range(nt)), True, lambda n, new, old, v: P.add(n, v))
    Pv = P.flush().reshape(rows, c["r"], -1)
    g = sum((Pu[i].double() * Pv[i]).sum(0) for i in range(rows)) / c["r"]
    if k == "adjoint":
        return {"g": g, "Pv": Pv.reshape((rows, c["r"]) + shape)} if c["keep_pv"] else {"g": g}
    return {"J": 0.5 * (res * res).sum(), "g": g.reshape(s["m"].shape)}
