"""Performance cases of the library's public entry points.

Every case is one call (or one short run of iterations) that a reconstruction
program makes: a projection, a transpose, a data-term gradient, a
preconditioner application, a few PSPS iterations.  Sizes are those of the
repository's workloads (64^2 parallel beam, 256^2..512^2 fan-beam slices,
128^3 and 256^3 cone beam, 720 x 888 projection-domain rays); ``draw`` spreads
them over the range in between, odd sizes included.

``exact`` evaluates the same mathematics in 64 bits with torch alone (Joseph's
projector, the polyenergetic model, the iteration), so results can be held to
it element by element.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2010_01371_gb300 as psps

PAR2D, FAN2D, CONE3D = 0, 1, 2
F64 = torch.float64
CHUNK = 1 << 25        # samples evaluated at once by the 64-bit projector


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # A small parallel-beam study (64^2 image, 90 x 96 rays), ten Haar-preconditioned iterations with line
        # search: every kernel is tiny, so launches and latency decide.
        {"name": "step_par64_haar", "kind": "step", "scan": "par", "nx": 64, "ny": 64, "views": 90, "bins": 96,
         "fov": 64.0, "mats": 1, "spectrum": "mono", "precond": "haar", "iters": 10},
        # The forward projection of a standard fan-beam slice (q = A p of every iteration).
        {"name": "project_fan512", "kind": "project", "scan": "fan", "nx": 512, "ny": 512, "views": 720, "bins": 888,
         "fov": 256.0, "mats": 1},
        # Its transpose for the two numerators (gradient and curvature) of one material.
        {"name": "backproject_fan512", "kind": "backproject", "scan": "fan", "nx": 512, "ny": 512, "views": 720,
         "bins": 888, "fov": 256.0, "chans": 2},
        # Three basis materials of a smaller slice of a batch (448^2, 780 bins).
        {"name": "project_fan448_3mat", "kind": "project", "scan": "fan", "nx": 448, "ny": 448, "views": 720,
         "bins": 780, "fov": 224.0, "mats": 3},
        # The six numerators of a three-material slice (320^2, 556 bins).
        {"name": "backproject_fan320_6ch", "kind": "backproject", "scan": "fan", "nx": 320, "ny": 320, "views": 720,
         "bins": 556, "fov": 160.0, "chans": 6},
        # Dual-energy cone beam at 128^3: forward projection of two basis volumes.
        {"name": "project_cone128_2mat", "kind": "project", "scan": "cone", "nx": 128, "ny": 128, "nz": 128,
         "views": 180, "bins": 256, "rows": 192, "mats": 2},
        # ... and the transpose of its four numerators.
        {"name": "backproject_cone128_4ch", "kind": "backproject", "scan": "cone", "nx": 128, "ny": 128, "nz": 128,
         "views": 180, "bins": 256, "rows": 192, "chans": 4},
        # The largest scan: data-term gradient of two basis volumes of 256^3 from 360 x 384 x 512 dual-energy counts
        # (the adjoint call of a program that brings its own optimiser).
        {"name": "gradient_cone256", "kind": "gradient", "scan": "cone", "nx": 256, "ny": 256, "nz": 256,
         "views": 360, "bins": 512, "rows": 384, "mats": 2, "spectrum": "dual", "blur": 0, "noise": 0.0},
        # Projection-domain decomposition of 720 x 888 dual-kVp rays, per-ray 2 x 2 blocks: no projector, the
        # spectral model and its line search are everything.
        {"name": "step_rays_dual_block", "kind": "step", "scan": "rays", "views": 720, "bins": 888, "mats": 2,
         "spectrum": "dual", "precond": "block", "iters": 2},
        # One-step decomposition of a 512^2 slice: 3 materials, 4 photon-counting channels, per-pixel 3 x 3 blocks.
        {"name": "step_fan512_3mat_block", "kind": "step", "scan": "fan", "nx": 512, "ny": 512, "views": 720,
         "bins": 888, "fov": 256.0, "mats": 3, "spectrum": "counting", "precond": "block", "iters": 2},
        # The cross-material Fourier preconditioner of a 448^2 slice (mixed radix), applied once.
        {"name": "apply_448_block_fourier", "kind": "apply", "nx": 448, "ny": 448, "mats": 3,
         "precond": "block_fourier", "op": "M"},
        # Data-term gradient with detector cross-talk and correlated noise along 888-cell rows.
        {"name": "gradient_rays_blur_noise", "kind": "gradient", "scan": "rays", "views": 720, "bins": 888, "mats": 2,
         "spectrum": "dual", "blur": 3, "noise": 0.4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_scan(rng, kinds):
    scan = rng.choice(kinds)
    if scan == "rays":
        return {"scan": "rays", "views": _log(rng, 60, 720), "bins": _log(rng, 64, 888)}
    if scan == "cone":
        n = _log(rng, 32, 160)
        return {"scan": "cone", "nx": n, "ny": max(24, int(n * rng.uniform(0.8, 1.0))),
                "nz": max(16, int(n * rng.uniform(0.4, 1.0))), "views": _log(rng, 24, 180),
                "bins": max(48, int(n * rng.uniform(1.5, 2.0))), "rows": max(32, int(n * rng.uniform(1.0, 1.5)))}
    n = _log(rng, 48, 512)
    return {"scan": scan, "nx": n, "ny": max(40, int(n * rng.uniform(0.75, 1.0))), "views": _log(rng, 60, 720),
            "bins": max(64, int(n * rng.uniform(1.3, 1.8))), "fov": n * rng.choice([0.5, 0.55, 0.4])}


def draw(rng):
    kind = rng.choice(["project", "project", "backproject", "backproject", "gradient", "step", "apply"])
    if kind == "project":
        c = _draw_scan(rng, ["par", "fan", "fan", "cone", "cone"])
        c["mats"] = rng.choice([1, 2, 3, 4])
    elif kind == "backproject":
        c = _draw_scan(rng, ["par", "fan", "fan", "cone", "cone"])
        c["chans"] = rng.choice([1, 2, 3, 4, 6])
    elif kind == "gradient":
        c = _draw_scan(rng, ["rays", "fan", "cone"])
        c["mats"], c["spectrum"] = rng.choice([(1, "mono"), (2, "dual"), (3, "counting")])
        c["blur"] = rng.choice([0, 0, 1, 3])
        c["noise"] = rng.choice([0.0, 0.0, 0.4])
    elif kind == "step":
        c = _draw_scan(rng, ["rays", "fan", "par", "cone"])
        c["mats"], c["spectrum"] = rng.choice([(1, "mono"), (2, "dual"), (3, "counting")])
        c["precond"] = rng.choice(["none", "block"])
        c["iters"] = rng.choice([1, 2, 3])
    else:
        c = {"precond": rng.choice(["haar", "block_fourier", "block"]), "mats": rng.choice([2, 3])}
        if c["precond"] == "haar":
            c["nx"] = c["ny"] = rng.choice([64, 128, 256, 512])
            c["mats"] = 1
        elif c["precond"] == "block_fourier":
            c["nx"], c["ny"] = (rng.choice([60, 90, 128, 160, 224, 250, 320, 384, 441, 512]) for _ in range(2))
        else:
            c["nx"], c["ny"] = _log(rng, 48, 512), _log(rng, 48, 512)
        c["op"] = rng.choice(["M", "MT", "absM", "absMT"])
    c["kind"] = kind
    return c


# ------------------------------------------------------------------ inputs

def _gen(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 8 + what)
    return g


def _geometry(case):
    """Scan geometry with the fields of ``mbir_geometry`` (None: bare rays)."""
    if case["scan"] == "rays":
        return None
    nx, ny, nz = case["nx"], case["ny"], case.get("nz", 1)
    g = SimpleNamespace(nx=nx, ny=ny, nz=nz, n_views=case["views"], n_u=case["bins"], n_v=case.get("rows", 1),
                        angle0=0.0, angle_span=2 * math.pi, sid=0.0, sdd=0.0, dz=1.0, dv=1.0)
    if case["scan"] == "cone":
        g.kind, g.sid, g.sdd = CONE3D, 600.0, 1200.0
        g.dx = g.dy = g.dz = 128.0 / max(nx, ny)
        g.du, g.dv = 0.8 * 512 / g.n_u, 0.8 * 384 / g.n_v
        g.image_shape, g.sino_shape = (nz, ny, nx), (g.n_views, g.n_v, g.n_u)
        return g
    g.dx = g.dy = case["fov"] / max(nx, ny)
    if case["scan"] == "fan":
        g.kind, g.sid, g.sdd = FAN2D, 500.0, 1000.0
        g.du = 888.0 / 256.0 * case["fov"] / g.n_u
    else:
        g.kind, g.angle_span = PAR2D, math.pi
        g.du = 1.5 * case["fov"] / g.n_u
    g.image_shape, g.sino_shape = (ny, nx), (g.n_views, g.n_u)
    return g


def _n_rays(case):
    return case["views"] * case["bins"] * case.get("rows", 1)


def _ellipses(seed, n):
    """Unit-square ellipses (cx, cy, cz, a, b, c, value): a body and n - 1 inserts."""
    r = np.random.default_rng(seed)
    out = [(0.0, 0.0, 0.0, 0.43, 0.35, 0.39, 1.0)]
    for _ in range(n - 1):
        rad, th = r.uniform(0, 0.25), r.uniform(0, 2 * math.pi)
        out.append((rad * math.cos(th), rad * math.sin(th), r.uniform(-0.2, 0.2), r.uniform(0.02, 0.09),
                    r.uniform(0.02, 0.09), r.uniform(0.02, 0.09), r.uniform(-0.4, 0.8)))
    return out


def _image(case, geom, seed, mats):
    """Basis images: piecewise-constant phantoms with a little texture."""
    size = geom.dx * max(geom.nx, geom.ny)
    ax = [(torch.arange(n, device="cuda", dtype=torch.float32) - (n - 1) / 2) * (d / size)
          for n, d in ((geom.nz, geom.dz), (geom.ny, geom.dy), (geom.nx, geom.dx))]
    z, y, x = torch.meshgrid(*ax, indexing="ij")
    if geom.kind != CONE3D:
        z = torch.zeros_like(z)
    out = torch.empty((mats,) + tuple(geom.image_shape), device="cuda")
    for m in range(mats):
        img = torch.zeros_like(x)
        for k, (cx, cy, cz, a, b, c, v) in enumerate(_ellipses(seed * 4 + m, 7)):
            if m > 0 and k == 0:
                continue                       # bone- and iodine-like materials are inserts only
            img += abs(v) * (((x - cx) / a) ** 2 + ((y - cy) / b) ** 2 + ((z - cz) / c) ** 2 <= 1.0)
        img *= (1.0, 0.3, 0.02, 0.05)[m % 4]
        img *= 1.0 + 0.02 * torch.randn(img.shape, generator=_gen(seed, m), device="cuda")
        out[m] = img.reshape(geom.image_shape)
    return out * (0.02 if mats == 1 else 1.0)


def _rays(geom, views=None):
    """Origins and unit directions of the rays of some views (64 bits)."""
    views = range(geom.n_views) if views is None else views
    be = torch.tensor([geom.angle0 + v * (geom.angle_span / geom.n_views) for v in views], dtype=F64, device="cuda")
    u = (torch.arange(geom.n_u, device="cuda", dtype=F64) - (geom.n_u - 1) / 2) * geom.du
    c, s = torch.cos(be)[:, None], torch.sin(be)[:, None]
    if geom.kind == PAR2D:
        o = torch.stack([-s * u, c * u], -1)
        d = torch.stack([-c + 0 * u, -s + 0 * u], -1)
    elif geom.kind == FAN2D:
        ga = u / geom.sdd
        o = torch.stack([geom.sid * c + 0 * u, geom.sid * s + 0 * u], -1)
        d = torch.stack([-torch.cos(be[:, None] - ga), -torch.sin(be[:, None] - ga)], -1)
    else:
        w = (torch.arange(geom.n_v, device="cuda", dtype=F64) - (geom.n_v - 1) / 2) * geom.dv
        c, s, u, w = c[..., None], s[..., None], u[None, None, :], w[None, :, None]
        o = torch.stack(torch.broadcast_tensors(geom.sid * c, geom.sid * s, 0 * u + 0 * w), -1)
        d = torch.stack(torch.broadcast_tensors(-geom.sdd * c - u * s, -geom.sdd * s + u * c, w), -1)
        o, d = torch.broadcast_tensors(o, d)
        d = d / d.norm(dim=-1, keepdim=True)
    return o, d


def _chords(case, geom, seed, mats):
    """Analytic line integrals of the phantoms, [mats][n_rays] (mm x density)."""
    n = _n_rays(case)
    out = torch.empty((mats, n), device="cuda")
    if geom is None:                           # bare rays: independent line integrals
        g = _gen(seed, 5)
        for m in range(mats):
            out[m] = torch.rand(n, generator=g, device="cuda") * (300.0, 30.0, 1.0, 1.0)[m % 4]
        return out
    size, per = geom.dx * max(geom.nx, geom.ny), geom.n_u * geom.n_v
    step = max(1, CHUNK // per)
    for v0 in range(0, geom.n_views, step):
        o, d = (t.float().reshape(-1, t.shape[-1]) for t in _rays(geom, range(v0, min(v0 + step, geom.n_views))))
        for m in range(mats):
            tot = torch.zeros(o.shape[0], device="cuda")
            for k, (cx, cy, cz, a, b, c, val) in enumerate(_ellipses(seed * 4 + m, 7)):
                if m > 0 and k == 0:
                    continue
                ctr = torch.tensor([cx, cy, cz][:o.shape[1]], device="cuda") * size
                ext = torch.tensor([a, b, c][:o.shape[1]], device="cuda") * size
                p, q = (o - ctr) / ext, d / ext
                A, B, C = (q * q).sum(-1), 2 * (p * q).sum(-1), (p * p).sum(-1) - 1
                tot += abs(val) * torch.sqrt(torch.clamp(B * B - 4 * A * C, min=0)) / A
            out[m, v0 * per:v0 * per + tot.numel()] = tot * (1.0, 0.3, 0.02, 0.05)[m % 4]
    return out * (0.02 if mats == 1 else 1.0)


def _spectrum(case):
    """(Q [E][m], S [c][E]): one energy, two kVp settings or four photon-counting windows."""
    kind, mats = case["spectrum"], case["mats"]
    if kind == "mono":
        return np.ones((1, mats)), np.full((1, 1), 1e5)
    E = np.arange(20.0, 141.0 if kind == "dual" else 121.0)

    def kramers(kvp):
        s = np.clip(kvp - E, 0, None) * np.exp(-2.0 * (0.27 * (E / 30) ** -3 + 0.035 * (E / 30) ** -0.3))
        return s / s.sum()
    Q = np.zeros((E.size, mats))
    for m in range(mats):
        a, b = ((0.2, 0.17), (1.0, 0.2), (10.0, 0.25))[m]
        Q[:, m] = 0.1 * (a * (E / 30) ** -3 + b * (E / 30) ** -0.3)
        if m == 2:
            Q[E >= 33.2, m] *= 6.0
    if kind == "dual":
        return Q, 1e5 * np.stack([kramers(80.0), kramers(140.0)])
    s, edges = kramers(120.0), [25.0, 40.0, 60.0, 80.0, 121.0]
    return Q, 1e5 * np.stack([s * ((E >= lo) & (E < hi)) for lo, hi in zip(edges[:-1], edges[1:])])


def _counts(case, l, Q, S, seed):
    """Poisson counts [c][n_rays] of the polyenergetic model at line integrals l."""
    y = torch.zeros((S.shape[0], l.shape[1]), device="cuda")
    for e in range(Q.shape[0]):
        if not S[:, e].any():
            continue
        z = sum(float(Q[e, m]) * l[m] for m in range(l.shape[0]))
        t = torch.exp_(z.neg_() if z.data_ptr() != l.data_ptr() else -z)
        for c in range(S.shape[0]):
            if S[c, e]:
                y[c].add_(t, alpha=float(S[c, e]))
    g = _gen(seed, 6)
    for c in range(S.shape[0]):
        y[c] = torch.poisson(y[c], generator=g)
    return y


def _numerators(case, geom, seed):
    """Gradient- and curvature-like sinograms, [chans][n_rays]: the first half signed residual terms of a fit to
    Poisson counts, the second half positive curvatures spanning the range of 1 / counts."""
    ch = case["chans"]
    l = _chords(case, geom, seed, 1)[0]
    l = l * (5.0 / l.max().clamp(min=1e-6))
    y = torch.poisson(1e5 * torch.exp(-l), generator=_gen(seed, 7))
    out = torch.empty((ch, l.numel()), device="cuda")
    for c in range(ch):
        m = c % ((ch + 1) // 2)
        yb = 1e5 * torch.exp(-l * (0.9 + 0.05 * m))
        v = (yb - y) / y.clamp(min=1.0) * (1.0, 0.2, 3.0)[m % 3]
        out[c] = -v * yb if c < (ch + 1) // 2 else 100.0 * (1e10 / y.clamp(min=1.0) + v * 1e5).clamp(min=0.0)
    return out


def _haar_scales(n, seed):
    """Eigenvalue estimates of a smoothing system in the Haar basis (larger at coarse levels) and its diagonal M0."""
    g = _gen(seed, 3)
    lam = torch.ones((n, n), device="cuda")
    h = n
    while h >= 2:
        lam[:h, :h] *= 1.6
        h //= 2
    lam *= 1.0 + 0.2 * torch.rand((n, n), generator=g, device="cuda")
    return lam, 0.5 + torch.rand((n, n), generator=g, device="cuda")


def _blocks(n, mats, seed):
    """Symmetric positive definite M0 blocks [m][k][n], materials of different scale."""
    g = _gen(seed, 4)
    d = torch.tensor([1.0, 2.0, 12.0, 5.0][:mats], device="cuda")
    out = torch.empty((mats, mats, n), device="cuda")
    for a in range(mats):
        for b in range(a, mats):
            v = (0.7 + 0.6 * torch.rand(n, generator=g, device="cuda")) * torch.sqrt(d[a] * d[b])
            out[a, b] = out[b, a] = v if a == b else -0.15 * v
    return out


def _cross_spectrum(nx, ny, mats, seed):
    """Per-frequency symmetric blocks [m][k][ny*nx], even in frequency, larger at low frequencies."""
    fy = torch.fft.fftfreq(ny, device="cuda").abs()[:, None]
    fx = torch.fft.fftfreq(nx, device="cuda").abs()[None, :]
    r = torch.sqrt(fx * fx + fy * fy)
    lam = torch.empty((mats, mats, ny * nx), device="cuda")
    s = np.random.default_rng(seed).uniform(0.5, 1.5, (mats, mats))
    for a in range(mats):
        for b in range(a, mats):
            v = (1.0 + 0.5 * a) / (0.05 + 0.5 * (s[a, b] + s[b, a]) * r) if a == b else 0.2 / (0.2 + s[a, b] * r)
            lam[a, b] = lam[b, a] = v.reshape(-1)
    return lam


BETA = np.array([[0.5, 0.1, 3.1], [0.1, 2.1, 6.4], [3.1, 6.4, 1960.0]])
TAPS = {1: (0.15, 0.70, 0.15), 3: (0.02, 0.06, 0.20, 0.44, 0.18, 0.07, 0.03)}


def _beta(case):
    if case["scan"] == "rays":
        return None
    return np.full((1, 1), 1e4) if case["mats"] == 1 else BETA[:case["mats"], :case["mats"]]


def _inputs(case, seed):
    """The arrays of a case (everything a pass reads), as CUDA tensors."""
    kind = case["kind"]
    if kind == "apply":
        n, mats = case["nx"] * case["ny"], case["mats"]
        shape = (mats, case["ny"], case["nx"])
        s = {"v": torch.randn(shape, generator=_gen(seed, 0), device="cuda")}
        if case["op"].startswith("abs"):
            s["v"] = s["v"].abs_()
        if case["precond"] == "haar":
            s["lam"], s["m0"] = _haar_scales(case["nx"], seed)
        else:
            s["blocks"] = _blocks(n, mats, seed)
            if case["precond"] == "block_fourier":
                s["lam"] = _cross_spectrum(case["nx"], case["ny"], mats, seed)
        return s
    geom = _geometry(case)
    if kind == "project":
        return {"x": _image(case, geom, seed, case["mats"])}
    if kind == "backproject":
        return {"s": _numerators(case, geom, seed)}
    Q, S = _spectrum(case)
    l = _chords(case, geom, seed, case["mats"])
    s = {"y": _counts(case, l, Q, S, seed)}
    if kind == "gradient":                     # an early iterate: most of the attenuation, with its own errors
        s["x"] = l * 0.6 if geom is None else 0.6 * _image(case, geom, seed, case["mats"])
        return s
    n = l.shape[1] if geom is None else int(np.prod(geom.image_shape))
    if case["precond"] == "block":
        s["blocks"] = _blocks(n, case["mats"], seed)
    elif case["precond"] == "haar":
        s["lam"], s["m0"] = _haar_scales(case["nx"], seed)
    return s


def prepare(case, seed):
    state = _inputs(case, seed)
    state["case"] = case
    kind = case["kind"]
    if kind == "apply":
        geom = SimpleNamespace(kind=PAR2D, nx=case["nx"], ny=case["ny"], nz=1, dx=1.0, dy=1.0, dz=1.0, n_views=4,
                               angle0=0.0, angle_span=math.pi, n_u=8, n_v=1, du=1.0, dv=1.0, sid=0.0, sdd=0.0,
                               image_shape=(case["ny"], case["nx"]), sino_shape=(4, 8))
    else:
        geom = _geometry(case)
    plan = state["plan"] = psps.Plan(geom) if geom is not None else None
    if kind in ("gradient", "step", "apply"):
        Q, S = _spectrum(case) if kind != "apply" else (np.ones((1, case["mats"])), np.ones((1, 1)))
        spec = state["spec"] = psps.Spectrum(Q, S)
        if case.get("blur"):
            spec.set_blur(TAPS[case["blur"]], case["bins"])
        if case.get("noise"):
            spec.set_noise(case["noise"], case["bins"])
    if kind == "apply" or (kind == "step" and case["precond"] != "none"):
        state["pc"] = psps.Precond(plan, spec, case["precond"], lam=state.get("lam"), m0=state.get("m0"),
                                   blocks=state.get("blocks"))
    if kind == "step":
        state["state"] = psps.State(plan, spec, state.get("pc"), state["y"], _beta(case), graph=True)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "project":
        return psps.mbir_project(state["plan"], state["x"])
    if kind == "backproject":
        return psps.mbir_backproject(state["plan"], state["s"])
    if kind == "gradient":
        return psps.mbmd_gradient(state["plan"], state["spec"], state["x"], state["y"], with_objective=False)[0]
    if kind == "apply":
        return psps.psps_precondition(state["pc"], case["op"], state["v"])
    psps.psps_step(state["state"], case["iters"], history=False)
    return psps.psps_get_image(state["state"])


def work(case):
    kind = case["kind"]
    if kind == "apply":
        n, m = case["nx"] * case["ny"], case["mats"]
        tab = {"haar": 2, "block": m * m, "block_fourier": 2 * m * m}[case["precond"]]
        fft = 10.0 * math.log2(n) if case["precond"] == "block_fourier" else 16.0
        return {"bytes": 4.0 * n * (2 * m + tab), "flops": n * m * (fft + 4.0 * m)}
    rays = _n_rays(case)
    image = case["scan"] != "rays"
    pix = case["nx"] * case["ny"] * case.get("nz", 1) if image else rays
    # samples: about three quarters of the driving planes of a ray lie inside the image
    smp = 0.75 * rays * max(case["nx"], case["ny"]) if image else 0.0
    tap = 11.0 if case["scan"] == "cone" else 4.0
    if kind in ("project", "backproject"):
        m = case.get("mats", case.get("chans"))
        return {"bytes": 4.0 * m * (pix + rays), "flops": smp * tap * m}
    Q, S = _spectrum(case)
    ne, m, nc = Q.shape[0], case["mats"], S.shape[0]
    if kind == "gradient":
        fl = 2 * smp * tap * m + rays * ne * (8.0 * m + 4.0 * nc)
        return {"bytes": 4.0 * (2 * m * pix + nc * rays), "flops": fl}
    per = (3 * m * smp * tap + rays * ne * (10.0 * m + 6.0 * nc) + 3 * rays * ne * (5.0 * m + 7.0 * nc))
    blk = {"none": 0, "block": m * m, "haar": 2}[case["precond"]]
    return {"bytes": case["iters"] * 4.0 * ((4 * m + blk) * pix + (4 * m + nc) * rays), "flops": case["iters"] * per}


# ------------------------------------------------------------------ 64 bits

class _Joseph:
    """Joseph's projector in 64 bits: the axis with the largest direction component drives, one linearly
    (3-D: bilinearly) interpolated sample per pixel plane of that axis."""

    def __init__(self, g):
        self.g = g

    def _chunks(self):
        g = self.g
        per = g.n_u * g.n_v * max(g.nx, g.ny)
        step = max(1, CHUNK // per)
        for v0 in range(0, g.n_views, step):
            views = range(v0, min(v0 + step, g.n_views))
            yield slice(v0 * g.n_u * g.n_v, views[-1] * g.n_u * g.n_v + g.n_u * g.n_v), views

    def _plane(self, o, d, fam):
        """In-plane split of the rays driven along axis fam (0: x, 1: y): lower index + 1 into a grid padded by one
        cell on each side, upper weight, and the ray parameter at every plane."""
        g = self.g
        n, n2 = (g.nx, g.ny) if fam == 0 else (g.ny, g.nx)
        h, h2 = (g.dx, g.dy) if fam == 0 else (g.dy, g.dx)
        t = ((torch.arange(n, device="cuda", dtype=F64) - (n - 1) / 2) * h - o[:, fam, None]) / d[:, fam, None]
        f = (o[:, 1 - fam, None] + t * d[:, 1 - fam, None]) / h2 + (n2 - 1) / 2
        return self._split(f, n2) + (t,)

    @staticmethod
    def _split(f, n):
        lo = torch.floor(f)
        w = f - lo
        lo = lo.long()
        w = torch.where((lo < -1) | (lo >= n), torch.full_like(w, float("nan")), w)
        out = torch.isnan(w)
        lo = lo.clamp(-1, n - 1) + 1
        return lo, torch.where(out, 0.0, 1.0 - w), torch.where(out, 0.0, w)

    def _sets(self):
        """(ray indices, driving axis, per-ray weight, in-plane split, row split) of every chunk."""
        g = self.g
        for sl, views in self._chunks():
            o, d = _rays(g, views)
            if g.kind != CONE3D:
                o, d = o.reshape(-1, 2), d.reshape(-1, 2)
                for fam in (0, 1):
                    x_drives = d[:, 0].abs() >= d[:, 1].abs()
                    k = torch.nonzero(x_drives if fam == 0 else ~x_drives).flatten()
                    if k.numel():
                        a, w0, w1, _ = self._plane(o[k], d[k], fam)
                        yield k + sl.start, fam, (g.dx if fam == 0 else g.dy) / d[k, fam].abs(), (a, w0, w1), None
                continue
            # all rows of a detector column share the in-plane path (the rows run along z)
            ray = torch.arange(sl.start, sl.stop, device="cuda").reshape(len(views), g.n_v, g.n_u)
            assert bool((d[..., 2].abs() <= torch.maximum(d[..., 0].abs(), d[..., 1].abs())).all())
            for q in range(len(views)):
                for fam in (0, 1):
                    x_drives = d[q, 0, :, 0].abs() >= d[q, 0, :, 1].abs()
                    k = torch.nonzero(x_drives if fam == 0 else ~x_drives).flatten()
                    if not k.numel():
                        continue
                    dk = d[q][:, k]                                         # [n_v][k][3]
                    a, w0, w1, _ = self._plane(o[q, 0, k, :2], dk[0, :, :2], fam)
                    n, h = (g.nx, g.dx) if fam == 0 else (g.ny, g.dy)
                    pl = (torch.arange(n, device="cuda", dtype=F64) - (n - 1) / 2) * h
                    t = (pl[None, :, None] - o[q, 0, k, fam][:, None, None]) / dk[:, :, fam].T[:, None, :]
                    z = self._split(t * dk[:, :, 2].T[:, None, :] / g.dz + (g.nz - 1) / 2, g.nz)  # [k][plane][n_v]
                    yield ray[q][:, k].T, fam, h / dk[:, :, fam].abs().T, (a, w0, w1), z

    def project(self, x):
        g = self.g
        x = x.reshape((-1,) + tuple(g.image_shape)).to(F64)
        out = torch.zeros((x.shape[0], g.n_views * g.n_u * g.n_v), dtype=F64, device="cuda")
        pads = {}
        for fam in (0, 1):
            if g.kind != CONE3D:               # [m][driving][interpolated + 2]
                v = x.transpose(1, 2) if fam == 0 else x
                pads[fam] = torch.nn.functional.pad(v, (1, 1)).contiguous()
            else:                              # [m][driving][interpolated + 2][z + 2]
                v = x.permute(0, 3, 2, 1) if fam == 0 else x.permute(0, 2, 3, 1)
                pads[fam] = torch.nn.functional.pad(v, (1, 1, 1, 1)).contiguous()
        for k, fam, w, (a, w0, w1), z in self._sets():
            i = torch.arange(a.shape[1], device="cuda")[None, :].expand_as(a)
            for m in range(x.shape[0]):
                v = pads[fam][m]
                if z is None:
                    out[m, k] = w * (w0 * v[i, a] + w1 * v[i, a + 1]).sum(1)
                else:
                    c = w0[..., None] * v[i, a] + w1[..., None] * v[i, a + 1]     # [k][plane][z + 2]
                    out[m, k] = w * (z[1] * c.gather(2, z[0]) + z[2] * c.gather(2, z[0] + 1)).sum(1)
        return out

    def backproject(self, s):
        g = self.g
        s = s.reshape(-1, g.n_views * g.n_u * g.n_v).to(F64)
        out = torch.zeros((s.shape[0],) + tuple(g.image_shape), dtype=F64, device="cuda")
        dims = {0: (g.nx, g.ny + 2), 1: (g.ny, g.nx + 2)}
        tail = (g.nz + 2,) if g.kind == CONE3D else ()
        acc = {f: [torch.zeros(dims[f] + tail, dtype=F64, device="cuda") for _ in range(s.shape[0])] for f in dims}
        for k, fam, w, (a, w0, w1), z in self._sets():
            at = (torch.arange(a.shape[1], device="cuda")[None, :] * dims[fam][1] + a).reshape(-1)
            for m in range(s.shape[0]):
                v = s[m, k] * w
                if z is None:
                    t = v[:, None].expand_as(a)
                    buf = acc[fam][m].view(-1)
                    buf.index_add_(0, at, (w0 * t).reshape(-1))
                    buf.index_add_(0, at + 1, (w1 * t).reshape(-1))
                    continue
                t = torch.zeros(a.shape + (g.nz + 2,), dtype=F64, device="cuda")
                t.scatter_add_(2, z[0], z[1] * v[:, None, :])
                t.scatter_add_(2, z[0] + 1, z[2] * v[:, None, :])
                buf = acc[fam][m].view(-1, g.nz + 2)
                buf.index_add_(0, at, (w0[..., None] * t).reshape(-1, g.nz + 2))
                buf.index_add_(0, at + 1, (w1[..., None] * t).reshape(-1, g.nz + 2))
        for m in range(s.shape[0]):
            for fam in (0, 1):
                v = acc[fam][m]
                if g.kind != CONE3D:
                    v = v[:, 1:-1]
                    out[m] += v.T if fam == 0 else v
                else:
                    v = v[:, 1:-1, 1:-1]
                    out[m] += v.permute(2, 1, 0) if fam == 0 else v.permute(2, 0, 1)
        return out


class _Identity:
    def project(self, x):
        return x

    def backproject(self, s):
        return s


class _Model:
    """Counts, residual weights and SPS numerators in 64 bits, rays in chunks."""

    def __init__(self, case, y):
        self.Q, self.S = _spectrum(case)
        self.y = y.to(F64)
        self.row, self.taps, self.a = case["bins"], TAPS.get(case.get("blur", 0)), float(case.get("noise", 0.0))

    def blur(self, v, flip=False):
        if self.taps is None:
            return v
        b = self.taps[::-1] if flip else self.taps
        r = len(b) // 2
        p = torch.nn.functional.pad(v.reshape(-1, self.row), (r, r))
        return sum(b[k] * p[:, k:k + self.row] for k in range(2 * r + 1)).reshape(v.shape)

    def weigh(self, v, y):
        w = 1.0 / y.clamp(min=1.0)
        if not self.a:
            return w * v
        sv, a = (w.sqrt() * v).reshape(-1, self.row), self.a
        out = sv.clone()
        out[:, 1:-1] *= 1 + a * a
        out[:, 1:] -= a * sv[:, :-1]
        out[:, :-1] -= a * sv[:, 1:]
        return w.sqrt() * (out / (1 - a * a)).reshape(v.shape)

    def counts(self, l, q=None):
        """ybar and, along q, its first two derivatives ([c][rays])."""
        out = [torch.zeros_like(self.y) for _ in range(1 if q is None else 3)]
        for e in range(self.Q.shape[0]):
            t = torch.exp(-sum(float(self.Q[e, m]) * l[m] for m in range(l.shape[0])))
            dz = None if q is None else sum(float(self.Q[e, m]) * q[m] for m in range(l.shape[0]))
            for c in range(self.S.shape[0]):
                if self.S[c, e]:
                    out[0][c] += float(self.S[c, e]) * t
                    if q is not None:
                        out[1][c] -= float(self.S[c, e]) * t * dz
                        out[2][c] += float(self.S[c, e]) * t * dz * dz
        return [torch.stack([self.blur(v) for v in o]) for o in out]

    def numerators(self, l, gamma=None):
        """Gradient numerator and (with gamma) curvature numerator, [m][rays]."""
        r = self.counts(l)[0] - self.y
        u = [self.blur(self.weigh(r[c], self.y[c]), True) for c in range(r.shape[0])]
        g, kap = torch.zeros_like(l), torch.zeros_like(l)
        for e in range(self.Q.shape[0]):
            if not self.S[:, e].any():
                continue
            t = torch.exp(-sum(float(self.Q[e, m]) * l[m] for m in range(l.shape[0])))
            v = sum(float(self.S[c, e]) * u[c] for c in range(len(u)))
            for m in range(l.shape[0]):
                g[m] -= float(self.Q[e, m]) * t * v
            if gamma is not None:
                eta = sum(float(self.S[c, e] * self.S[c].sum()) / self.y[c].clamp(min=1.0) for c in range(len(u)))
                hi = t.clamp(min=1.0)
                cE = ((2 * eta * hi + v - eta * t) * hi).clamp(min=0.0)
                gE = sum(float(self.Q[e, m]) * gamma[m] for m in range(l.shape[0]))
                for m in range(l.shape[0]):
                    kap[m] += float(self.Q[e, m]) * gE * cE
        return g, kap


def _haar(v, absolute=False, inverse=False):
    """Orthonormal 2-D Haar pyramid (Mallat layout) of [n][n]."""
    v = v.clone()
    n = v.shape[0]
    sg = 1.0 if absolute else -1.0
    h = 2 if inverse else n
    while 2 <= h <= n:
        k, b = h // 2, v[:h, :h].clone()
        if inverse:
            p, q, r, s = b[:k, :k], b[:k, k:], b[k:, :k], b[k:, k:]
        else:
            p, q, r, s = b[0::2, 0::2], b[0::2, 1::2], b[1::2, 0::2], b[1::2, 1::2]
        o = (0.5 * (p + q + r + s), 0.5 * (p + sg * q + r + sg * s), 0.5 * (p + q + sg * r + sg * s),
             0.5 * (p + sg * q + sg * r + s))
        if inverse:
            v[0:h:2, 0:h:2], v[0:h:2, 1:h:2], v[1:h:2, 0:h:2], v[1:h:2, 1:h:2] = o
            h *= 2
        else:
            v[:k, :k], v[:k, k:h], v[k:h, :k], v[k:h, k:h] = o
            h //= 2
    return v


class _Precond:
    """M, its transpose and the absolute bounds in 64 bits."""

    def __init__(self, case, s):
        self.kind = case["precond"]
        if "blocks" in s:
            self.B = s["blocks"].to(F64)
        if self.kind == "haar":
            lam = s["lam"].to(F64).abs()
            self.scale, self.m0 = lam.clamp(min=1e-6 * float(lam.max())) ** -0.5, s["m0"].to(F64)
        elif self.kind == "block_fourier":
            self.shape = (case["ny"], case["nx"])
            w, V = torch.linalg.eigh(s["lam"].to(F64).permute(2, 0, 1).cpu())
            w = w.clamp(min=1e-6 * float(w.max())) ** -0.5
            self.L = ((V * w[:, None, :]) @ V.transpose(1, 2)).permute(1, 2, 0).cuda()
            self.L = self.L.reshape(self.L.shape[:2] + self.shape)
            self.Labs = torch.fft.fft2(torch.fft.ifft2(self.L).real.abs()).real

    def apply(self, op, v):
        ab, tr = op.startswith("abs"), op.endswith("MT")
        if self.kind == "none":
            return v
        if self.kind == "haar":
            # |U^T D U| is bounded by |U|^T D |U|
            w = _haar(v[0] * self.m0, ab) * self.scale
            return (_haar(w, ab, True) * self.m0)[None]
        B = self.B.abs() if ab else self.B
        flat = v.reshape(v.shape[0], -1)
        if self.kind == "block":
            return torch.einsum("kmn,kn->mn" if tr else "mkn,kn->mn", B, flat).reshape(v.shape)
        if tr:
            flat = torch.einsum("mkn,kn->mn", B, flat)
        Z = torch.einsum("abyx,byx->ayx", (self.Labs if ab else self.L).to(torch.complex128),
                         torch.fft.fft2(flat.reshape((-1,) + self.shape)))
        flat = torch.fft.ifft2(Z).real.reshape(v.shape[0], -1)
        if not tr:
            flat = torch.einsum("kmn,kn->mn", B, flat)
        return flat.reshape(v.shape)


def _penalty(beta, x, absolute=False):
    """R x = (beta (x) Gamma) x (|R| x), non-periodic nearest neighbours."""
    if beta is None:
        return torch.zeros_like(x)
    out = torch.zeros_like(x)
    for d in range(1, x.ndim):
        n = x.shape[d]
        if n < 2:
            continue
        lo, hi = x.narrow(d, 0, n - 1), x.narrow(d, 1, n - 1)
        sg = 1.0 if absolute else -1.0
        out.narrow(d, 0, n - 1).add_(lo + sg * hi)
        out.narrow(d, 1, n - 1).add_(hi + sg * lo)
    b = torch.as_tensor(np.abs(beta) if absolute else beta, dtype=F64, device="cuda")
    return torch.einsum("mk,k...->m...", b, out)


def _exact_step(case, s):
    """``iters`` iterations from x = 0 with the safeguarded Newton line search (3 evaluations, 8 halvings)."""
    geom = _geometry(case)
    A = _Identity() if geom is None else _Joseph(geom)
    M, mod, beta = _Precond(case, s), _Model(case, s["y"]), _beta(case)
    n = (case["mats"], _n_rays(case)) if geom is None else (case["mats"],) + tuple(geom.image_shape)
    x = torch.zeros(n, dtype=F64, device="cuda")
    l = torch.zeros((case["mats"], _n_rays(case)), dtype=F64, device="cuda")
    bound = M.apply("absM", torch.ones_like(x))
    gamma = A.project(bound)
    dR = M.apply("absMT", _penalty(beta, bound, True))
    w, a_prev, zmin = 1.0 / mod.y.clamp(min=1.0), 1.0, -20.0
    Qd = torch.as_tensor(mod.Q, dtype=F64, device="cuda")
    for _ in range(case["iters"]):
        phi0 = 0.5 * float((w * (mod.counts(l)[0] - mod.y) ** 2).sum()) + 0.5 * float((x * _penalty(beta, x)).sum())
        g, kap = mod.numerators(l, gamma)
        gp = M.apply("MT", A.backproject(g).reshape(n) + _penalty(beta, x))
        dp = M.apply("absMT", A.backproject(kap).reshape(n)) + dR
        p = M.apply("M", torch.where(dp > 0, -gp / torch.where(dp > 0, dp, 1.0), 0.0))
        q = A.project(p)
        Rx, Rp = _penalty(beta, x), _penalty(beta, p)
        R0, pRx, pRp = 0.5 * float((x * Rx).sum()), float((p * Rx).sum()), float((p * Rp).sum())

        def phi(a):
            la = l + a * q
            if min(float((Qd[e] @ la).min()) for e in range(Qd.shape[0])) < zmin:
                return math.inf, math.nan, math.nan
            yb, d1, d2 = mod.counts(la, q)
            r = yb - mod.y
            return (0.5 * float((w * r * r).sum()) + R0 + a * pRx + 0.5 * a * a * pRp,
                    float((w * r * d1).sum()) + pRx + a * pRp,
                    float((w * (d1 * d1 + r * d2)).sum()) + pRp)
        a = a_prev
        for k in range(3):
            f, f1, f2 = phi(a)
            if k < 2:
                if not all(map(math.isfinite, (f, f1, f2))):
                    a = a / 8
                elif f2 > 0:
                    a = min(max(a - f1 / f2, a / 8), a * 8)
        best, k = a, 0
        while not (math.isfinite(f) and f <= phi0) and k < 8:
            a, k = a / 2, k + 1
            f = phi(a)[0]
        if not (math.isfinite(f) and f <= phi0):
            a = 0.0
        a_prev = a if a > 0 else best / 2.0 ** 9
        x, l = x + a * p, l + a * q
    return x


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "apply":
        return _Precond(case, s).apply(case["op"], s["v"].to(F64))
    geom = _geometry(case)
    if kind == "project":
        return _Joseph(geom).project(s["x"])
    if kind == "backproject":
        return _Joseph(geom).backproject(s["s"])
    if kind == "gradient":
        A = _Identity() if geom is None else _Joseph(geom)
        l = A.project(s["x"].to(F64))
        g = _Model(case, s["y"]).numerators(l)[0]
        return A.backproject(g).reshape(s["x"].shape)
    return _exact_step(case, s)
