"""Performance cases of the RBF terrain library: what a mapping or odometry program has it do.

Every case goes through ``paper_2509_26222_gb300.native`` as a user's program does.  ``prepare``
makes the inputs from the seed (scans, queries, poses, maps) and the context a program keeps,
``run`` is one pass, ``work`` what a pass cannot do without, and ``exact`` the same results in
64 bits, written here in plain torch.

Kinds of cases
  eval     h and grad h at scattered queries of a map with known weights
  raster   h and grad h of a Gaussian map on a regular raster
  soft     soft-constraint cost of a body-frame scan and its gradients (pose, weights, centers)
  align    one Levenberg-Marquardt step on the pose of a scan
  map      a new map: install a lattice of centers, one update with a cloud, evaluate it
  scans    a stretch of the staircase sequence: the map starts over, then every scan updates it
           and is evaluated on it (centers enter, stay, leave and come back)
  survey   the paper's Gaussian parameters: choose the centers under a scan, update, evaluate
  patches  a batch of independent patches of uneven size, updated and evaluated in one call
"""
from __future__ import annotations

import math

import torch

F64, F32 = torch.float64, torch.float32


def listed():
    return [
        # height queries of a planner on a small map: the smallest call, bound by its launch
        dict(name="eval_scan", kind="eval", side=16, spacing=0.25, rho=0.6, queries=10_000),
        # dense queries (a rendered or exported terrain): the largest plain evaluation
        dict(name="eval_dense", kind="eval", side=64, spacing=0.2, rho=0.6, queries=1 << 24),
        # an elevation raster of the paper's Gaussian terrain at 5 mm
        dict(name="raster_5mm", kind="raster", lattice=366, nqx=5120, nqy=5120, dq=0.005, grad=True),
        # the soft constraint as a differentiable term: cost, then gradients to pose, weights, centers
        dict(name="soft_grad", kind="soft", points=65_536, loss="huber", outliers=0.05),
        # scan matching: one LM step on the pose with the ground returns of a scan
        dict(name="align_pose", kind="align", points=8_000, loss="huber", outliers=0.05),
        # a small map in the default (float64) update precision, from the centers to the heights
        dict(name="map_small", kind="map", side=16, spacing=0.25, rho=0.6, bx=16, by=16, points=2_000,
             queries=10_000, mixed=False),
        # a large map: 65,536 centers, a block of 8,192 touched at once, a million queries
        dict(name="map_block", kind="map", side=256, spacing=0.1, rho=0.3, bx=128, by=64, points=32_768,
             queries=1 << 20, mixed=True),
        # odometry on level ground, mixed precision: the ordinary frame
        dict(name="scans_ground", kind="scans", first=3, frames=6, points=8_000, mixed=True, exact=False),
        # odometry on the upper stairs: nearly the whole map is active, hundreds of centers leave and return
        dict(name="scans_stairs", kind="scans", first=150, frames=4, points=8_000, mixed=True, exact=False),
        # the same ground frames in float64, for programs that ask for the plain precision
        dict(name="scans_fp64", kind="scans", first=3, frames=3, points=8_000, mixed=False, exact=False),
        # the paper's own terrain parameters: adaptive centers, Gaussian rows (about 118 neighbours a point)
        dict(name="survey_gauss", kind="survey", mesh=64, points=8_000, queries=65_536, mixed=True),
        # many terrains at once: patches of 64 to 4,096 centers with 500 to 50,000 points each
        dict(name="patches_256", kind="patches", patches=256, m_lo=64, m_hi=4096, n_lo=500, n_hi=50_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "raster", "soft", "align", "map", "scans", "scans", "survey", "patches"])
    if kind == "eval":
        h, rho = rng.choice([(0.25, 0.6), (0.2, 0.6), (0.1, 0.3)])
        return dict(kind=kind, side=_log(rng, 16, 256), spacing=h, rho=rho, queries=_log(rng, 1_000, 1 << 24))
    if kind == "raster":
        return dict(kind=kind, lattice=rng.randint(40, 366), nqx=_log(rng, 100, 5120), nqy=_log(rng, 100, 5120),
                    dq=round(rng.uniform(0.004, 0.03), 5), grad=rng.random() < 0.7)
    if kind in ("soft", "align"):
        return dict(kind=kind, points=_log(rng, 1_000, 131_072), loss=rng.choice(["huber", "huber", "l2"]),
                    outliers=round(rng.uniform(0.0, 0.1), 3))
    if kind == "map":
        h, rho = rng.choice([(0.25, 0.6), (0.2, 0.6), (0.1, 0.3)])
        side = _log(rng, 16, 256)
        return dict(kind=kind, side=side, spacing=h, rho=rho, bx=rng.randint(10, min(side, 128)),
                    by=rng.randint(10, min(side, 64)), points=_log(rng, 500, 32_768),
                    queries=_log(rng, 1_000, 1 << 20), mixed=rng.random() < 0.6)
    if kind == "scans":
        mixed = rng.random() < 0.75
        return dict(kind=kind, first=rng.randint(0, 190), frames=rng.randint(2, 6 if mixed else 2),
                    points=_log(rng, 2_000, 16_000), mixed=mixed, exact=mixed and rng.random() < 0.2)
    if kind == "survey":
        return dict(kind=kind, mesh=rng.randint(24, 64), points=_log(rng, 1_000, 16_000),
                    queries=_log(rng, 1_000, 262_144), mixed=rng.random() < 0.7)
    return dict(kind=kind, patches=_log(rng, 8, 256), m_lo=64, m_hi=_log(rng, 512, 4096), n_lo=500,
                n_hi=_log(rng, 4_000, 50_000))


# ----------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------
# The ridge weight: at the default of 1e-3 the weights that hardly any return constrains come out of the mixed
# precision to 1e-10 .. 1e-9 only, at 1e-2 to 1e-11 or better, so that two correct builds agree to float64's bounds.
LAM, RANGE_SIGMA, SIGMA, CUT, SURVEY_NOISE, HUBER = 1e-2, 0.03, 0.04, 4.0, 0.1, 0.05
SEQ_SIDE, SEQ_H, SEQ_X0, SEQ_RHO = 64, 0.2, -6.4, 0.6     # the staircase map
MESH_H, MESH_R = 0.07, 0.1                                  # the paper's candidate mesh


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _rng(seed, *more):
    g = torch.Generator(device=_dev())
    k = seed & 0x3FFFFFFF
    for m in more:
        k = (k * 1_000_003 + 7919 * int(m) + 17) & 0x3FFFFFFFFFFF
    g.manual_seed(k)
    return g


def _u(g, n, lo, hi):
    return torch.rand(n, generator=g, device=_dev(), dtype=F64) * (hi - lo) + lo


def _normal(g, n, sd):
    return torch.randn(n, generator=g, device=_dev(), dtype=F64) * sd


def _lattice(nx, ny, x0, y0, h):
    """Centers (x0 + (i + 0.5) h, y0 + (j + 0.5) h), row-major, id = j nx + i."""
    cx = x0 + (torch.arange(nx, device=_dev(), dtype=F64) + 0.5) * h
    cy = y0 + (torch.arange(ny, device=_dev(), dtype=F64) + 0.5) * h
    return torch.stack([cx.repeat(ny), cy.repeat_interleave(nx)], 1).contiguous()


def _rolling(x, y):
    """A sinusoidal surface with a 0.15 m step."""
    return 0.1 * torch.sin(2.0 * x) * torch.cos(1.5 * y) + 0.15 * (x >= 2.0)


def _stairs(x, y):
    """Flat, then ten stairs (tread 0.30 m, rise 0.15 m), with bumps of 2 cm."""
    steps = 0.15 * torch.clamp(torch.floor(x / 0.3) + 1.0, 0.0, 10.0)
    return steps + 0.02 * torch.sin(2.0 * math.pi * x / 0.5) * torch.cos(2.0 * math.pi * y / 0.7)


def _scan(g, n, x):
    """n ground returns (world frame, float32) of a LiDAR 0.6 m above the staircase at (x, 0)."""
    z = float(_stairs(torch.tensor([x], dtype=F64), torch.zeros(1, dtype=F64))) + 0.6
    az, el = _u(g, n, 0.0, 2.0 * math.pi), torch.deg2rad(_u(g, n, -52.0, -7.0))
    d = torch.stack([torch.cos(el) * torch.cos(az), torch.cos(el) * torch.sin(az), torch.sin(el)], 1)
    o = torch.tensor([x, 0.0, z], device=_dev(), dtype=F64)

    def below(t, d):
        p = o + t[..., None] * d
        return p[..., 2] <= _stairs(p[..., 0], p[..., 1])

    ts = torch.arange(1, 1001, device=_dev(), dtype=F64) * 0.025
    first = torch.cat([torch.argmax(below(ts[None, :], e[:, None, :]).to(torch.uint8), 1) for e in d.split(4096)])
    hi = ts[first]
    lo = hi - 0.025
    for _ in range(24):
        mid = 0.5 * (lo + hi)
        b = below(mid, d)
        hi, lo = torch.where(b, mid, hi), torch.where(b, lo, mid)
    t = hi + _normal(g, n, RANGE_SIGMA)
    return (o + t[:, None] * d).to(F32).contiguous()


def _sensor_x(k):
    return -3.0 + 0.04 * k


def _quasi(c, f, h, vol):
    """Weights of a smooth terrain: the surface's values times cell area over the kernel's volume."""
    return f(c[:, 0], c[:, 1]) * (h * h / vol)


def _wendland_volume(rho):
    return math.pi * rho * rho / 7.0


def _pose(g):
    yaw, pitch, roll = (float(v) for v in (_u(g, 1, 0.0, 2 * math.pi), _u(g, 1, -0.0873, 0.0873),
                                           _u(g, 1, -0.0873, 0.0873)))
    cy, sy, cp, sp, cr, sr = (f(a) for a in (yaw, pitch, roll) for f in (math.cos, math.sin))
    Rz = torch.tensor([[cy, -sy, 0], [sy, cy, 0], [0, 0, 1]], dtype=F64)
    Ry = torch.tensor([[cp, 0, sp], [0, 1, 0], [-sp, 0, cp]], dtype=F64)
    Rx = torch.tensor([[1, 0, 0], [0, cr, -sr], [0, sr, cr]], dtype=F64)
    return Rz @ Ry @ Rx, (_u(g, 3, -0.5, 0.5)).cpu()


def _inputs(case, seed):
    """The tensors a pass takes, by name, from the seed alone."""
    k, g = case["kind"], _rng(seed)
    if k == "eval":
        s, h = case["side"], case["spacing"]
        c = _lattice(s, s, 0.0, 0.0, h)
        w = _quasi(c, _rolling, h, _wendland_volume(case["rho"])) + _normal(g, s * s, 0.005)
        q = torch.stack([_u(g, case["queries"], 0.0, s * h), _u(g, case["queries"], 0.0, s * h)], 1).to(F32)
        return dict(c=c, w=w, q=q.contiguous())
    if k == "raster":
        n = case["lattice"]
        c = _lattice(n, n, 0.0, 0.0, MESH_H)
        w = _quasi(c, lambda x, y: _stairs(x - 6.0, y), MESH_H, 2.0 * math.pi * SIGMA * SIGMA)
        x0, y0 = (float(v) for v in _u(g, 2, 0.0, 0.05))
        return dict(c=c, w=w + _normal(g, n * n, 0.002), x0=x0, y0=y0)
    if k in ("soft", "align"):
        n = case["points"]
        c = _lattice(SEQ_SIDE, SEQ_SIDE, SEQ_X0, SEQ_X0, SEQ_H)
        w = _quasi(c, _rolling, SEQ_H, _wendland_volume(SEQ_RHO)) + _normal(g, len(c), 0.002)
        R, t = _pose(g)
        x, y = _u(g, n, -5.5, 5.5), _u(g, n, -5.5, 5.5)
        z = _rolling(x, y) + _normal(g, n, 0.03)
        out = torch.rand(n, generator=g, device=_dev()) < case["outliers"]
        z = z + out * torch.where(torch.rand(n, generator=g, device=_dev()) < 0.5, 0.3, -0.3)
        body = (torch.stack([x, y, z], 1) - t.to(_dev())) @ R.to(_dev())
        if k == "align":  # the pose to be corrected is a little off
            t = t + _u(g, 3, -0.02, 0.02).cpu()
        return dict(c=c, w=w, R=R, t=t, body=body.to(F32).contiguous())
    if k == "map":
        s, h, rho, bx, by = (case[x] for x in ("side", "spacing", "rho", "bx", "by"))
        c = _lattice(s, s, 0.0, 0.0, h)
        i0, j0 = (s - bx) // 2, (s - by) // 2
        in_x, in_y = (rho - 0.5 * h if bx < s else 0.0), (rho - 0.5 * h if by < s else 0.0)
        x = _u(g, case["points"], i0 * h + in_x, (i0 + bx) * h - in_x)
        y = _u(g, case["points"], j0 * h + in_y, (j0 + by) * h - in_y)
        z = _rolling(x, y) + _normal(g, case["points"], 0.02)
        q = torch.stack([_u(g, case["queries"], 0.0, s * h), _u(g, case["queries"], 0.0, s * h)], 1).to(F32)
        return dict(c=c, pts=torch.stack([x, y, z], 1).to(F32).contiguous(), q=q.contiguous())
    if k == "scans":
        c = _lattice(SEQ_SIDE, SEQ_SIDE, SEQ_X0, SEQ_X0, SEQ_H)
        scans = [_scan(_rng(seed, case["first"] + f), case["points"], _sensor_x(case["first"] + f))
                 for f in range(case["frames"])]
        return dict(c=c, scans=scans, q=[p[:, :2].contiguous() for p in scans])
    if k == "survey":
        half = 0.5 * case["mesh"] * MESH_H
        x = float(_u(g, 1, -1.0, 1.0))
        q = torch.stack([_u(g, case["queries"], x - half, x + half), _u(g, case["queries"], -half, half)], 1).to(F32)
        return dict(pts=_scan(g, case["points"], x), q=q.contiguous(), x0=x - half, y0=-half)
    patches = []
    sizes = _rng(12345, case["patches"], case["m_hi"], case["n_hi"])  # a batch shape stays, its points change
    um, un = (_u(sizes, case["patches"], 0.0, 1.0).tolist() for _ in range(2))
    par = _u(g, 6 * case["patches"], 0.0, 1.0).tolist()
    h = 0.2
    for b in range(case["patches"]):
        M = int(round(case["m_lo"] * (case["m_hi"] / case["m_lo"]) ** um[b]))
        n = int(round(case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** un[b]))
        gx = int(math.ceil(math.sqrt(M)))
        a, fx, fy, sx, sh, _ = par[6 * b:6 * b + 6]
        x, y = _u(g, n, 0.0, gx * h), _u(g, n, 0.0, max(M // gx, 1) * h)
        z = (0.02 + 0.18 * a) * torch.sin((0.5 + 2.5 * fx) * x) * torch.cos((0.5 + 2.5 * fy) * y)
        z = z + (0.4 * sh - 0.2) * (x >= (0.2 + 0.6 * sx) * gx * h) + _normal(g, n, 0.02)
        pts = torch.stack([x, y, z], 1).to(F32).contiguous()
        patches.append(dict(M=M, nx=gx, h=h, pts=pts, q=pts[:, :2].contiguous()))
    return dict(patches=patches)


# ----------------------------------------------------------------------------------------------
# a pass
# ----------------------------------------------------------------------------------------------
def prepare(case, seed):
    from paper_2509_26222_gb300 import native as N

    k, s = case["kind"], _inputs(case, seed)
    s["case"] = case
    prec = N.UPDATE_MIXED if case.get("mixed") else N.UPDATE_FP64
    if k in ("eval", "raster"):
        T = (N.Terrain(rho=case["rho"], lam=LAM) if k == "eval"
             else N.Terrain(kernel=N.KERNEL_GAUSSIAN, sigma=SIGMA, cutoff_mult=CUT, lam=LAM))
    elif k in ("soft", "align"):
        T = N.Terrain(rho=SEQ_RHO, lam=LAM, huber_delta=HUBER,
                      loss=N.LOSS_HUBER if case["loss"] == "huber" else N.LOSS_L2)
    elif k == "map":
        T = N.Terrain(rho=case["rho"], lam=LAM, update_precision=prec)
    elif k == "scans":
        T = N.Terrain(rho=SEQ_RHO, lam=LAM, update_precision=prec, exact=case["exact"])
    elif k == "survey":
        T = N.Terrain(kernel=N.KERNEL_GAUSSIAN, sigma=SIGMA, cutoff_mult=CUT, lam=LAM, update_precision=prec,
                      mesh=(s["x0"], s["y0"], MESH_H, case["mesh"], case["mesh"]), r_kd=MESH_R, min_count=1)
    else:
        T = N.Terrain(rho=SEQ_RHO, lam=LAM, update_precision=N.UPDATE_MIXED)
        P = s["patches"]
        s["arr"] = (N.RbfPatch * len(P))()
        tot_m, tot_q = sum(p["M"] for p in P), sum(len(p["q"]) for p in P)
        s["w"] = torch.empty(tot_m, dtype=F64, device="cuda")
        s["h"] = torch.empty(tot_q, dtype=F32, device="cuda")
        s["g"] = torch.empty(tot_q, 2, dtype=F32, device="cuda")
        m0 = q0 = 0
        for d, p in zip(s["arr"], P):
            d.x0, d.y0, d.spacing, d.nx, d.M = 0.0, 0.0, p["h"], p["nx"], p["M"]
            d.n, d.pts, d.Q, d.q = len(p["pts"]), p["pts"].data_ptr(), len(p["q"]), p["q"].data_ptr()
            d.w, d.h, d.grad = s["w"][m0:].data_ptr(), s["h"][q0:].data_ptr(), s["g"][q0:].data_ptr()
            m0, q0 = m0 + p["M"], q0 + len(p["q"])
    s["T"] = T
    if k in ("eval", "raster", "soft", "align"):
        T.set_centers(s["c"])
        T.set_weights(s["w"])
    return s


def run(s):
    case, T = s["case"], s["T"]
    k = case["kind"]
    if k == "eval":
        return T.eval(s["q"])
    if k == "raster":
        h, g = T.eval_grid(s["x0"], s["y0"], case["dq"], case["nqx"], case["nqy"], with_grad=case["grad"])
        return (h, g) if case["grad"] else (h,)
    if k == "soft":
        cost, g6, r = T.soft_cost(s["R"], s["t"], s["body"], with_resid=True)
        dw, dc, dpose = T.soft_cost_backward(s["R"], s["t"], s["body"])
        return cost, g6, r, dw, dc, dpose
    if k == "align":
        return T.lm_step(s["R"], s["t"], s["body"])
    if k == "map":
        T.set_centers(s["c"])
        T.update(s["pts"], noise=0.02)
        return (T.weights(), *T.eval(s["q"]))
    if k == "scans":
        T.set_centers(s["c"])
        out = []
        for p, q in zip(s["scans"], s["q"]):
            T.update(p, noise=RANGE_SIGMA)
            out.append(T.eval(q))
        return T.weights(), out
    if k == "survey":
        m, counts = T.build_centers(s["pts"], return_counts=True)
        T.update(s["pts"], noise=SURVEY_NOISE)
        kept = torch.zeros(case["mesh"] ** 2, dtype=F64, device="cuda")  # the weights back on the mesh
        kept.masked_scatter_(counts >= 1, T.weights())
        return (m, counts, kept, *T.eval(s["q"]))
    T.batch_update_eval_into(s["arr"], len(s["arr"]))
    return s["w"], s["h"], s["g"]


def work(case):
    k = case["kind"]
    if k == "eval":  # about 15 operations for each center within the support
        near = math.pi * (case["rho"] / case["spacing"]) ** 2
        m = case["side"] ** 2
        return dict(bytes=20.0 * case["queries"] + 24.0 * m, flops=15.0 * near * case["queries"])
    if k == "raster":  # five products per tile of 128 x 128 points with a window of the nodes it touches
        n, m = case["nqx"] * case["nqy"], case["lattice"] ** 2
        win = (127 * case["dq"] + 2 * CUT * SIGMA) / MESH_H
        return dict(bytes=(12.0 if case["grad"] else 4.0) * n + 24.0 * m,
                    flops=n * (2 if case["grad"] else 1) * 2.0 * win * (1.5 + win / 128))
    if k in ("soft", "align"):
        near = math.pi * (SEQ_RHO / SEQ_H) ** 2
        n, m = case["points"], SEQ_SIDE ** 2
        if k == "align":
            return dict(bytes=12.0 * n + 24.0 * m, flops=n * (15.0 * near + 100))
        return dict(bytes=16.0 * n + 36.0 * m, flops=n * (40.0 * near + 60))
    if k == "patches":
        s = _inputs(case, 0)["patches"]
        flops = bts = 0.0
        for p in s:
            n, m, bw = len(p["pts"]), p["M"], min(p["M"], 5 * (p["nx"] + 1))
            flops += n * 28.0 * 28 + m * float(bw) * bw + 8.0 * m * bw + n * 15.0 * 28
            bts += 12.0 * n + 8.0 * m + 20.0 * n
        return dict(bytes=bts, flops=flops)
    # updates: rows, products, factorization (within the band where no center has left), solves, evaluation
    s = _inputs(case, 0)
    if k == "map":
        a = case["bx"] * case["by"]
        bw = min(a, int(2 * case["rho"] / case["spacing"]) * min(case["bx"], case["by"]))
        near = math.pi * (case["rho"] / case["spacing"]) ** 2
        n, q, m = case["points"], case["queries"], case["side"] ** 2
        return dict(bytes=12.0 * n + 20.0 * q + 24.0 * m,
                    flops=n * near * near + a * float(bw) * bw + 4.0 * a * bw + 15.0 * near * q)
    if k == "survey":
        L, m = _survey_lattice(case, s)[:2]
        near = math.pi * (CUT * math.hypot(SIGMA, SURVEY_NOISE) / MESH_H) ** 2
        n, q = case["points"], case["queries"]
        return dict(bytes=12.0 * n + 20.0 * q + 24.0 * m + 4.0 * case["mesh"] ** 2,
                    flops=n * near * near / 2 + m ** 3 / 3.0 + 4.0 * m * m + 8.0 * 16 * q)
    flops = bts = 0.0
    L = _Lat(s["c"], SEQ_SIDE, SEQ_SIDE, SEQ_X0, SEQ_X0, SEQ_H, None)
    near = math.pi * (SEQ_RHO / SEQ_H) ** 2
    for f, p in enumerate(s["scans"]):
        a = len(s["c"]) if case["exact"] else int(L.rows(p, False, 0.0)[2].sum())
        bw = min(a, 5 * SEQ_SIDE) if f == 0 or case["exact"] else a
        flops += len(p) * near * near + (a * float(bw) * bw if bw < a / 2 else a ** 3 / 3.0) + 4.0 * a * bw
        flops += 15.0 * near * len(p)
        bts += 32.0 * len(p)
    return dict(bytes=bts + 24.0 * len(s["c"]), flops=flops)


# ----------------------------------------------------------------------------------------------
# the same in 64 bits
# ----------------------------------------------------------------------------------------------
def _phi(d2, rho):
    s = torch.sqrt(d2) / rho
    t = torch.clamp(1.0 - s, min=0.0)
    return t ** 4 * (4.0 * s + 1.0), -20.0 / (rho * rho) * t ** 3


class _Lat:
    """Windows of lattice nodes around points.  `ids`: node -> center id (-1: none), default row-major."""

    def __init__(self, c, nx, ny, x0, y0, h, ids, rho=SEQ_RHO, count=None):
        self.c, self.nx, self.ny, self.x0, self.y0, self.h, self.rho = c, nx, ny, x0, y0, h, rho
        self.ids = torch.arange(nx * ny, device=c.device) if ids is None else ids
        if count is not None and count < nx * ny:  # the last row may be partial
            self.ids = torch.where(self.ids < count, self.ids, -1)
        self.M = len(c)

    def window(self, xy, r):
        """For float32 points: (first node i, first node j, size of the window)."""
        w = 2 * int(math.ceil(r / self.h) + 1)
        i = torch.floor((xy[:, 0].double() - self.x0) / self.h - 0.5).long() - w // 2 + 1
        j = torch.floor((xy[:, 1].double() - self.y0) / self.h - 0.5).long() - w // 2 + 1
        return i, j, w

    def near(self, xy, r, i=None, j=None, w=None):
        """ids (n, w w; -1 outside), dx, dy in 64 bits, and the float32 rule d2 < r^2."""
        if i is None:
            i, j, w = self.window(xy, r)
        o = torch.arange(w, device=xy.device)
        ii = (i[:, None, None] + o[None, None, :]).expand(-1, w, -1).reshape(len(xy), -1)
        jj = (j[:, None, None] + o[None, :, None]).expand(-1, -1, w).reshape(len(xy), -1)
        ok = (ii >= 0) & (ii < self.nx) & (jj >= 0) & (jj < self.ny)
        ids = torch.where(ok, self.ids[(jj.clamp(0, self.ny - 1) * self.nx + ii.clamp(0, self.nx - 1))], -1)
        c = self.c[ids.clamp(min=0)]
        c32 = c.to(F32)
        ex, ey = xy[:, None, 0] - c32[..., 0], xy[:, None, 1] - c32[..., 1]
        r32 = torch.tensor(r, dtype=F32, device=xy.device)
        inside = ((ex * ex) + (ey * ey) < r32 * r32) & (ids >= 0)
        x = xy.double()
        return ids, x[:, None, 0] - c[..., 0], x[:, None, 1] - c[..., 1], inside

    def rows(self, pts, gauss, noise, radius=None):
        """Regression rows: per point the window's ids and values; and which centers are touched."""
        r = (CUT * math.sqrt(SIGMA * SIGMA + noise * noise) if gauss else self.rho) if radius is None else radius
        act = torch.zeros(self.M + 1, dtype=torch.bool, device=pts.device)
        ids, dx, dy, inside = self.near(pts[:, :2].contiguous(), r)
        d2 = dx * dx + dy * dy
        if gauss:
            s2 = SIGMA * SIGMA + noise * noise
            m = SIGMA * SIGMA / s2 * torch.exp(-d2 / (2 * s2))
        else:
            m = _phi(d2, self.rho)[0]
        m = torch.where(inside, m, 0.0)
        act[torch.where(inside, ids, self.M)] = True
        return ids, m, act[:self.M]

    def gram(self, pts, z, gauss, noise):
        """m m^T (M x M) and m z (M), by cells: the points of a cell share their window."""
        r = CUT * math.sqrt(SIGMA * SIGMA + noise * noise) if gauss else self.rho
        i, j, w = self.window(pts[:, :2], r)
        key = (j + 4096) * 16384 + (i + 4096)
        order = torch.argsort(key)
        uniq, cnt = torch.unique_consecutive(key[order], return_counts=True)
        G = torch.zeros((self.M + 1) * (self.M + 1), dtype=F64, device=pts.device)
        u = torch.zeros(self.M + 1, dtype=F64, device=pts.device)
        start = torch.cumsum(cnt, 0) - cnt
        ww = w * w
        by = torch.argsort(cnt)  # cells of like counts together
        at = 0
        while at < len(uniq):
            step = max(1, int(2e7 // (ww * max(ww, int(cnt[by[min(at + 8192, len(uniq)) - 1]])))))
            cells = by[at:at + min(step, 8192)]
            at += len(cells)
            cm = int(cnt[cells].max())
            k = torch.arange(cm, device=pts.device)
            have = k[None, :] < cnt[cells][:, None]
            pt = order[(start[cells][:, None] + torch.where(have, k[None, :], 0)).reshape(-1)]
            ids, dx, dy, inside = self.near(pts[pt, :2], r, i[pt], j[pt], w)
            d2 = dx * dx + dy * dy
            if gauss:
                s2 = SIGMA * SIGMA + noise * noise
                m = SIGMA * SIGMA / s2 * torch.exp(-d2 / (2 * s2))
            else:
                m = _phi(d2, self.rho)[0]
            m = torch.where(inside & have.reshape(-1, 1), m, 0.0).reshape(len(cells), cm, ww)
            ids = ids.reshape(len(cells), cm, ww)[:, 0, :]
            ids = torch.where(ids >= 0, ids, self.M)
            g = m.transpose(1, 2) @ m
            G.index_add_(0, (ids[:, :, None] * (self.M + 1) + ids[:, None, :]).reshape(-1), g.reshape(-1))
            u.index_add_(0, ids.reshape(-1), (m * z[pt].reshape(len(cells), cm, 1)).sum(1).reshape(-1))
        return G.reshape(self.M + 1, self.M + 1)[:self.M, :self.M], u[:self.M]

    def height(self, q, w, gauss, chunk=1 << 18):
        h = torch.empty(len(q), dtype=F64, device=q.device)
        g = torch.empty(len(q), 2, dtype=F64, device=q.device)
        r = CUT * SIGMA if gauss else self.rho
        for at in range(0, len(q), chunk):
            ids, dx, dy, inside = self.near(q[at:at + chunk], r)
            d2 = dx * dx + dy * dy
            if gauss:
                f = torch.exp(-d2 / (2 * SIGMA * SIGMA))
                k = -f / (SIGMA * SIGMA)
            else:
                f, k = _phi(d2, self.rho)
            wj = torch.where(inside, w[ids.clamp(min=0)], 0.0)
            h[at:at + chunk] = (wj * f).sum(1)
            g[at:at + chunk, 0] = (wj * k * dx).sum(1)
            g[at:at + chunk, 1] = (wj * k * dy).sum(1)
        return h, g


def _solve(H, b):
    return torch.cholesky_solve(b[:, None], torch.linalg.cholesky(H))[:, 0]


class _Recursion:
    """The update restricted to the touched centers, in information form; every center outside the
    block keeps the covariance of the block it last left (none with the centers of another)."""

    def __init__(self, lat, lam, every=False):
        self.lat, self.lam, self.every = lat, lam, every
        self.w = torch.zeros(lat.M, dtype=F64, device=lat.c.device)
        self.P = None       # covariance of the centers outside the block, built when one leaves
        self.A, self.H = torch.zeros(0, dtype=torch.long, device=lat.c.device), None

    def update(self, pts, gauss, noise):
        lat, M = self.lat, self.lat.M
        ids, m, act = lat.rows(pts, gauss, noise)
        if self.every:
            act[:] = True
        A = torch.nonzero(act)[:, 0]
        innov = pts[:, 2].double() - (m * self.w[ids.clamp(min=0)]).sum(1)
        G, u = lat.gram(pts, innov, gauss, noise)
        H = G[A][:, A].clone()
        new = torch.full((M,), -1, dtype=torch.long, device=A.device)
        new[A] = torch.arange(len(A), device=A.device)
        if self.H is None:
            H.diagonal().add_(self.lam)
        else:
            stay = new[self.A] >= 0
            S, D = torch.nonzero(stay)[:, 0], torch.nonzero(~stay)[:, 0]
            Hs = self.H[S][:, S]
            if len(D):
                Hds = self.H[D][:, S]
                Hs = Hs - Hds.T @ torch.cholesky_solve(Hds, torch.linalg.cholesky(self.H[D][:, D]))
            at = new[self.A[S]]
            H[at[:, None], at[None, :]] += Hs
            old = torch.zeros(M, dtype=torch.bool, device=A.device)
            old[self.A] = True
            E = A[~old[A]]
            if len(E):
                if self.P is None:
                    H[new[E], new[E]] += self.lam
                else:
                    inv = torch.cholesky_inverse(torch.linalg.cholesky(self.P[E][:, E]))
                    H[new[E][:, None], new[E][None, :]] += inv
            if len(D):
                if self.P is None:
                    self.P = torch.eye(M, dtype=F64, device=A.device) / self.lam
                ids_d = self.A[D]
                unit = torch.zeros(len(self.A), len(D), dtype=F64, device=A.device)
                unit[D, torch.arange(len(D), device=A.device)] = 1.0
                pd = torch.cholesky_solve(unit, torch.linalg.cholesky(self.H))[D]
                self.P[ids_d, :] = 0.0
                self.P[:, ids_d] = 0.0
                self.P[ids_d[:, None], ids_d[None, :]] = 0.5 * (pd + pd.T)
        self.w[A] += _solve(H, u[A])
        self.A, self.H = A, H


def _survey_lattice(case, s):
    """The accepted candidates of the mesh as centers: (lattice, M, counts)."""
    n, p = case["mesh"], s["pts"]
    c = _lattice(n, n, s["x0"], s["y0"], MESH_H)
    full = _Lat(c, n, n, s["x0"], s["y0"], MESH_H, None)
    counts = torch.zeros(n * n + 1, dtype=torch.int32, device=c.device)
    ids, _, _, inside = full.near(p[:, :2].contiguous(), MESH_R)
    sel = torch.where(inside, ids, n * n).reshape(-1)
    counts.index_add_(0, sel, torch.ones_like(sel, dtype=torch.int32))
    counts = counts[:n * n]
    keep = counts >= 1
    ids = torch.where(keep, torch.cumsum(keep.long(), 0) - 1, -1)
    return _Lat(c[keep].contiguous(), n, n, s["x0"], s["y0"], MESH_H, ids), int(keep.sum()), counts


def _soft_terms(case, s, w, c, R, t):
    """cost and residuals in 64 bits, differentiable in w, c, R and t."""
    L = _Lat(s["c"], SEQ_SIDE, SEQ_SIDE, SEQ_X0, SEQ_X0, SEQ_H, None)
    q = s["body"].double() @ R.T + t
    ids, _, _, inside = L.near(q[:, :2].detach().to(F32), SEQ_RHO * 1.01)  # zero beyond the support anyway
    cc = c[ids.clamp(min=0)]
    d = q[:, None, :2] - cc
    d2 = (d * d).sum(-1)
    f = _phi(torch.where(inside, d2, 4.0), SEQ_RHO)[0]
    r = q[:, 2] - (w[ids.clamp(min=0)] * f).sum(1)
    if case["loss"] == "l2":
        return (r * r).sum(), r, q
    a = r.abs()
    return torch.where(a <= HUBER, 0.5 * r * r, HUBER * (a - 0.5 * HUBER)).sum(), r, q


def _skew(v):
    z = torch.zeros_like(v[..., 0])
    return torch.stack([torch.stack([z, -v[..., 2], v[..., 1]], -1), torch.stack([v[..., 2], z, -v[..., 0]], -1),
                        torch.stack([-v[..., 1], v[..., 0], z], -1)], -2)


def _exact_soft(case, s):
    dev = s["c"].device
    w, c = s["w"].clone().requires_grad_(), s["c"].clone().requires_grad_()
    R0, t0 = s["R"].to(dev), s["t"].to(dev)
    dt = torch.zeros(3, dtype=F64, device=dev, requires_grad=True)
    th = torch.zeros(3, dtype=F64, device=dev, requires_grad=True)
    cost, r, q = _soft_terms(case, s, w, c, R0 @ (torch.eye(3, dtype=F64, device=dev) + _skew(th)), t0 + dt)
    if case["kind"] == "soft":
        gw, gc, gth, gt = torch.autograd.grad(cost, (w, c, th, dt))
        g6 = torch.cat([gth, gt])
        return cost.detach(), g6, r.detach(), gw, gc, g6
    # LM: J rows = d r / d [theta, t], A = sum omega J J^T, (A + mu diag A) delta = -g
    L = _Lat(s["c"], SEQ_SIDE, SEQ_SIDE, SEQ_X0, SEQ_X0, SEQ_H, None)
    q = q.detach()
    r = r.detach()
    ids, _, _, inside = L.near(q[:, :2].to(F32), SEQ_RHO * 1.01)
    d = q[:, None, :2] - s["c"][ids.clamp(min=0)]
    k = _phi(torch.where(inside, (d * d).sum(-1), 4.0), SEQ_RHO)[1]
    slope = ((s["w"][ids.clamp(min=0)] * k)[..., None] * d).sum(1)
    drdq = torch.cat([-slope, torch.ones(len(q), 1, dtype=F64, device=dev)], 1)
    J = torch.cat([(drdq[:, None, :] @ (-R0 @ _skew(s["body"].double())))[:, 0, :], drdq], 1)
    if case["loss"] == "l2":
        psi, omega = 2.0 * r, torch.full_like(r, 2.0)
    else:
        psi = r.clamp(-HUBER, HUBER)
        omega = torch.where(r.abs() <= HUBER, 1.0, HUBER / r.abs())
    A, g6 = (J * omega[:, None]).T @ J, J.T @ psi
    step = torch.linalg.solve(A + 1e-3 * torch.diag(A.diagonal()), -g6)
    v, ang = step[:3], step[:3].norm()
    K = _skew(v)
    eye = torch.eye(3, dtype=F64, device=dev)
    E = eye if float(ang) == 0.0 else eye + torch.sin(ang) / ang * K + (1 - torch.cos(ang)) / ang ** 2 * (K @ K)
    return R0 @ E, t0 + step[3:], float(cost.detach())


def _exact_raster(case, s):
    n = case["lattice"]
    r32 = torch.tensor(CUT * SIGMA, dtype=F32, device=s["c"].device)

    def axis(q0, nq, c):
        x = (q0 + torch.arange(nq, device=c.device, dtype=F64) * case["dq"]).to(F32)
        e = x[:, None] - c.to(F32)[None, :]
        d = x.double()[:, None] - c[None, :]
        f = torch.where(e * e < r32 * r32, torch.exp(-d * d / (2 * SIGMA * SIGMA)), 0.0)
        return f, -f * d / (SIGMA * SIGMA)

    ex, dx = axis(s["x0"], case["nqx"], s["c"][:n, 0])
    ey, dy = axis(s["y0"], case["nqy"], s["c"][::n, 1])
    W = s["w"].reshape(n, n)
    a = W @ ex.T
    h = ey @ a
    return (h, torch.stack([ey @ (W @ dx.T), dy @ a], -1)) if case["grad"] else (h,)


def exact(case, seed):
    k, s = case["kind"], _inputs(case, seed)
    if k == "eval":
        n = case["side"]
        return _Lat(s["c"], n, n, 0.0, 0.0, case["spacing"], None, case["rho"]).height(s["q"], s["w"], False)
    if k == "raster":
        return _exact_raster(case, s)
    if k in ("soft", "align"):
        return _exact_soft(case, s)
    if k == "map":
        n = case["side"]
        full = _Lat(s["c"], n, n, 0.0, 0.0, case["spacing"], None, case["rho"])
        A = torch.nonzero(full.rows(s["pts"], False, 0.0)[2])[:, 0]
        ids = torch.full((n * n,), -1, dtype=torch.long, device=A.device)
        ids[A] = torch.arange(len(A), device=A.device)
        sub = _Lat(s["c"][A].contiguous(), n, n, 0.0, 0.0, case["spacing"], ids, case["rho"])
        G, u = sub.gram(s["pts"], s["pts"][:, 2].double(), False, 0.0)
        G = G.clone()
        G.diagonal().add_(LAM)
        w = torch.zeros(n * n, dtype=F64, device=A.device)
        w[A] = _solve(G, u)
        return (w, *full.height(s["q"], w, False))
    if k == "scans":
        L = _Lat(s["c"], SEQ_SIDE, SEQ_SIDE, SEQ_X0, SEQ_X0, SEQ_H, None)
        rec, out = _Recursion(L, LAM, case["exact"]), []
        for p, q in zip(s["scans"], s["q"]):
            rec.update(p, False, RANGE_SIGMA)
            out.append(L.height(q, rec.w, False))
        return rec.w, out
    if k == "survey":
        L, m, counts = _survey_lattice(case, s)
        rec = _Recursion(L, LAM)
        rec.update(s["pts"], True, SURVEY_NOISE)
        kept = torch.zeros(len(counts), dtype=F64, device=counts.device)
        kept[counts >= 1] = rec.w
        return (None, None, kept, *L.height(s["q"], rec.w, True))
    ws, hs, gs = [], [], []
    for p in s["patches"]:
        M, nx = p["M"], p["nx"]
        ny = -(-M // nx)
        c = _lattice(nx, ny, 0.0, 0.0, p["h"])[:M].contiguous()
        L = _Lat(c, nx, ny, 0.0, 0.0, p["h"], None, SEQ_RHO, count=M)
        G, u = L.gram(p["pts"], p["pts"][:, 2].double(), False, 0.0)
        G = G.clone()
        G.diagonal().add_(LAM)
        w = _solve(G, u)
        h, g = L.height(p["q"], w, False)
        ws.append(w), hs.append(h), gs.append(g)
    return torch.cat(ws), torch.cat(hs), torch.cat(gs)
