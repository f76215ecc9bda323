"""The work that users of this framework have it do, as cases to time and to compare.

A case is one call, or one short sequence of calls, through the public entry points
(`paper_2503_17491_gb300.api`): forward renders, renders differentiated by autograd, refinement
steps (graph replays and plain launches, single keyframes, batches and a sampled window), a
tracking step that registers a new pose, point-cloud export and map growth.  Scenes are analytic
streets, rooms and city blocks with the parameter distributions of
`paper_2503_17491_gb300.scenes`, generated on the GPU.  `exact` recomputes a case in binary64 with
plain torch operations: every ray against every primitive near its columns, blended in range
order, differentiated by torch's autograd.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2503_17491_gb300 import api

DEV = "cuda"
F64 = torch.float64
GROUND = -1.7
ALPHA_MIN = float(np.float32(1.0 / 255.0))
ALPHA_MAX = float(np.float32(0.99))
T_MIN = float(np.float32(1e-4))
SIGMA = 3.0


def listed():
    return [
        # A viewer or a unit of a larger pipeline renders one small scan of a small local map:
        # the smallest call, all latency.
        {"name": "render_room_32x512_2k", "kind": "render", "scene": "room", "n": 2000,
         "shapes": "32x512", "views": 1, "tile": "16x16"},
        # The smallest refinement step, replayed from its CUDA graph (a freshly started local
        # model with one keyframe).
        {"name": "refine_room_32x512_2k", "kind": "refine", "scene": "room", "n": 2000,
         "shapes": "32x512", "views": 1, "tile": "16x16", "graph": True},
        # A user's own training loop: the differentiable render inside torch's autograd, one
        # 64-beam scan of a street.
        {"name": "autograd_street_64x1024_100k", "kind": "autograd", "scene": "street",
         "n": 100_000, "shapes": "64x1024", "views": 1, "tile": "16x16"},
        # One tracking iteration: a new pose is registered, rendered and compared with the query
        # scan (photometric normal equations); ragged image, odd primitive count.
        {"name": "track_street_61x1187_37k", "kind": "track", "scene": "street", "n": 37_501,
         "shapes": "61x1187", "views": 1, "tile": "8x32"},
        # A short window of three sensors of odd sizes refined with plain launches and every
        # optional loss term (opacity, scale, relative range).
        {"name": "refine_ragged_3kf_83k", "kind": "refine", "scene": "street", "n": 83_001,
         "shapes": "40x870,61x1187,33x1801", "views": 3, "tile": "4x64", "graph": False,
         "lambda_o": 0.1, "lambda_s": 0.05, "rho_exp": -1.0},
        # The step of a data-parallel rank: render, loss, parameter gradients, separate Adam.
        {"name": "split_street_4kf_200k", "kind": "split", "scene": "street", "n": 200_000,
         "shapes": "64x1024", "views": 4, "tile": "16x16"},
        # A single large keyframe refined against a dense map of an urban block.
        {"name": "refine_block_128x2048_1m", "kind": "refine", "scene": "block", "n": 1_000_000,
         "shapes": "128x2048", "views": 1, "tile": "16x16", "graph": True},
        # The batched refinement of a local model: twelve keyframes of three sensors, one map.
        {"name": "refine_street_12kf_500k", "kind": "refine", "scene": "street", "n": 500_000,
         "shapes": "64x1024,128x1024,32x1800", "views": 12, "tile": "8x32", "graph": True},
        # A long mapping run near its end: a window of eight scans over a map of 3 M primitives,
        # two keyframes drawn per step, normals of the rendered range map.
        {"name": "refine_city_window_3m", "kind": "refine", "scene": "city", "n": 3_000_000,
         "shapes": "128x1024", "views": 8, "tile": "32x8", "graph": False, "draws": 2,
         "normal_mode": 1, "lambda_n": 0.1},
        # Export of a local model: eight scans rendered forward only and back-projected.
        {"name": "cloud_city_8x128x1024_1m", "kind": "cloud", "scene": "city", "n": 1_000_000,
         "shapes": "128x1024", "views": 8, "tile": "16x16"},
        # Map growth from the registered keyframes: masks, weights and a draw of new primitives.
        {"name": "grow_street_12kf_50k", "kind": "grow", "scene": "street", "n": 50_000,
         "shapes": "64x1024,128x1024,32x1800", "views": 12, "tile": "16x16"},
    ]


def draw(rng):
    kind = rng.choice(["render", "autograd", "track", "refine", "refine", "refine", "split",
                       "cloud", "grow"])
    log_uniform = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    views = 1 if kind in ("track", "autograd") else log_uniform(1, 8)
    budget = 700_000 // views                      # pixels a view, at most
    shapes = []
    for _ in range(min(views, rng.choice([1, 2, 3]))):
        rows = log_uniform(16, 128)
        cols = log_uniform(256, 2048)
        while rows * cols > budget:
            cols = cols // 2 + 1
        shapes.append("%dx%d" % (rows, max(cols, 64)))
    n = log_uniform(1500, max(3000, min(1_000_000, 3_000_000 // views)))
    case = {"kind": kind, "scene": "room" if n < 10_000 else rng.choice(["street", "block"]),
            "n": n, "shapes": ",".join(shapes), "views": views,
            "tile": rng.choice(["16x16", "8x32", "32x8", "4x64"])}
    if kind == "grow":
        case["n"] = log_uniform(500, 60_000)
        case["scene"] = "street"
    if kind == "refine":
        case["graph"] = rng.random() < 0.5
        case["normal_mode"] = rng.choice([0, 0, 1])
        if rng.random() < 0.3:
            case.update(lambda_o=0.1, lambda_s=0.05, rho_exp=-1.0)
        if views > 1 and rng.random() < 0.4:
            case["draws"] = 2
    return case


# ---------------------------------------------------------------------------------------------
# scenes: rectangles and vertical cylinders, sampled and ray-cast with torch on the GPU
# ---------------------------------------------------------------------------------------------

class _Surfaces:
    def __init__(self):
        self.rect, self.cyl = [], []

    def plane(self, c, n, u, hu, hv):
        n, u = np.asarray(n, float), np.asarray(u, float)
        self.rect.append(np.concatenate([c, n, u, np.cross(n, u), [hu, hv]]))

    def box(self, cx, cy, cz, hx, hy, hz, yaw):
        c, s = math.cos(yaw), math.sin(yaw)
        ex, ey, ez = np.array([c, s, 0.0]), np.array([-s, c, 0.0]), np.array([0, 0, 1.0])
        o = np.array([cx, cy, cz])
        for sg in (1.0, -1.0):
            self.plane(o + sg * hx * ex, sg * ex, ey, hy, hz)
            self.plane(o + sg * hy * ey, sg * ey, ex, hx, hz)
        self.plane(o + hz * ez, ez, ex, hx, hy)

    def pole(self, x, y, r, z0, z1):
        self.cyl.append([x, y, r, z0, z1])


def _scene(kind, rng):
    """The surfaces of a scene and the length of the sensor's path along x."""
    s = _Surfaces()
    ez = [0, 0, 1.0]
    if kind == "room":
        s.plane([0, 0, GROUND], ez, [1.0, 0, 0], 25, 25)
        for nx, ny in ((-1.0, 0.0), (0.0, -1.0), (0.0, 1.0)):
            d = rng.uniform(5, 20)
            s.plane([-nx * d, -ny * d, (4.0 + GROUND) / 2], [nx, ny, 0], [ny, -nx, 0], 20.0,
                    (4.0 - GROUND) / 2)
        return s, 2.0
    if kind == "street":
        yl, yr = rng.uniform(8, 30), rng.uniform(8, 30)
        s.plane([25, (yl - yr) / 2, GROUND], ez, [1.0, 0, 0], 65, (yl + yr) / 2)
        hz = (12.0 - GROUND) / 2
        s.plane([25, yl, GROUND + hz], [0, -1.0, 0], [1.0, 0, 0], 65, hz)
        s.plane([25, -yr, GROUND + hz], [0, 1.0, 0], [1.0, 0, 0], 65, hz)
        for _ in range(200):
            y = (yl - 2.0) if rng.random() < 0.5 else 2.0 - yr
            s.pole(rng.uniform(-40, 90), y + rng.uniform(-0.5, 0.5), 0.3, GROUND, 4.0)
        return s, 50.0
    if kind == "block":
        s.plane([0, 0, GROUND], ez, [1.0, 0, 0], 50, 50)
        for gx in range(-40, 41, 16):
            for gy in range(-40, 41, 16):
                if abs(gx) < 10 or abs(gy) < 10:
                    continue
                h = rng.uniform(5, 25)
                s.box(gx + rng.uniform(-1, 1), gy + rng.uniform(-1, 1), GROUND + h / 2,
                      rng.uniform(3, 6.5), rng.uniform(3, 6.5), h / 2, rng.uniform(-0.2, 0.2))
        for _ in range(60):
            x, y = rng.uniform(-45, 45), rng.uniform(-45, 45)
            if min(abs(x), abs(y)) < 8 and math.hypot(x, y) > 1.5:
                s.pole(x, y, 0.3, GROUND, 4.0)
        s.pole(1.2, 0.8, 0.3, GROUND, -0.2)            # near objects
        s.box(-2.5, -1.5, GROUND + 0.75, 0.8, 0.4, 0.75, 0.0)
        return s, 4.0
    # city: a long street through buildings, trunks and vehicles; the window is its middle
    length = 600.0
    s.plane([length / 2, 0, GROUND], ez, [1.0, 0, 0], length / 2 + 60, 60)
    x = -40.0
    while x < length + 40:
        for side in (-1, 1):
            w, d, h = rng.uniform(8, 25), rng.uniform(8, 15), rng.uniform(6, 30)
            s.box(x + w / 2, side * (rng.uniform(10, 18) + d / 2), GROUND + h / 2, w / 2, d / 2,
                  h / 2, rng.uniform(-0.05, 0.05))
        x += rng.uniform(15, 35)
    for _ in range(50):
        s.pole(rng.uniform(-20, length + 20), rng.choice([-1, 1]) * rng.uniform(6, 8), 0.25,
               GROUND, 2.5)
    for _ in range(40):
        s.box(rng.uniform(-20, length + 20), rng.choice([-1, 1]) * rng.uniform(2.5, 5),
              GROUND + 0.8, 2.2, 0.9, 0.8, rng.uniform(-0.1, 0.1))
    return s, 16.0


def _tables(s):
    t = lambda a, w: torch.tensor(np.array(a, np.float64).reshape(-1, w), device=DEV)  # noqa: E731
    return t(s.rect, 14), t(s.cyl, 5)


def _map(s, n, gen):
    """n primitives on the surfaces (area-proportional), float32 parameter tensors."""
    R, C = _tables(s)
    area = torch.cat([4 * R[:, 12] * R[:, 13], 2 * math.pi * C[:, 2] * (C[:, 4] - C[:, 3])])
    uni = lambda *sh: torch.rand(*sh, generator=gen, device=DEV, dtype=F64)       # noqa: E731
    gauss = lambda *sh: torch.randn(*sh, generator=gen, device=DEV, dtype=F64)    # noqa: E731
    cum = torch.cumsum(area, 0)
    k = torch.searchsorted(cum, uni(n) * cum[-1]).clamp(max=len(area) - 1)
    on_rect = (k < len(R))[:, None]
    r = R[k.clamp(max=len(R) - 1)]
    a, b = 2 * uni(n, 1) - 1, 2 * uni(n, 1) - 1
    p = r[:, 0:3] + a * r[:, 12:13] * r[:, 6:9] + b * r[:, 13:14] * r[:, 9:12]
    nrm = r[:, 3:6]
    if len(C):
        c = C[(k - len(R)).clamp(min=0)]
        ang = math.pi * a
        nc = torch.cat([torch.cos(ang), torch.sin(ang), torch.zeros_like(ang)], 1)
        z = c[:, 3:4] + 0.5 * (b + 1) * (c[:, 4:5] - c[:, 3:4])
        pc = torch.cat([c[:, 0:1] + c[:, 2:3] * nc[:, 0:1], c[:, 1:2] + c[:, 2:3] * nc[:, 1:2], z],
                       1)
        p, nrm = torch.where(on_rect, p, pc), torch.where(on_rect, nrm, nc)
    mu = p + 0.02 * gauss(n, 1) * nrm
    # shortest rotation e_z -> normal, after a random turn about e_z, plus quaternion noise
    w = 1 + nrm[:, 2:3]
    q1 = torch.cat([w, -nrm[:, 1:2], nrm[:, 0:1], torch.zeros_like(w)], 1)
    q1 = torch.where(w > 1e-6, q1, torch.tensor([0.0, 1.0, 0.0, 0.0], device=DEV, dtype=F64))
    q1 = q1 / q1.norm(dim=1, keepdim=True)
    h = math.pi * uni(n)
    cw, sw = torch.cos(h), torch.sin(h)
    q = torch.stack([q1[:, 0] * cw - q1[:, 3] * sw, q1[:, 1] * cw + q1[:, 2] * sw,
                     q1[:, 2] * cw - q1[:, 1] * sw, q1[:, 3] * cw + q1[:, 0] * sw], 1)
    q = q + 0.05 * gauss(n, 4)
    q = q / q.norm(dim=1, keepdim=True)
    o = 0.3 + 0.69 * uni(n, 1)
    return [torch.cat([mu, torch.log(o / (1 - o))], 1).float().contiguous(),
            q.float().contiguous(), (-3.0 + 2.0 * uni(n, 2)).float().contiguous()]


def _shapes(case):
    sh = [tuple(int(v) for v in t.split("x")) for t in case["shapes"].split(",")]
    return [sh[k % len(sh)] for k in range(case["views"])]


def _pose(rng, x, y):
    T = np.eye(4)
    a, b, c = rng.uniform(-0.15, 0.15), rng.uniform(-0.03, 0.03), rng.uniform(-0.03, 0.03)
    ca, sa, cb, sb, cc, sc = (math.cos(a), math.sin(a), math.cos(b), math.sin(b), math.cos(c),
                              math.sin(c))
    T[:3, :3] = (np.array([[ca, -sa, 0], [sa, ca, 0], [0, 0, 1.0]]) @
                 np.array([[cb, 0, sb], [0, 1.0, 0], [-sb, 0, cb]]) @
                 np.array([[1.0, 0, 0], [0, cc, -sc], [0, sc, cc]]))
    T[:3, 3] = [x + rng.uniform(-0.3, 0.3), y, rng.uniform(-0.2, 0.2)]
    return T


def _views(case, path, rng):
    out = []
    shapes = _shapes(case)
    x0 = 300.0 if case["scene"] == "city" else 0.0
    for k, (h, w) in enumerate(shapes):
        e = float(np.float32(math.radians(15.0 if h <= 33 else 22.5)))
        T = _pose(rng, x0 + path * k / max(1, len(shapes) - 1), rng.uniform(-0.8, 0.8))
        out.append(api.ViewSpec(T, h, w, -e, e))
    return out


def _angles(view):
    """Azimuth of each column and elevation of each row, binary64."""
    g = math.pi - 2 * math.pi * (torch.arange(view.cols, device=DEV, dtype=F64) + 0.5) / view.cols
    e = view.elev_max - torch.arange(view.rows, device=DEV, dtype=F64) * (
        (view.elev_max - view.elev_min) / (view.rows - 1))
    return g, e


def _rays(g, e):
    """Unit rays (rows, cols, 3) of azimuths g and elevations e."""
    cg, sg, ce, se = torch.cos(g), torch.sin(g), torch.cos(e)[:, None], torch.sin(e)[:, None]
    return torch.stack([ce * cg, ce * sg, se.expand(-1, len(g))], 2)


def _target(s, view, gen):
    """Ray-cast range (P,) with 1 cm noise and normals (3, P) in the sensor frame; 0 where the ray
    meets nothing within 100 m."""
    R, C = _tables(s)
    Rw = torch.tensor(view.T_ws[:3, :3], device=DEV)
    o = torch.tensor(view.T_ws[:3, 3], device=DEV)
    vs = _rays(*_angles(view)).reshape(-1, 3)
    d = vs @ Rw.T
    best = torch.full((len(d),), math.inf, device=DEV, dtype=F64)
    nrm = torch.zeros_like(d)
    for k0 in range(0, len(R), 64):
        r = R[k0:k0 + 64]
        t = ((r[:, 0:3] - o) * r[:, 3:6]).sum(1) / (d @ r[:, 3:6].T)
        qu = t * (d @ r[:, 6:9].T) - ((r[:, 0:3] - o) * r[:, 6:9]).sum(1)
        qv = t * (d @ r[:, 9:12].T) - ((r[:, 0:3] - o) * r[:, 9:12]).sum(1)
        ok = (t > 1e-6) & (qu.abs() <= r[:, 12]) & (qv.abs() <= r[:, 13])
        t, k = torch.where(ok, t, math.inf).min(1)
        m = t < best
        best = torch.where(m, t, best)
        nrm = torch.where(m[:, None], r[k, 3:6], nrm)
    for k0 in range(0, len(C), 64):
        c = C[k0:k0 + 64]
        ox, oy = o[0] - c[:, 0], o[1] - c[:, 1]
        a = d[:, 0:1] ** 2 + d[:, 1:2] ** 2
        b = d[:, 0:1] * ox + d[:, 1:2] * oy
        disc = b * b - a * (ox * ox + oy * oy - c[:, 2] ** 2)
        t = (-b - disc.clamp(min=0).sqrt()) / a
        z = o[2] + t * d[:, 2:3]
        ok = (disc > 0) & (t > 1e-6) & (z >= c[:, 3]) & (z <= c[:, 4])
        t, k = torch.where(ok, t, math.inf).min(1)
        m = t < best
        p = o + torch.where(m, t, 0.0)[:, None] * d
        nc = torch.stack([(p[:, 0] - c[k, 0]) / c[k, 2], (p[:, 1] - c[k, 1]) / c[k, 2],
                          torch.zeros_like(t)], 1)
        best = torch.where(m, t, best)
        nrm = torch.where(m[:, None], nc, nrm)
    valid = best <= 100.0
    ns = nrm @ Rw
    ns = torch.where(((ns * vs).sum(1) > 0)[:, None], -ns, ns) * valid[:, None]
    noise = 0.01 * torch.randn(len(d), generator=gen, device=DEV, dtype=F64)
    depth = torch.where(valid, best + noise, 0.0).clamp(min=0)
    return depth.float().contiguous(), ns.T.float().contiguous()


def _inputs(case, seed):
    """Everything a case is made of, from the seed alone."""
    rng = random.Random(seed * 7919 + 17)
    gen = torch.Generator(device=DEV).manual_seed(seed * 104729 + 5)
    s, path = _scene(case["scene"], rng)
    views = _views(case, path, rng)
    inp = {"views": views, "P": sum(v.rows * v.cols for v in views), "seed": seed}
    kind = case["kind"]
    if kind != "grow":
        inp["params"] = _map(s, case["n"], gen)
    if kind in ("refine", "split", "grow"):
        inp["targets"] = [_target(s, v, gen) for v in views]
    if kind == "track":
        inp["query"] = _target(s, views[0], gen)[0]
        # the poses tried, each off the query's by a few centimetres and a fraction of a degree
        inp["poses"], inp["T_qm"] = [], []
        for _ in range(4):
            x = np.array([rng.gauss(0, 1) for _ in range(6)]) * ([0.03] * 3 + [0.002] * 3)
            E = np.eye(4)
            E[:3, :3] = _rodrigues(x[3:])
            E[:3, 3] = x[:3]
            v = views[0]
            inp["poses"].append(api.ViewSpec(v.T_ws @ E, v.rows, v.cols, v.elev_min, v.elev_max))
            inp["T_qm"].append(torch.tensor(E[:3], device=DEV).float().contiguous())
    if kind == "autograd":
        P = inp["P"]
        up = lambda *sh: torch.randn(*sh, generator=gen, device=DEV)   # noqa: E731
        inp["up"] = (up(P), 0.5 * up(3, P), 0.3 * up(P))
    if kind == "grow":
        td = torch.cat([t[0] for t in inp["targets"]])
        u = torch.rand(inp["P"], generator=gen, device=DEV)
        inp["alpha"] = (1.2 * u).clamp(max=0.9999)
        inp["depth"] = td * inp["alpha"] + 0.05 * torch.randn(inp["P"], generator=gen, device=DEV)
    if kind in ("refine", "split"):
        # moments of a refinement in progress (100 steps taken)
        inp["state"] = []
        for w in (4, 4, 2):
            inp["state"].append(torch.randn(case["n"], w, generator=gen, device=DEV))
        for w in (4, 4, 2):
            inp["state"].append(1.0 + 4.0 * torch.rand(case["n"], w, generator=gen, device=DEV))
        inp["state"].append(torch.full((1,), 100, dtype=torch.int32, device=DEV))
    return inp


def _rodrigues(w):
    th = float(np.linalg.norm(w))
    if th == 0:
        return np.eye(3)
    k = w / th
    K = np.array([[0, -k[2], k[1]], [k[2], 0, -k[0]], [-k[1], k[0], 0]])
    return np.eye(3) + math.sin(th) * K + (1 - math.cos(th)) * K @ K


def _render_cfg(case):
    th, tw = (int(v) for v in case["tile"].split("x"))
    return api.RenderConfig(tile_h=th, tile_w=tw)


def _loss_cfg(case):
    return api.LossConfig(lambda_n=case.get("lambda_n", 1.0), lambda_o=case.get("lambda_o", 0.0),
                          lambda_s=case.get("lambda_s", 0.0), tau_s=0.2,
                          normal_mode=case.get("normal_mode", 0),
                          rho_exp=case.get("rho_exp", 0.0))


# ---------------------------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------------------------

def prepare(case, seed):
    inp = _inputs(case, seed)
    st = {"kind": case["kind"], "inp": inp}
    kind = case["kind"]
    if kind == "refine":
        views = inp["views"]
        r = api.Refiner([p.clone() for p in inp["params"]], views, inp["targets"],
                        mode="batched", cfg=_render_cfg(case), loss_cfg=_loss_cfg(case))
        if case.get("draws"):
            r.ctx.set_view_sampling(case["draws"], 0.4, seed)
        if case.get("graph"):
            r.capture()
            if case.get("draws"):   # the captured steps' draws restart with the run
                r.ctx.set_view_sampling(case["draws"], 0.4, seed)
        for dst, src in zip((*r.params, *r.state), (*inp["params"], *inp["state"])):
            dst.copy_(src)
        st["refiner"] = r
        return st
    n = 1 if kind == "grow" else case["n"]
    ctx = api.SplatContext(n, len(inp["views"]), inp["P"], None, _render_cfg(case))
    ctx.set_views(inp["views"])
    st["ctx"] = ctx
    if kind == "autograd":
        st["leaves"] = [p.clone().requires_grad_() for p in inp["params"]]
    if kind == "split":
        st["params"] = [p.clone() for p in inp["params"]]
        st["state"] = tuple(t.clone() for t in inp["state"])
        st["t_depth"] = torch.cat([t[0] for t in inp["targets"]]).contiguous()
        st["t_normal"] = torch.cat([t[1] for t in inp["targets"]], 1).contiguous()
    if kind == "track":
        st["k"] = 0
    if kind == "grow":
        st["t_depth"] = torch.cat([t[0] for t in inp["targets"]]).contiguous()
        st["slots"] = [torch.zeros(case["n"], w, device=DEV) for w in (4, 4, 2)]
        st["cfg"] = api.DensifyConfig(refine=True, seed=seed)
    return st


def run(st):
    kind, inp = st["kind"], st["inp"]
    if kind == "refine":
        r = st["refiner"]
        loss = r.step()
        # the loss as a training log keeps it: it is a sum of binary32 terms
        return {"params": r.params, "moments": list(r.state[:6]), "step": r.state[6],
                "loss": loss.float()}
    ctx = st["ctx"]
    if kind == "render":
        return ctx.render(*inp["params"])
    if kind == "autograd":
        img = api.render(*st["leaves"], ctx)
        return {"images": img, "grads": torch.autograd.grad(img, st["leaves"], inp["up"])}
    if kind == "split":
        p = st["params"]
        depth, normal, alpha = ctx.render(*p)
        loss, gD, gN, gO = ctx.view_loss(depth, normal, alpha, st["t_depth"], st["t_normal"])
        grads = ctx.backward(*p, gD, gN, gO)
        api.adam_step(p, grads, st["state"])
        return {"grads": grads, "params": p, "moments": list(st["state"][:6]),
                "loss": loss.float()}
    if kind == "track":
        k = st["k"] % 4
        st["k"] += 1
        ctx.set_views([inp["poses"][k]])
        depth, normal, alpha = ctx.render(*inp["params"])
        eqs = ctx.photometric(0, depth, alpha, inp["query"], inp["T_qm"][k])
        return {"images": (depth, normal, alpha), "normal_equations": eqs}
    if kind == "cloud":
        depth, normal, alpha = ctx.render(*inp["params"])
        return {"points": ctx.backproject(depth, alpha), "normal": normal, "alpha": alpha}
    ctx.densify(st["slots"], 0, st["slots"][0].shape[0], st["t_depth"], inp["depth"],
                inp["alpha"], st["cfg"])
    return st["slots"]


def work(case):
    """Bytes: parameters, moments, gradients, targets and images, each once.  Operations: the
    intersection (48 binary32 operations) and the adjoint (150) of the pairs that contribute to a
    pixel; their number follows the density of the map and is about 40 a pixel for the dense
    scenes and 10 for the small room."""
    shapes = _shapes(case)
    if case.get("draws"):
        shapes = shapes[:1]         # the newest keyframe always comes up most: one or two views
    P, n, kind = sum(h * w for h, w in shapes), case["n"], case["kind"]
    hits = P * (10 if case["scene"] == "room" else 40)
    img, par = 20 * P, 40 * n
    if kind == "render":
        return {"bytes": par + img, "flops": 48 * hits}
    if kind == "autograd":
        return {"bytes": 2 * par + 2 * img, "flops": 198 * hits}
    if kind == "refine":
        return {"bytes": 6 * par + 16 * P, "flops": 198 * hits + 150 * n}
    if kind == "split":
        return {"bytes": 7 * par + 16 * P, "flops": 198 * hits + 150 * n}
    if kind == "track":
        return {"bytes": par + img + 4 * P, "flops": 48 * hits + 100 * P}
    if kind == "cloud":
        return {"bytes": par + 28 * P, "flops": 48 * hits + 30 * P}
    return {"bytes": 12 * P + 40 * n, "flops": 10 * P}


# ---------------------------------------------------------------------------------------------
# binary64 reference
# ---------------------------------------------------------------------------------------------

def _sensor(params, view):
    """Sensor-frame quantities of every primitive: b_alpha, b_beta, n, b_c, opacity (N, 13),
    differentiable in the parameters; the quaternion is normalised inside."""
    pl, q, ls = params
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    ta = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + w * z), 2 * (x * z - w * y)], 1)
    tb = torch.stack([2 * (x * y - w * z), 1 - 2 * (x * x + z * z), 2 * (y * z + w * x)], 1)
    tn = torch.stack([2 * (x * z + w * y), 2 * (y * z - w * x), 1 - 2 * (x * x + y * y)], 1)
    R = torch.tensor(view.T_ws[:3, :3].T.copy(), device=DEV)
    t = torch.tensor(-(view.T_ws[:3, :3].T @ view.T_ws[:3, 3]), device=DEV)
    s = torch.exp(ls)
    return torch.cat([(s[:, 0:1] * ta) @ R.T, (s[:, 1:2] * tb) @ R.T, tn @ R.T,
                      pl[:, 0:3] @ R.T + t, torch.sigmoid(pl[:, 3:4])], 1)


def _strip(Q, idx, rays):
    """Blend the primitives idx (in range order) along the rays (M, 3): range, normal, opacity."""
    with torch.no_grad():
        c = Q.detach()[idx]
        ba, bb, n, bc, o = c[:, 0:3], c[:, 3:6], c[:, 6:9], c[:, 9:12], c[:, 12]
        t = (bc * n).sum(1) / (rays @ n.T)
        sa = (t * (rays @ ba.T) - (bc * ba).sum(1)) / (ba * ba).sum(1)
        sb = (t * (rays @ bb.T) - (bc * bb).sum(1)) / (bb * bb).sum(1)
        ok = (t > 0) & torch.isfinite(t) & (torch.maximum(sa.abs(), sb.abs()) <= SIGMA)
        sa.mul_(sa).add_(sb.mul_(sb))
        ok &= o * torch.exp(-0.5 * sa) >= ALPHA_MIN
        px, m = ok.nonzero(as_tuple=True)
        del t, sa, sb, ok
        cnt = torch.bincount(px, minlength=len(rays))
        pos = torch.arange(len(px), device=DEV) - (torch.cumsum(cnt, 0) - cnt)[px]
        K = max(1, int(cnt.max()))
        # the sign that turns each normal towards the sensor is fixed
        flip = torch.where((n * bc).sum(1) > 0, -1.0, 1.0)[m]
    c = Q[idx[m]]
    ba, bb, n, bc, o = c[:, 0:3], c[:, 3:6], c[:, 6:9], c[:, 9:12], c[:, 12]
    v = rays[px]
    t = (bc * n).sum(1) / (v * n).sum(1)
    X = t[:, None] * v - bc
    sa = (X * ba).sum(1) / (ba * ba).sum(1)
    sb = (X * bb).sum(1) / (bb * bb).sum(1)
    a = (o * torch.exp(-0.5 * (sa * sa + sb * sb))).clamp(max=ALPHA_MAX)
    A = torch.zeros(len(rays), K, device=DEV, dtype=F64).index_put((px, pos), a)
    T = torch.cumprod(1 - A, 1)
    before = torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
    wgt = (A * before * (T.detach() >= T_MIN))[px, pos]
    zero = torch.zeros(len(rays), 5, device=DEV, dtype=F64)
    terms = torch.cat([(wgt * t)[:, None], (wgt * flip)[:, None] * n, wgt[:, None]], 1)
    return zero.index_add(0, px, terms)


def _strips(Q, view):
    """(column range, candidate primitives in range order, rays) of the view's column strips."""
    g, e = _angles(view)
    q = Q.detach()
    bc = q[:, 9:12]
    reach = SIGMA * ((q[:, 0:3] ** 2).sum(1) + (q[:, 3:6] ** 2).sum(1)).sqrt() * 1.0001
    rxy = bc[:, 0:2].norm(dim=1)
    az = torch.atan2(bc[:, 1], bc[:, 0])
    half = torch.where(rxy > reach, torch.asin((reach / rxy).clamp(max=1.0)), 7.0)
    # primitives that stay clear of the view's elevations are left out
    el, r3 = torch.atan2(bc[:, 2], rxy), bc.norm(dim=1)
    dh = torch.where(r3 > reach, torch.asin((reach / r3).clamp(max=1.0)), 7.0) + 1e-6
    keep = (el + dh >= view.elev_min) & (el - dh <= view.elev_max) & (q[:, 12] >= ALPHA_MIN)
    order = torch.argsort(bc.norm(dim=1).float(), stable=True)   # range in binary32, ties by id
    order = order[keep[order]]
    az, half = az[order], half[order]
    step = 8
    for c0 in range(0, view.cols, step):
        c1 = min(view.cols, c0 + step)
        mid = 0.5 * (g[c0] + g[c1 - 1])
        off = torch.remainder(az - mid + math.pi, 2 * math.pi) - math.pi
        near = off.abs() <= half + 0.5 * (g[c0] - g[c1 - 1]) + 1e-6
        yield c0, c1, order[near], _rays(g[c0:c1], e).reshape(-1, 3)


def _images(params, view):
    """Binary64 images (5, rows, cols): range, normal, opacity."""
    with torch.no_grad():
        Q = _sensor(params, view)
        out = torch.zeros(view.rows, view.cols, 5, device=DEV, dtype=F64)
        for c0, c1, idx, rays in _strips(Q, view):
            if len(idx):
                out[:, c0:c1] = _strip(Q, idx, rays).reshape(view.rows, c1 - c0, 5)
    return out.permute(2, 0, 1)


def _gradients(params, view, up):
    """Adds the gradient of sum(up * images) to the parameters' .grad."""
    Q = _sensor(params, view)
    leaf = Q.detach().requires_grad_()
    for c0, c1, idx, rays in _strips(Q, view):
        if len(idx):
            img = _strip(leaf, idx, rays).reshape(view.rows, c1 - c0, 5)
            img.backward(up[:, :, c0:c1].permute(1, 2, 0))
    if leaf.grad is not None:
        Q.backward(leaf.grad)


def _range_normals(D, view, t_depth):
    """Normals of the range map D and the pixels that have one."""
    P = D[:, :, None] * _rays(*_angles(view))
    dx = torch.roll(P, -1, 1)[:-1] - P[:-1]
    dy = P[1:] - P[:-1]
    m = torch.linalg.cross(dx, dy)
    side = torch.where((m.detach() * P[:-1].detach()).sum(2) > 0, -1.0, 1.0)
    ok = (t_depth > 0) & (D.detach() > 0)
    ok = ok[:-1] & torch.roll(ok, -1, 1)[:-1] & ok[1:] & (m.detach().norm(dim=2) > 0)
    m = torch.where(ok[..., None], m, torch.ones_like(m))
    return side[..., None] * m / m.norm(dim=2, keepdim=True), ok


def _loss64(img, view, target, cfg):
    td = target[0].double().reshape(view.rows, view.cols)
    on = td > 0
    D, N, O = img[0], img[1:4], img[4]
    rho = torch.where(on, td, torch.ones_like(td)) ** cfg.rho_exp
    L = (rho * (D - td).abs())[on].sum()
    if cfg.normal_mode == 0:
        tn = target[1].double().reshape(3, view.rows, view.cols)
        L = L + cfg.lambda_n * (1 - (N * tn).sum(0))[on].sum()
    else:
        nd, ok = _range_normals(D, view, td)
        L = L + cfg.lambda_n * (1 - (N[:, :-1].permute(1, 2, 0) * nd).sum(2))[ok].sum()
    if cfg.lambda_o:
        L = L - cfg.lambda_o * torch.log(O.clamp(min=cfg.o_eps))[on].sum()
    return L


def _philox(counter, key):
    c, k = [int(v) for v in counter], [int(v) for v in key]
    M = 0xFFFFFFFF
    for r in range(10):
        a, b = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [((b >> 32) ^ c[1] ^ k[0]) & M, b & M, ((a >> 32) ^ c[3] ^ k[1]) & M, a & M]
        k = [(k[0] + 0x9E3779B9) & M, (k[1] + 0xBB67AE85) & M]
    return c


def _drawn(case, seed, step=0):
    """The views drawn for a step: ages from the truncated geometric law, one Philox word each."""
    V = case["views"]
    if not case.get("draws"):
        return list(range(V))
    p = [0.4 * 0.6 ** a for a in range(V)]
    cum = np.cumsum(np.array(p) / sum(p))
    thr = [math.floor(c * 4294967296.0) for c in cum[:-1]]
    ages = {sum(_philox((j, step, 0, 0), (seed & 0xFFFFFFFF, seed >> 32))[0] >= t for t in thr)
            for j in range(case["draws"])}
    return sorted(V - 1 - a for a in ages)


def _photometric64(img, view, query, T):
    """Normal equations (29 values) of the photometric residual, pixel by pixel."""
    D, O = img[0], img[4]
    g, e = _angles(view)
    H, W = view.rows, view.cols
    q = query.double().reshape(H, W)
    T = T.double()
    d = D / O.clamp(min=1e-30)
    p = d[..., None] * _rays(g, e)
    x = p @ T[:, :3].T + T[:, 3]
    rxy = x[..., 0:2].norm(dim=2)
    rng = x.norm(dim=2)
    dg, dt = 2 * math.pi / W, (view.elev_max - view.elev_min) / (H - 1)
    cc = (math.pi - torch.atan2(x[..., 1], x[..., 0])) / dg - 0.5
    rr = (view.elev_max - torch.atan2(x[..., 2], rxy)) / dt
    r0, c0 = torch.floor(rr), torch.floor(cc)
    fr, fc = rr - r0, cc - c0
    ok = (O >= 0.5) & (r0 >= 0) & (r0 + 1 <= H - 1)
    ri, ci = r0.clamp(0, H - 2).long(), torch.remainder(c0, W).long()
    cj = (ci + 1) % W
    a, b, c, f = q[ri, ci], q[ri, cj], q[ri + 1, ci], q[ri + 1, cj]
    ok &= (a > 0) & (b > 0) & (c > 0) & (f > 0)
    s = (1 - fr) * ((1 - fc) * a + fc * b) + fr * ((1 - fc) * c + fc * f)
    sc = (1 - fr) * (b - a) + fr * (f - c)
    sr = (1 - fc) * (c - a) + fc * (f - b)
    zero = torch.zeros_like(rxy)
    dgam = torch.stack([-x[..., 1] / rxy ** 2, x[..., 0] / rxy ** 2, zero], 2)
    dele = torch.stack([-x[..., 2] * x[..., 0] / (rxy * rng ** 2),
                        -x[..., 2] * x[..., 1] / (rxy * rng ** 2), rxy / rng ** 2], 2)
    gx = x / rng[..., None] + (sc / dg)[..., None] * dgam + (sr / dt)[..., None] * dele
    gp = gx @ T[:, :3]
    J = torch.cat([gp, torch.linalg.cross(p, gp)], 2)[ok]
    r = (rng - s)[ok]
    w = (0.2 / r.abs().clamp(min=1e-30)).clamp(max=1.0)
    Hm = (w[:, None, None] * J[:, :, None] * J[:, None, :]).sum(0)
    iu = torch.triu_indices(6, 6, device=DEV)
    cost = torch.where(r.abs() <= 0.2, 0.5 * r * r, 0.2 * (r.abs() - 0.1)).sum()
    return torch.cat([Hm[iu[0], iu[1]], (w[:, None] * r[:, None] * J).sum(0), cost[None],
                      torch.tensor([float(len(r))], device=DEV, dtype=F64)])


def _adam64(p, g, m, v, lr, step):
    f = lambda x: float(np.float32(x))   # noqa: E731
    b1, b2 = f(0.9), f(0.999)
    m = b1 * m.double() + (1 - b1) * g
    v = b2 * v.double() + (1 - b2) * g * g
    mh, vh = m / (1 - b1 ** step), v / (1 - b2 ** step)
    return p.detach() - lr * mh / (vh.sqrt() + f(1e-15)), m, v


def exact(case, seed):
    kind = case["kind"]
    # rays against the primitives near their columns: under 20 s at the listed sizes
    pairs = sum(h * w for h, w in _shapes(case)[:case.get("draws") or None]) * case["n"]
    if kind == "grow" or pairs > 1.1e12:
        return None          # drawn by exact integer arithmetic on binary32 weights, or too long
    inp = _inputs(case, seed)
    views = inp["views"]
    if kind == "track":
        views = [inp["poses"][0]]
    live = _drawn(case, seed) if kind == "refine" else range(len(views))
    params = [p.double().requires_grad_() for p in inp["params"]]
    imgs = {k: _images(params, views[k]) for k in live}
    pack = lambda f: torch.cat([f(imgs[k]).reshape(-1) for k in live])   # noqa: E731
    planes = lambda: torch.cat([imgs[k][1:4].reshape(3, -1) for k in live], 1)   # noqa: E731
    if kind == "render":
        return pack(lambda i: i[0]), planes(), pack(lambda i: i[4])
    if kind == "track":
        i = imgs[0]
        return {"images": (pack(lambda i: i[0]), planes(), pack(lambda i: i[4])),
                "normal_equations": _photometric64(i, views[0], inp["query"], inp["T_qm"][0])}
    if kind == "cloud":
        pts = []
        for k in live:
            v, i = views[k], imgs[k]
            T = torch.tensor(v.T_ws, device=DEV)
            x = (i[0] / i[4])[..., None] * _rays(*_angles(v)) @ T[:3, :3].T + T[:3, 3]
            x = torch.where((i[4] >= 0.5)[..., None], x, math.nan)
            pts.append(x.reshape(-1, 3).T)
        return {"points": torch.cat(pts, 1), "normal": planes(), "alpha": pack(lambda i: i[4])}
    if kind == "autograd":
        v = views[0]
        up = torch.cat([inp["up"][0][None], inp["up"][1], inp["up"][2][None]]).double()
        _gradients(params, v, up.reshape(5, v.rows, v.cols))
        return {"images": (pack(lambda i: i[0]), planes(), pack(lambda i: i[4])),
                "grads": [p.grad for p in params]}
    cfg = _loss_cfg(case) if kind == "refine" else api.LossConfig()
    loss = torch.zeros(1, device=DEV, dtype=F64)
    for k in live:
        leaf = imgs[k].detach().requires_grad_()
        L = _loss64(leaf, views[k], inp["targets"][k], cfg)
        L.backward()
        loss += L.detach()
        _gradients(params, views[k], leaf.grad)
    grads = [p.grad if p.grad is not None else torch.zeros_like(p) for p in params]
    if kind == "refine" and cfg.lambda_s:
        s = torch.exp(params[2].detach())
        big, which = s.max(1)
        over = big > cfg.tau_s
        loss += cfg.lambda_s * (big - cfg.tau_s)[over].sum()
        add = torch.zeros_like(s)
        add[torch.arange(len(s), device=DEV), which] = torch.where(over, cfg.lambda_s * big, 0.0)
        grads[2] = grads[2] + add
    f = lambda x: float(np.float32(x))   # noqa: E731
    lr = (torch.tensor([f(1e-3)] * 3 + [f(2e-2)], device=DEV, dtype=F64), f(2e-3), f(5e-3))
    st, step = inp["state"], int(inp["state"][6]) + 1
    new = [_adam64(params[k], grads[k], st[k], st[3 + k], lr[k], step) for k in range(3)]
    out = {"params": [x[0] for x in new], "moments": [x[1] for x in new] + [x[2] for x in new],
           "loss": loss}
    if kind == "split":
        out["grads"] = grads
    else:
        out["step"] = None
    return out
