"""The planner's work as its users call it: each case is one pass through the
public entry points (Context.plan, plan_batch, plan_est, sample, lod_smooth,
costmap, terrain_prepare, and the autograd functions and refinement), with the
inputs, the bytes and operations the pass cannot do without, and what plain
torch in 64 bits gives for the same inputs.

Terrains are made here, on the GPU, in 64 bits from the seed alone: sums of
plane waves with the amplitudes a 0.3 m (or, for the planar model, 1.5 m)
Gaussian level of detail leaves them, berms, ruts and side slopes.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2603_20525_gb300 import atp, autograd

DEV = "cuda"

BASE_VEH = dict(M=1000.0, Jxx=280.9, Jyy=692.1, Jzz=810.7, Lf=2.5 * 1.565 / 2.713, Lr=2.5 * 1.148 / 2.713,
                e=1.5, hR=0.6, kf=4.0e4, kr=4.0e4, bf=3.0e3, br=3.0e3, C=6.1, mu=0.6, delta_max=0.639,
                delta_rate_max=1.0, g=9.81)
MRZR_VEH = dict(M=969.0, Jxx=280.9, Jyy=692.1, Jzz=810.7, Lf=1.565, Lr=1.148, e=1.280, hR=0.671, kf=4.2e4,
                kr=5.8e4, bf=3.1e3, br=4.3e3, C=6.1, mu=0.6, delta_max=0.639, delta_rate_max=1.0, g=9.81)

# algorithmic additions, multiplications and divisions of one Euler step of
# each model (a fused multiply-add counts as two)
SRB_FLOPS, EST_FLOPS, GRAD_FLOPS = 623.0, 190.0, 2000.0


def listed():
    return [
        # a replanning tick of a short horizon: the smallest call, launch and
        # host time count
        dict(name="plan_tick_256x16", kind="plan", N=256, H=16, dt=0.02, map="plain", side=256, cell=0.2,
             speed=8.0, veh="base"),
        # one plan of one vehicle: 1024 candidates over 2 s
        dict(name="plan_plain_1024x40", kind="plan", N=1024, H=40, dt=0.05, map="plain", side=256, cell=0.2,
             speed=8.0, veh="base"),
        # the benchmark's plan: 16384 candidates, each with its own start speed
        dict(name="plan_scaled_16384x100", kind="plan", N=16384, H=100, dt=0.02, map="scaled", side=1024,
             cell=0.1, speed=10.0, veh="base", per_x0=True),
        # the paper's real-time configuration: uniform steering over 4 s
        dict(name="plan_paper_204288x16", kind="plan", N=204288, H=16, dt=0.25, map="scaled", side=1024,
             cell=0.1, speed=7.5, veh="mrzr", draws="uniform"),
        # a large map kept in BF16, with a costmap, FP64 cost accumulation, the
        # best candidate's margins and every final state; odd sizes
        dict(name="plan_bf16_4099x61", kind="plan", N=4099, H=61, dt=0.035, map="tile", side=1531, cell=0.1,
             speed=7.0, veh="mrzr", bf16=True, costmap=True, cost64=True, margins=True, xf=True),
        # one admission of the serving loop: six vehicles' requests, each
        # sampled about its warm start, planned in one launch
        dict(name="serve_batch_6", kind="batch", n=6, big=16384, h_lo=40, h_hi=100),
        # the planar model on the benchmark's sizes
        dict(name="est_scaled_16384x100", kind="est", N=16384, H=100, dt=0.02, map="scaled", side=1024, cell=0.1,
             speed=10.0, veh="base", per_x0=True),
        # cost and its gradient for the best 64 candidates of a plan, forward
        # and backward through autograd
        dict(name="grad_64x100", kind="grad", K=64, H=100, dt=0.02, objective="cost", ckpt=10),
        # the constraint's gradient for a whole candidate set
        dict(name="grad_margin_4096x30", kind="grad", K=4096, H=30, dt=0.05, objective="margin", ckpt=5),
        # ten iterations of gradient refinement of the best 64
        dict(name="refine_64x50", kind="refine", K=64, H=50, dt=0.02, iters=10),
        # a new map for both models: level of detail, costmap of obstacles and
        # path boundary, texels
        dict(name="map_update_2048", kind="map", nx=2048, ny=2048, cell=0.1, n_obs=24, planar=True),
        # the largest serving request's candidates
        dict(name="sample_32768x150", kind="sample", N=32768, H=150, warm=True),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plan", "plan", "plan", "batch", "est", "grad", "refine", "map", "sample"])
    if kind in ("plan", "est"):
        mp = rng.choice(["plain", "scaled", "tile"])
        dt = rng.choice([0.02, 0.03, 0.05, 0.1, 0.25])
        H = _logint(rng, 8, 150)
        ns = math.ceil(round(dt / 0.005, 9))
        H = max(4, min(H, 1000 // ns))
        c = dict(kind=kind, N=min(_logint(rng, 100, 200000), int(1.2e8 / (H * ns))), H=H, dt=dt, map=mp,
                 side={"plain": 256, "scaled": 1024}.get(mp) or rng.randint(512, 2048),
                 cell=0.2 if mp == "plain" else 0.1, speed=round(rng.uniform(5.0, 10.0), 2),
                 veh=rng.choice(["base", "mrzr"]), per_x0=rng.random() < 0.3, costmap=rng.random() < 0.4,
                 margins=rng.random() < 0.3)
        if kind == "plan":
            c.update(draws=rng.choice(["gauss", "gauss", "uniform"]), bf16=rng.random() < 0.25,
                     cost64=rng.random() < 0.2, xf=rng.random() < 0.5)
        return c
    if kind == "batch":
        return dict(kind="batch", n=rng.randint(1, 8), big=rng.choice([4096, 16384, 32768]),
                    h_lo=rng.randint(20, 60), h_hi=rng.randint(61, 150))
    if kind == "grad":
        return dict(kind="grad", K=_logint(rng, 8, 8192), H=rng.randint(10, 100), dt=rng.choice([0.02, 0.05]),
                    objective=rng.choice(["cost", "margin"]), ckpt=rng.choice([5, 7, 10, 20]))
    if kind == "refine":
        return dict(kind="refine", K=_logint(rng, 8, 1024), H=rng.randint(20, 100), dt=0.02, iters=rng.randint(3, 10))
    if kind == "map":
        return dict(kind="map", nx=_logint(rng, 200, 4096), ny=_logint(rng, 200, 4096),
                    cell=rng.choice([0.1, 0.2]), n_obs=_logint(rng, 1, 200), planar=rng.random() < 0.5,
                    bf16=rng.random() < 0.3, sdist=rng.random() < 0.2)
    return dict(kind="sample", N=_logint(rng, 200, 60000), H=rng.randint(10, 150), warm=rng.random() < 0.7)


# ---------------------------------------------------------------------------
# inputs

def _gen(seed, stream):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1000003 + stream) & 0x7FFFFFFF)


def _smooth(t):
    t = t.clamp(0.0, 1.0)
    return t * t * (3.0 - 2.0 * t)


def _waves(ny, nx, cell, amp, lod, rng):
    """Five octaves of plane waves from 12.8 m, each scaled as a Gaussian of
    `lod` metres leaves it; max |f| near amp."""
    x = cell * torch.arange(nx, device=DEV, dtype=torch.float64)[None, :]
    y = cell * torch.arange(ny, device=DEV, dtype=torch.float64)[:, None]
    f = torch.zeros((ny, nx), device=DEV, dtype=torch.float64)
    for o in range(5):
        lam = 12.8 / 2.0 ** o
        g = 0.5 ** o * math.exp(-2.0 * math.pi ** 2 * lod ** 2 / lam ** 2)
        for _ in range(8):
            a, p = 2.0 * math.pi * rng.random(), 2.0 * math.pi * rng.random()
            kx, ky = 2.0 * math.pi / lam * math.cos(a), 2.0 * math.pi / lam * math.sin(a)
            cx, sx = torch.cos(kx * x), torch.sin(kx * x)
            cy, sy = torch.cos(ky * y + p), torch.sin(ky * y + p)
            f += g * (cy * cx - sy * sx)
    return f * (amp / 8.0)


def _terrain(kind, ny, nx, cell, seed, lod=0.3):
    """float32 [ny, nx]: hills with two berms and a bank ("plain"), ruts and
    alternating side slopes ("scaled"), one berm and a bank ("tile"), or with
    unsmoothed detail ("raw", the input of a level of detail)."""
    rng = np.random.default_rng(int(seed) * 7 + 3)
    X = cell * torch.arange(nx, device=DEV, dtype=torch.float64)[None, :]
    Y = cell * torch.arange(ny, device=DEV, dtype=torch.float64)[:, None]
    yc = 0.5 * ny * cell
    amp = {"plain": 0.5, "scaled": 0.8, "tile": 0.6, "raw": 0.8}[kind]
    f = _waves(ny, nx, cell, amp, 0.0 if kind == "raw" else lod, rng)
    if kind == "plain":
        for xc, deg in ((9.0, 30.0), (13.0, -30.0)):
            s = (X - xc) * math.cos(math.radians(deg)) - (Y - yc) * math.sin(math.radians(deg))
            f += torch.where(s.abs() < 1.0, 0.16 * (1.0 + torch.cos(math.pi * s)), 0.0 * s)
        w = _smooth((X - 13.0) / 2.0) * _smooth((25.0 - X) / 2.0)
        f += w * math.tan(math.radians(15.0)) * (Y - yc)
    elif kind == "scaled":
        wander = 0.5 * torch.sin(2.0 * math.pi * X / 17.0)
        for off in (-0.75, 0.75):
            f -= 0.045 * torch.exp(-0.5 * ((Y - (yc + off + wander)) / (lod + 0.06)) ** 2)
        b = torch.round(X / 8.0)
        right = torch.where(torch.remainder(b, 2.0) == 0.0, 1.0, -1.0)
        s = -right + 2.0 * right * _smooth((X - 8.0 * b + 1.0) / 2.0)
        f += s * math.tan(math.radians(20.0)) * (Y - yc)
    else:
        s = X - nx * cell * (0.3 + 0.4 * rng.random()) - 0.3 * (Y - yc)
        f += torch.where(s.abs() < 1.0, 0.16 * (1.0 + torch.cos(math.pi * s)), 0.0 * s)
        f += 0.06 * (2.0 * rng.random() - 1.0) * (Y - yc)
    return f.to(torch.float32).contiguous()


def _polygons(nx, ny, cell, n, seed):
    """n convex obstacles over the middle of the map and the path boundary."""
    rng = np.random.default_rng(int(seed) * 11 + 5)
    ex, ey = (nx - 1) * cell, (ny - 1) * cell
    out = []
    for _ in range(n):
        k = int(rng.integers(5, 10))
        c = np.array([ex * rng.uniform(0.2, 0.8), ey * rng.uniform(0.3, 0.7)])
        r = rng.uniform(0.6, 1.5)
        a = rng.uniform(0, 2 * math.pi) + 2 * math.pi * (np.arange(k) + 0.3 * (rng.random(k) - 0.5)) / k
        out.append((np.stack([c[0] + r * np.cos(a), c[1] + r * np.sin(a)], 1), 0))
    m = min(4.0, 0.2 * ex, 0.2 * ey)
    out.append((np.array([[m, m], [ex - m, m], [ex - m, ey - m], [m, ey - m]]), 1))
    return out


def _costmap64(polys, nx, ny, cell, eps=0.25, sigma=1e6):
    """(costmap, smallest signed distance) in 64 bits."""
    px = cell * torch.arange(nx, device=DEV, dtype=torch.float64)[None, :]
    py = cell * torch.arange(ny, device=DEV, dtype=torch.float64)[:, None]
    c = torch.zeros((ny, nx), device=DEV, dtype=torch.float64)
    smin = torch.full_like(c, math.inf)
    for v, kind in polys:
        d2 = torch.full_like(c, math.inf)
        inside = torch.zeros((ny, nx), device=DEV, dtype=torch.bool)
        for a, b in zip(v, np.roll(v, -1, axis=0)):
            (ax, ay), (bx, by) = map(float, a), map(float, b)
            ex, ey = bx - ax, by - ay
            l2 = ex * ex + ey * ey
            u = (((px - ax) * ex + (py - ay) * ey) / l2).clamp(0.0, 1.0)
            d2 = torch.minimum(d2, (px - (ax + u * ex)) ** 2 + (py - (ay + u * ey)) ** 2)
            if ay != by:
                cross = ((ay > py) != (by > py)) & (px < ax + (py - ay) / (by - ay) * ex)
                inside ^= cross
        s = torch.where(inside if kind == 0 else ~inside, -d2.sqrt(), d2.sqrt())
        c += sigma * (1.0 - s / eps).clamp(min=0.0) ** 2
        smin = torch.minimum(smin, s)
    return c, smin


def _settled(h, cell, veh, x, y, psi, vx):
    """The chassis on the least-squares plane through the nodes under its
    wheels, heading psi, CoM at h+R above it: 13 floats."""
    ny, nx = h.shape
    cps, sps = math.cos(psi), math.sin(psi)
    pts = []
    for lx in (veh["Lf"], -veh["Lr"]):
        for ly in (0.5 * veh["e"], -0.5 * veh["e"]):
            i = min(max(int(round((x + cps * lx - sps * ly) / cell)), 0), nx - 1)
            j = min(max(int(round((y + sps * lx + cps * ly) / cell)), 0), ny - 1)
            pts.append((i, j))
    ii, jj = torch.tensor([p[0] for p in pts]), torch.tensor([p[1] for p in pts])
    z = h[jj.to(h.device), ii.to(h.device)].double().cpu().numpy()
    P = np.array(pts, np.float64) * cell
    (a, b, c), *_ = np.linalg.lstsq(np.stack([np.ones(4), P[:, 0], P[:, 1]], 1), z, rcond=None)
    n = np.array([-b, -c, 1.0])
    n /= np.linalg.norm(n)
    hx = np.array([cps, sps, 0.0])
    bx = hx - (hx @ n) * n
    bx /= np.linalg.norm(bx)
    by = np.cross(n, bx)
    s = np.zeros(13)
    s[:3] = x, y, a + b * (x - veh["hR"] * n[0]) + c * (y - veh["hR"] * n[1]) + veh["hR"] * n[2]
    s[3:7] = math.atan2(bx[1], bx[0]), -math.asin(bx[2]), math.atan2(by[2], n[2]), vx
    return [float(np.float32(v)) for v in s]


def _cost(gx, gy):
    return dict(wt=5.0, wc=8.0, wg=15.0, sigma=1.0e6, eps_esm=0.0, goal_x=gx, goal_y=gy, goal_r=2.5)


def _controls(N, H, seed, uniform=False):
    g = _gen(seed, 21)
    if uniform:      # steering over its admissible set, no acceleration
        u = torch.zeros((H, N, 2), device=DEV)
        u[..., 0] = 2.0 * torch.rand((H, N), device=DEV, generator=g) - 1.0
    else:
        u = torch.randn((H, N, 2), device=DEV, generator=g) * torch.tensor([0.2, 0.3], device=DEV)
    u[:, 0] = 0.0
    return u


def _n_sub(dt):
    return math.ceil(round(dt / 0.005, 9))


def _problem(c, seed, planar=False):
    """Everything of one vehicle's plan but the library's own objects."""
    veh = BASE_VEH if c.get("veh", "base") == "base" else MRZR_VEH
    side, cell = c.get("side", 256), c.get("cell", 0.2)
    h = _terrain(c.get("map", "plain"), side, side, cell, seed, 1.5 if planar else 0.3)
    ext = side * cell
    x, y = (5.0 if c.get("map", "plain") == "plain" else 0.1 * ext), 0.5 * ext
    x0 = _settled(h, cell, veh, x, y, 0.0, c.get("speed", 8.0))
    if planar:
        x0 = [x0[q] for q in (0, 1, 3, 7, 11, 12, 6)]
    cm = None
    if c.get("costmap"):
        cm = _costmap64(_polygons(side, side, cell, 4, seed), side, side, cell, sigma=1e3)[0].float()
    N, H = c.get("N") or c["K"], c["H"]
    if c.get("per_x0"):
        q = 6
        s = torch.tensor(x0, device=DEV)[:, None].repeat(1, N)
        s[q] = 5.0 + 10.0 * torch.rand(N, device=DEV, generator=_gen(seed, 31))
        x0 = s.contiguous()
    return dict(veh=veh, cost=_cost(x + min(40.0, 0.85 * ext), y), h=h, cell=cell, cm=cm, x0=x0, dt=c["dt"],
                n_sub=_n_sub(c["dt"]), ctrl=_controls(N, H, seed, c.get("draws") == "uniform"))


def _request(c, i, seed):
    """Request i of a serving batch: sizes, horizon and interval."""
    rng = np.random.default_rng(int(c["n"]) * 977 + i)     # sizes belong to the case, not to the seed
    N = int(min(rng.choice([1024, 4096, 16384, 32768]), c["big"]))
    return N, int(rng.integers(c["h_lo"], c["h_hi"] + 1)), float(0.005 * rng.integers(4, 11))


# ---------------------------------------------------------------------------

def prepare(case, seed):
    c, k = case, case["kind"]
    ctx = atp.Context(0)
    s = dict(case=c, ctx=ctx)
    if k in ("plan", "est", "grad", "refine"):
        p = _problem(c, seed, planar=k == "est")
        s.update(p, ter=ctx.terrain_prepare(p["h"], p["cell"], costmap=p["cm"],
                                            fmt=atp.BF16X4 if c.get("bf16") else atp.F32X4))
        if c.get("cost64"):
            ctx.set_option(atp.OPT_COST_FP64, 1)
        if k in ("plan", "est"):
            ctx.reserve(c["N"], c["H"])
            # the planner's own output buffers, kept from plan to plan
            o = atp.plan_outputs(c["N"], c["H"], candidates=True, xf=k == "plan" and bool(c.get("xf")))
            if not c.get("margins"):
                del o["best_margin"]
            s["out"] = o
        if k == "grad":
            s["ctrl"].requires_grad_(True)
    elif k == "batch":
        ctx.reserve(sum(_request(c, i, seed)[0] for i in range(c["n"])), c["h_hi"])
        rng = np.random.default_rng(int(seed) * 13 + 1)
        reqs, pre = [], []
        for i in range(c["n"]):
            N, H, dt = _request(c, i, seed)
            side = [512, 768, 1024][i % 3]
            veh = BASE_VEH if i % 2 == 0 else MRZR_VEH
            h = _terrain("tile", side, side, 0.1, int(seed) * 100 + i)
            psi, m = math.pi * (2.0 * rng.random() - 1.0), 0.05 * side
            x0 = _settled(h, 0.1, veh, m, m, psi, 5.0 + 5.0 * rng.random())
            prev = torch.randn((H, 2), device=DEV, generator=_gen(seed, 50 + i)) * 0.1
            ctrl = torch.empty((H, N, 2), device=DEV)
            out = atp.plan_outputs(N, H, candidates=False)
            del out["best_margin"]
            reqs.append(dict(veh=veh, cost=_cost(m + 40.0 * math.cos(psi), m + 40.0 * math.sin(psi)),
                             terrain=ctx.terrain_prepare(h, 0.1), x0=x0, ctrl=ctrl, dt=dt, n_sub=0, out=out))
            pre.append((N, H, (int(seed) + 1, i + 1), prev))
        s.update(reqs=reqs, pre=pre, nonce=int(seed))
    elif k == "map":
        s.update(h=_terrain("raw", c["ny"], c["nx"], c["cell"], seed),
                 polys=_polygons(c["nx"], c["ny"], c["cell"], c["n_obs"], seed))
    else:
        N, H = c["N"], c["H"]
        s.update(prev=torch.randn((H, 2), device=DEV, generator=_gen(seed, 51)) * 0.1 if c["warm"] else None,
                 out=torch.empty((H, N, 2), device=DEV), key=(int(seed) + 1, 7), nonce=int(seed))
    return s


def _result(o):
    """The fields of a plan's result and its arrays."""
    w = o["out"]
    r = dict(best_idx=w[0:1], n_feasible=w[1:2], best_cost=w[2:3].view(torch.float32),
             best_min_margin=w[3:4].view(torch.float32), best_min_step=w[4:5])
    r.update({q: o[q] for q in o if q != "out"})
    return r


def run(state):
    s, c, k = state, state["case"], state["case"]["kind"]
    ctx = s["ctx"]
    if k == "plan":
        return _result(ctx.plan(s["veh"], s["cost"], s["ter"], s["x0"], s["ctrl"], s["dt"], s["n_sub"], out=s["out"]))
    if k == "est":
        return _result(ctx.plan_est(s["veh"], s["cost"], s["ter"], s["x0"], s["ctrl"], s["dt"], s["n_sub"],
                                    out=s["out"]))
    if k == "batch":
        for (N, H, key, prev), q in zip(s["pre"], s["reqs"]):
            ctx.sample(N, H, 0.2, 0.3, key, s["nonce"], prev=prev, out=q["ctrl"])
        return [dict(_result(o), ctrl=q["ctrl"]) for o, q in zip(ctx.plan_batch(s["reqs"]), s["reqs"])]
    if k == "grad":
        f = autograd.RolloutCost if c["objective"] == "cost" else autograd.RolloutMargin
        J = f.apply(s["ctrl"], ctx, s["veh"], s["cost"], s["ter"], s["x0"], s["dt"], s["n_sub"], c["ckpt"])
        (g,) = torch.autograd.grad(J.sum(), s["ctrl"])
        return dict(J=J.detach(), grad=g)
    if k == "refine":
        u, hist = autograd.refine(ctx, s["veh"], s["cost"], s["ter"], s["x0"], s["ctrl"], s["dt"], s["n_sub"],
                                  iters=c["iters"])
        return dict(ctrl=u, hist=hist)
    if k == "map":
        nx, ny, cell = c["nx"], c["ny"], c["cell"]
        r = {}
        cm = ctx.costmap(s["polys"], nx, ny, cell, want_sdist=bool(c.get("sdist")))
        if c.get("sdist"):
            cm, r["sdist"] = cm
        r["costmap"] = cm
        for name, sigma in (("srb", 0.3), ("planar", 1.5)):
            if name == "planar" and not c["planar"]:
                continue
            h = ctx.lod_smooth(s["h"], cell, sigma)
            t = ctx.terrain_prepare(h, cell, costmap=cm, fmt=atp.BF16X4 if c.get("bf16") else atp.F32X4).texels
            r[name] = h
            if c.get("bf16"):      # packed words: the nodes, then the block planes (between them, padding)
                n, at = nx * ny * 2, (nx * ny * 8 + 255) // 256 * 64
                r[name + "_nodes"], r[name + "_planes"] = t[:n].view(torch.int32), t[at:].view(torch.int32)
            else:
                r[name + "_texels"] = t
        return r
    return ctx.sample(c["N"], c["H"], 0.2, 0.3, s["key"], s["nonce"], prev=s["prev"], out=s["out"])


def work(case):
    c, k = case, case["kind"]
    if k in ("plan", "est", "grad", "refine"):
        N, H = c.get("N") or c["K"], c["H"]
        steps = N * H * _n_sub(c["dt"])
        b = 8.0 * N * H                                   # controls read
        if c.get("per_x0"):
            b += 4.0 * N * (7 if k == "est" else 13)
        if k in ("plan", "est"):
            b += 9.0 * N + (52.0 * N if c.get("xf") else 0.0)
            return dict(bytes=b, flops=steps * (EST_FLOPS if k == "est" else SRB_FLOPS))
        if k == "grad":                                   # the forward step, then its adjoint
            return dict(bytes=2 * b + 4.0 * N, flops=steps * (SRB_FLOPS + GRAD_FLOPS))
        it = c["iters"]
        return dict(bytes=2 * b + 4.0 * N * (it + 1), flops=steps * (it + 1) * (SRB_FLOPS + GRAD_FLOPS))
    if k == "batch":
        b = f = 0.0
        for i in range(c["n"]):
            N, H, dt = _request(c, i, 0)
            b += 8.0 * N * H
            f += N * H * (_n_sub(dt) * SRB_FLOPS + 60.0)
        return dict(bytes=b, flops=f)
    if k == "map":
        n = c["nx"] * c["ny"]
        maps = 2 if c["planar"] else 1
        taps = sum(2 * int(4 * sg / c["cell"] + 0.5) + 1 for sg in (0.3, 1.5)[:maps])
        tex = 8.25 if c.get("bf16") else 16.0
        return dict(bytes=n * (4.0 + 4.0 * (2 if c.get("sdist") else 1) + maps * (4.0 + tex)), flops=n * (4.0 * taps + 100.0))
    return dict(bytes=8.0 * c["N"] * c["H"] + 8.0 * c["H"], flops=60.0 * c["N"] * c["H"])


# ---------------------------------------------------------------------------
# the same in 64 bits, plain torch

class _Map64:
    def __init__(self, h, cell, cm):
        f = h.double()
        gx, gy = torch.empty_like(f), torch.empty_like(f)
        gx[:, 1:-1] = (f[:, 2:] - f[:, :-2]) / (2 * cell)
        gx[:, 0], gx[:, -1] = (f[:, 1] - f[:, 0]) / cell, (f[:, -1] - f[:, -2]) / cell
        gy[1:-1] = (f[2:] - f[:-2]) / (2 * cell)
        gy[0], gy[-1] = (f[1] - f[0]) / cell, (f[-1] - f[-2]) / cell
        z = torch.zeros_like(f) if cm is None else cm.double()
        self.cell, self.ny, self.nx = cell, f.shape[0], f.shape[1]
        self.t = torch.stack([f, gx, gy, z], -1).reshape(-1, 4)

    def at(self, x, y):
        u, w = (x / self.cell).clamp(0, self.nx - 1), (y / self.cell).clamp(0, self.ny - 1)
        i, j = u.detach().floor().clamp(max=self.nx - 2), w.detach().floor().clamp(max=self.ny - 2)
        a, b = (u - i)[..., None], (w - j)[..., None]
        o = (j * self.nx + i).long()
        lo = self.t[o] * (1 - a) + self.t[o + 1] * a
        hi = self.t[o + self.nx] * (1 - a) + self.t[o + self.nx + 1] * a
        return (lo * (1 - b) + hi * b).unbind(-1)


def _srb64(p, ctrl):
    """J, min U_ESM and final state [13, N] of every candidate."""
    v, c = p["veh"], p["cost"]
    m = _Map64(p["h"], p["cell"], p["cm"])
    N = ctrl.shape[1]
    d64 = dict(dtype=torch.float64, device=DEV)
    x0 = p["x0"].double() if isinstance(p["x0"], torch.Tensor) else torch.tensor(p["x0"], **d64)[:, None].expand(13, N)
    x, y, z, psi, th, ph, vx, vy, vz, wx, wy, wz, dl = x0.unbind(0)
    L = v["Lf"] + v["Lr"]
    col = lambda a: torch.tensor(a, **d64)[:, None]
    rx, ry = col([v["Lf"], v["Lf"], -v["Lr"], -v["Lr"]]), col([0.5 * v["e"], -0.5 * v["e"]] * 2)
    kk, bb = col([v["kf"]] * 2 + [v["kr"]] * 2), col([v["bf"]] * 2 + [v["br"]] * 2)
    Fs = col([0.5 * v["g"] * v["M"] * v["Lr"] / L] * 2 + [0.5 * v["g"] * v["M"] * v["Lf"] / L] * 2)
    fr = col([1.0, 1.0, 0.0, 0.0])
    hR, g, M = v["hR"], v["g"], v["M"]
    Rb, pb = math.hypot(hR, 0.5 * v["e"]), math.atan(2 * hR / v["e"])
    eps = c["eps_esm"] or 0.1 * M * g * Rb * (1 - math.sin(pb))
    h = float(np.float32(p["dt"])) / p["n_sub"]
    sgn = torch.tensor(1.0, **d64)

    def esm(th, ph):
        a = ph.abs() + pb
        return torch.where(a < 0.5 * math.pi, sgn, -sgn) * M * g * Rb * (1 - torch.sin(a)) * torch.cos(th)

    J = torch.zeros(N, **d64)
    margin = torch.full((N,), math.inf, **d64)
    done = torch.zeros(N, dtype=torch.bool, device=DEV)
    r2 = c["goal_r"] ** 2
    for k in range(ctrl.shape[0]):
        dd, ax = ctrl[k, :, 0].clamp(-v["delta_rate_max"], v["delta_rate_max"]), ctrl[k, :, 1]
        for _ in range(p["n_sub"]):
            U = esm(th, ph)
            margin = torch.where(U < margin, U, margin)
            done = done | ((x - c["goal_x"]) ** 2 + (y - c["goal_y"]) ** 2 <= r2)
            go = ~done
            cps, sps, cth, sth, cph, sph = psi.cos(), psi.sin(), th.cos(), th.sin(), ph.cos(), ph.sin()
            R = (cps * cth, cps * sph * sth - cph * sps, sph * sps + cph * cps * sth,
                 cth * sps, cph * cps + sph * sps * sth, cph * sps * sth - cps * sph, -sth, cth * sph, cph * cth)
            ox, oy, oz = (rx * R[3 * q] + ry * R[3 * q + 1] - hR * R[3 * q + 2] for q in range(3))
            f, fx, fy, cm = m.at(x + ox, y + oy)
            tx, ty, tz = (R[6 + q] - fx * R[q] - fy * R[3 + q] for q in range(3))
            chi = (z + oz - f) / tz
            vix, viy, viz = vx - wz * ry - wy * hR, vy + wz * rx + wx * hR, vz + wx * ry - wy * rx
            chid = (tx * (vix - chi * wy) + ty * (viy + chi * wx) + tz * viz) / tz
            Fk = (Fs - kk * chi).clamp(min=0)
            Fz = torch.where(Fk > 0, (Fk - bb * chid).clamp(min=0), 0 * Fk)
            Ca = v["C"] * (torch.atan2(viy, vix) - fr * dl)
            Fy = -Fz * Ca * v["mu"] / (v["mu"] ** 2 + Ca * Ca).sqrt() * (1 + fr * (dl.cos() - 1))
            gx, gy, gz = -g * R[6], -g * R[7], -g * R[8]
            FyB, FzB = Fy.sum(0), Fz.sum(0)
            Fx = 0.5 * M * (ax - gx + wy * vz - wz * vy)
            Mx = hR * FyB + (ry * Fz).sum(0)
            My = -(rx * Fz).sum(0) - 2 * hR * Fx
            Mz = (rx * Fy).sum(0)
            soft = (1 - U / eps).clamp(min=0)
            Lr = c["wt"] + c["wc"] * dd * dd + c["sigma"] * soft * soft + cm.sum(0)
            J = torch.where(go, J + h * Lr, J)
            wsc = sph * wy + cph * wz
            new = (x + h * (R[0] * vx + R[1] * vy + R[2] * vz), y + h * (R[3] * vx + R[4] * vy + R[5] * vz),
                   z + h * (R[6] * vx + R[7] * vy + R[8] * vz), psi + h * wsc / cth, th + h * (cph * wy - sph * wz),
                   ph + h * (wx + wsc * sth / cth), vx + h * ax, vy + h * (gy + FyB / M + wx * vz - wz * vx),
                   vz + h * (gz + FzB / M + wy * vx - wx * vy), wx + h * ((v["Jyy"] - v["Jzz"]) * wy * wz + Mx) / v["Jxx"],
                   wy + h * (-(v["Jxx"] - v["Jzz"]) * wx * wz + My) / v["Jyy"],
                   wz + h * ((v["Jxx"] - v["Jyy"]) * wx * wy + Mz) / v["Jzz"],
                   (dl + h * dd).clamp(-v["delta_max"], v["delta_max"]))
            x, y, z, psi, th, ph, vx, vy, vz, wx, wy, wz, dl = (
                torch.where(go, n, o) for n, o in zip(new, (x, y, z, psi, th, ph, vx, vy, vz, wx, wy, wz, dl)))
    U = esm(th, ph)
    margin = torch.where(U < margin, U, margin)
    J = J + c["wg"] * ((x - c["goal_x"]) ** 2 + (y - c["goal_y"]) ** 2).sqrt()
    return J, margin, torch.stack([x, y, z, psi, th, ph, vx, vy, vz, wx, wy, wz, dl])


def _est64(p, ctrl):
    """J, minimum lateral-acceleration margin and final state [7, N]."""
    v, c = p["veh"], p["cost"]
    m = _Map64(p["h"], p["cell"], p["cm"])
    N = ctrl.shape[1]
    d64 = dict(dtype=torch.float64, device=DEV)
    x0 = p["x0"].double() if isinstance(p["x0"], torch.Tensor) else torch.tensor(p["x0"], **d64)[:, None].expand(7, N)
    x, y, psi, vy, wz, dl, vx = x0.unbind(0)
    L, hR, g, M = v["Lf"] + v["Lr"], v["hR"], v["g"], v["M"]
    Kf, Kr, Kx, abar = M * v["Lr"] / L, M * v["Lf"] / L, M * hR / L, g * v["e"] / (2 * hR)
    eps = c["eps_esm"] or 0.1 * abar
    h = float(np.float32(p["dt"])) / p["n_sub"]
    J = torch.zeros(N, **d64)
    margin = torch.full((N,), math.inf, **d64)
    done = torch.zeros(N, dtype=torch.bool, device=DEV)

    def tire(Fz, a):
        Ca = v["C"] * a
        return -Fz * Ca * v["mu"] / (v["mu"] ** 2 + Ca * Ca).sqrt()

    for k in range(ctrl.shape[0]):
        dd, ax = ctrl[k, :, 0].clamp(-v["delta_rate_max"], v["delta_rate_max"]), ctrl[k, :, 1]
        for _ in range(p["n_sub"]):
            done = done | ((x - c["goal_x"]) ** 2 + (y - c["goal_y"]) ** 2 <= c["goal_r"] ** 2)
            go = ~done
            _, fx, fy, _ = m.at(x, y)
            rn = 1 / (1 + fx * fx + fy * fy).sqrt()
            sth, ty, tz = -fx * rn, -fy * rn, rn
            cth = (ty * ty + tz * tz).sqrt()
            sph, cph, sps, cps = -ty / cth, tz / cth, psi.sin(), psi.cos()
            R00, R01, R02 = cth * cps, -cth * sps, sth
            R10, R11, R12 = cps * sph * sth + cph * sps, cph * cps - sph * sth * sps, -cth * sph
            gy, gz = -g * (cph * sth * sps + cps * sph), -g * cph * cth
            aBx = ax - wz * vy
            Fyf = tire(-Kf * gz - Kx * aBx, torch.atan2(vy + wz * v["Lf"], vx) - dl)
            Fyr = tire(-Kr * gz + Kx * aBx, torch.atan2(vy - wz * v["Lr"], vx))
            dvy = gy + (Fyf + Fyr) / M - wz * vx
            mg = abar - (dvy + wz * vx - gy).abs()
            margin = torch.where(go & (mg < margin), mg, margin)
            cs = 0.0
            if p["cm"] is not None:
                for lx in (v["Lf"], -v["Lr"]):
                    for ly in (0.5 * v["e"], -0.5 * v["e"]):
                        cs = cs + m.at(x + R00 * lx + R01 * ly - R02 * hR, y + R10 * lx + R11 * ly - R12 * hR)[3]
            J = torch.where(go, J + h * (c["wt"] + c["wc"] * dd * dd + c["sigma"] * (1 - mg / eps).clamp(min=0) ** 2 + cs), J)
            new = (x + h * (R00 * vx + R01 * vy), y + h * (R10 * vx + R11 * vy), psi + h * wz, vy + h * dvy,
                   wz + h * (Fyf * v["Lf"] * dl.cos() - Fyr * v["Lr"]) / v["Jzz"],
                   (dl + h * dd).clamp(-v["delta_max"], v["delta_max"]), vx + h * ax)
            x, y, psi, vy, wz, dl, vx = (torch.where(go, n, o) for n, o in zip(new, (x, y, psi, vy, wz, dl, vx)))
    J = J + c["wg"] * ((x - c["goal_x"]) ** 2 + (y - c["goal_y"]) ** 2).sqrt()
    return J, margin, torch.stack([x, y, psi, vy, wz, dl, vx])


def _lod64(h, cell, sigma):
    s = sigma / cell
    r = int(4.0 * s + 0.5)
    w = torch.exp(-0.5 * (torch.arange(-r, r + 1, device=DEV, dtype=torch.float64) / s) ** 2)
    w = (w / w.sum()).tolist()
    f = h.double()
    for dim in (1, 0):
        n = f.shape[dim]
        at = torch.arange(n, device=DEV)
        f = sum(wk * f.index_select(dim, (at + q - r).clamp(0, n - 1)) for q, wk in enumerate(w))
    return f


def _pick(J, margin, feasible):
    """Cost and margin of the best candidate."""
    q = torch.where(feasible, J, math.inf) if bool(feasible.any()) else J
    b = int(torch.argmin(q))
    return J[b:b + 1], margin[b:b + 1]


def exact(case, seed):
    c, k = case, case["kind"]
    if k in ("plan", "est"):
        # a rollout that tumbles is not computable to any accuracy in 32 bits,
        # and a BF16 map is another map: only the gentler ones have a value
        mild = c["map"] == "plain" and c["dt"] * c["H"] <= 2.05 and c.get("draws") != "uniform"
        if k == "plan" and (not mild or c.get("bf16") or c["speed"] > 8.5 or c.get("per_x0") or c["veh"] != "base"):
            return None
        if c["N"] * c["H"] * _n_sub(c["dt"]) > 3e7:
            return None
        p = _problem(c, seed, planar=k == "est")
        with torch.no_grad():
            J, m, xf = (_est64 if k == "est" else _srb64)(p, p["ctrl"].double())
        bc, bm = _pick(J, m, m > 0)
        r = dict(best_idx=None, n_feasible=None, best_cost=bc, best_min_margin=bm, best_min_step=None,
                 best_ctrl=None, cost=J, margin=m, flags=None)
        if c.get("margins"):
            r["best_margin"] = None
        if k == "plan" and c.get("xf"):
            r["xf"] = xf
        return r
    if k == "grad":
        if c["K"] * c["H"] * _n_sub(c["dt"]) > 2e6 or c["dt"] * c["H"] > 2.05:
            return None
        p = _problem(c, seed)
        u = p["ctrl"].double().requires_grad_(True)
        J, m, _ = _srb64(p, u)
        out = J if c["objective"] == "cost" else m
        (g,) = torch.autograd.grad(out.sum(), u)
        # which of two nearly equal states holds the minimum is not decided in
        # 32 bits, so the margin's gradient has no such value
        return dict(J=out.detach(), grad=g if c["objective"] == "cost" else None)
    if k == "map":
        nx, ny, cell = c["nx"], c["ny"], c["cell"]
        polys = _polygons(nx, ny, cell, c["n_obs"], seed)
        if nx * ny * sum(len(v) for v, _ in polys) > 2e9:
            return None
        h = _terrain("raw", ny, nx, cell, seed)
        cm, sd = _costmap64(polys, nx, ny, cell)
        r = dict(costmap=cm, **(dict(sdist=sd) if c.get("sdist") else {}))
        for name, sigma in (("srb", 0.3), ("planar", 1.5)):
            if name == "planar" and not c["planar"]:
                continue
            f = _lod64(h, cell, sigma)
            r[name] = f
            if c.get("bf16"):
                r[name + "_nodes"] = r[name + "_planes"] = None
            else:
                r[name + "_texels"] = _Map64(f, cell, cm).t.reshape(-1)
        return r
    if k == "sample":
        N, H = c["N"], c["H"]
        nom = torch.zeros((H, 2), dtype=torch.float64)
        if c["warm"]:
            prev = (torch.randn((H, 2), device=DEV, generator=_gen(seed, 51)) * 0.1).double().cpu()
            nom = prev[torch.arange(1, H + 1).clamp(max=H - 1)]
        out = np.zeros((H, N, 2))
        for kq in range((H + 3) // 4):
            # numpy's Philox steps its counter before each block of four words
            ctr = int(seed) * 2 ** 128 + kq * 2 ** 64 - 1
            w = np.random.Philox(key=np.array([int(seed) + 1, 7], np.uint64),
                                 counter=ctr % 2 ** 256).random_raw(4 * N).reshape(N, 4)
            for q in range(4):
                if 4 * kq + q >= H:
                    break
                a, b = w[:, 2 * (q & 1)], w[:, 2 * (q & 1) + 1]
                sh = np.uint64(41 if q < 2 else 9)
                u1, u2 = ((((t >> sh) & np.uint64(0x7FFFFF)).astype(np.float64) + 0.5) / 8388608.0 for t in (a, b))
                r = np.sqrt(-2.0 * np.log(u1))
                out[4 * kq + q, :, 0] = float(np.float32(0.2)) * r * np.cos(2 * math.pi * u2)
                out[4 * kq + q, :, 1] = float(np.float32(0.3)) * r * np.sin(2 * math.pi * u2)
        out[:, 0] = 0.0
        return out + nom.numpy()[:, None, :]
    return None
