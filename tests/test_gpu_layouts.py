"""The two-warp layouts of a plan (geometry and forces in separate warps, one,
two or four lanes of each per candidate) against one thread per candidate,
which the parity tests hold to the oracle: every output the same bits (a NaN
equal to a NaN), where a layout can go wrong."""
import numpy as np
import pytest
import torch

import gen

pytestmark = pytest.mark.gpu

KEYS = ("cost", "margin", "flags", "xf", "best_ctrl", "best_margin", "out")


@pytest.fixture(scope="module")
def ctx():
    from paper_2603_20525_gb300 import atp
    c = atp.Context(0)
    yield c
    c.close()


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


def plan(ctx, w, x0, lanes, fmt=0, acc64=0, cm=None):
    from paper_2603_20525_gb300 import atp
    ctx.set_option(atp.OPT_LANES, lanes)
    ctx.set_option(atp.OPT_COST_FP64, acc64)
    try:
        t = w.terrain
        ter = ctx.terrain_prepare(dev(t.heights), t.cell, t.x0, t.y0, costmap=cm, fmt=fmt)
        o = ctx.plan(w.vehicle, w.cost, ter, x0, dev(w.ctrl), w.dt, w.n_sub, want_xf=True)
        torch.cuda.synchronize()
    finally:
        ctx.set_option(atp.OPT_LANES, 0)
        ctx.set_option(atp.OPT_COST_FP64, 0)
    return {k: o[k].cpu().numpy() for k in KEYS}


def same(a, b):
    for k in KEYS:
        assert np.array_equal(a[k], b[k], equal_nan=a[k].dtype.kind == "f"), k


# a pair of warps holds 8, 16 or 32 candidates: around those, and around the
# sizes at which the layout changes
@pytest.mark.parametrize("N", [1, 7, 9, 15, 17, 31, 33, 4864, 4865, 16384, 16385, 29184, 29185])
def test_sizes(ctx, N):
    w = gen.workload_plain(1, N=N, H=3 if N > 100 else 11)
    x0 = [float(v) for v in w.x0]
    one = plan(ctx, w, x0, 1)
    for lanes in (0, 2, 4):
        same(plan(ctx, w, x0, lanes), one)


@pytest.mark.parametrize("fmt,acc64,n_sub", [(0, 0, 3), (0, 1, 1), (1, 0, 4), (1, 1, 5)])
def test_goal_costmap_and_formats(ctx, fmt, acc64, n_sub):
    """Candidates that reach the goal at different steps, some warps whole,
    with an odd and an even number of Euler steps per control step."""
    w = gen.workload_plain(0, N=700, H=40)
    w.n_sub = n_sub
    w.cost = gen.cost_default(17.0, 25.6)
    s = np.repeat(w.x0[None, :], w.N, 0)
    s[:, 6] = np.where(np.arange(w.N) < 128, 9.0, 2.0 + 10.0 * gen.uniform(3, 5, w.N)).astype(np.float32)
    cm = dev(gen.uniform(4, 6, 256 * 256).reshape(256, 256).astype(np.float32) * 50.0)
    x0 = dev(s.T.copy())
    one = plan(ctx, w, x0, 1, fmt, acc64, cm)
    assert 0 < np.sum(one["flags"] & 2) and np.any((one["flags"] & 2) == 0)
    for lanes in (2, 4):
        same(plan(ctx, w, x0, lanes, fmt, acc64, cm), one)


def test_degenerate_starts(ctx):
    """Starts far off the map, with angles beyond the fast reduction's range,
    and non-finite in each component; NaN and infinite controls."""
    w = gen.workload_plain(2, N=96, H=6)
    s = np.repeat(w.x0[None, :], w.N, 0)
    for i, (q, v) in enumerate([(0, -3.0), (1, 60.0), (0, 1e7), (1, -1e7), (0, 9e8), (1, -9e8), (0, 1e20), (3, 4.0),
                                (3, -2.4e5), (4, 1.4e5), (5, 3e6), (12, 5e5), (6, 1e5), (9, 1e6), (11, -1e9)]):
        s[2 + i, q] = v
    for q in range(13):
        s[20 + q, q] = np.nan
        s[40 + q, q] = np.inf
        s[60 + q, q] = -np.inf
    w.ctrl[2, 80, 0], w.ctrl[3, 81, 1], w.ctrl[1, 82, 1] = np.nan, np.nan, np.inf
    x0 = dev(s.T.copy())
    one = plan(ctx, w, x0, 1)
    for lanes in (2, 4):
        same(plan(ctx, w, x0, lanes), one)


@pytest.mark.parametrize("acc64,n_sub,costmap", [(0, 4, False), (1, 3, True)])
def test_planar_plan(ctx, acc64, n_sub, costmap):
    """The planar plan's two-warp form (up to 48640 candidates) against one
    thread per candidate (more of them, the same ones repeated)."""
    from paper_2603_20525_gb300 import atp
    w = gen.workload_est(0, N=70, H=25)
    s = np.repeat(w.x0[None, :], 70, 0)
    s[:, 6] = (1.0 + 12.0 * gen.uniform(5, 6, 70)).astype(np.float32)
    for i, (q, v) in enumerate([(0, -5.0), (1, 1e9), (2, 3.0), (2, -1e7), (5, 2e5), (3, 1e20), (4, 1e6)]):
        s[3 + i, q] = v
    for q in range(7):
        s[20 + q, q], s[40 + q, q] = np.nan, np.inf
    cost = gen.cost_default(14.0, 25.6)
    cm = dev(gen.uniform(4, 6, 256 * 256).reshape(256, 256).astype(np.float32)) if costmap else None
    ter = ctx.terrain_prepare(dev(w.terrain.heights), w.terrain.cell, costmap=cm)
    ctx.set_option(atp.OPT_COST_FP64, acc64)
    try:
        r = {}
        for N in (1, 33, 70, 48640, 48641):
            i = np.arange(N) % 70
            o = ctx.plan_est(w.vehicle, cost, ter, dev(s[i].T.copy()), dev(w.ctrl[:, i]), w.dt, n_sub, want_xf=True)
            torch.cuda.synchronize()
            r[N] = {k: v.cpu().numpy() for k, v in o.items()}
    finally:
        ctx.set_option(atp.OPT_COST_FP64, 0)
    one = r[48641]
    assert 0 < np.sum(one["flags"][:70] & 2) // 2 < 70
    for N in (1, 33, 70, 48640):
        for k in ("cost", "margin", "flags", "xf"):
            assert np.array_equal(r[N][k], one[k][..., :N], equal_nan=k != "flags"), (N, k)
    for k in ("best_ctrl", "best_margin", "out"):
        a, b = r[70][k], r[48640][k]
        if k == "out":
            a, b = np.delete(a, 1), np.delete(b, 1)          # not the feasible count
        assert np.array_equal(a, b), k
