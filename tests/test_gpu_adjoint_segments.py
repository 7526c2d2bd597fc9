"""The adjoint in several segments against the whole trace: the same candidates
give the same bits in every layout of the forward pass and both of the backward
one, with middle segments, a ragged last one, candidates that reach the goal and
rollouts that diverge."""
import numpy as np
import pytest
import torch

import gen

pytestmark = pytest.mark.gpu

N_SUB, BASE = 20, 40


@pytest.fixture(scope="module")
def ctx():
    from paper_2603_20525_gb300 import atp
    c = atp.Context(0)
    yield c
    c.close()


# eight, four and two threads per candidate forwards; backwards one candidate
# per CTA up to 304, two per warp above.  The traces of the first two are above
# 128 MiB by their length.  `ckpt` = 2 takes 4 to 8 segments, 7 takes 2 to 17, the
# whole horizon one.
@pytest.mark.parametrize("objective", ["cost", "margin"])
@pytest.mark.parametrize("K,H", [(40, 2701), (305, 449), (5000, 101), (16385, 101)])
def test_segments_same_bits(ctx, K, H, objective):
    w = gen.workload_plain(0, N=BASE, H=H, dt=0.02)
    s = np.repeat(w.x0[None, :], BASE, 0)
    s[:, 6] = (0.5 + 8.5 * gen.uniform(1, 2, BASE)).astype(np.float32)
    s[5, 9], s[6, 6] = 1e9, np.nan
    ter = ctx.terrain_prepare(torch.as_tensor(w.terrain.heights).cuda(), w.terrain.cell)
    i = np.arange(K) % BASE
    x0 = torch.as_tensor(s[i].T.copy()).cuda()
    ctrl = torch.as_tensor(np.ascontiguousarray(w.ctrl[:, i])).cuda()
    r = {}
    for ckpt in (H, 2, 7):
        J, G = ctx.grad(w.vehicle, gen.cost_default(14.0, 25.6), ter, x0, ctrl, w.dt, N_SUB, ckpt, objective=objective)
        torch.cuda.synchronize()
        r[ckpt] = J.cpu().numpy(), G.cpu().numpy()
    J, G = r[H]
    done = np.all(G[-1, :BASE] == 0.0, axis=1)
    assert objective == "margin" or 0 < done.sum() < BASE
    assert np.array_equal(J, J[i], equal_nan=True) and np.array_equal(G, G[:, i], equal_nan=True)
    for ckpt in (2, 7):
        assert np.array_equal(r[ckpt][0], J, equal_nan=True)
        assert np.array_equal(r[ckpt][1], G, equal_nan=True)
