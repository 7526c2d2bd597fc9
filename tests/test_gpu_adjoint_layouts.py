"""The adjoint's layouts: one candidate per CTA or two per warp, odd counts, a
trace kept whole or recomputed in segments from checkpoints, candidates that
reach the goal at different steps, and rollouts that diverge.  The same
candidates must give the same bits in each (a NaN equal to a NaN)."""
import numpy as np
import pytest
import torch

import gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2603_20525_gb300 import atp
    c = atp.Context(0)
    yield c
    c.close()


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


# 8192 x 220 x 10 steps of 64 bytes are above the 1 GiB of a whole trace
@pytest.mark.parametrize("objective", ["cost", "margin"])
@pytest.mark.parametrize("ckpt", [10, 300])
def test_counts_and_segments(ctx, objective, ckpt):
    w = gen.workload_plain(0, N=64, H=220, dt=0.02)
    w.n_sub = 10
    cost = gen.cost_default(14.0, 25.6)
    s = np.repeat(w.x0[None, :], 64, 0)
    s[:, 6] = (0.5 + 8.5 * gen.uniform(1, 2, 64)).astype(np.float32)
    s[5, 9] = 1e9                       # tumbles off
    s[6, 6] = np.nan
    ter = ctx.terrain_prepare(dev(w.terrain.heights), w.terrain.cell)

    def grad(idx):
        J, G = ctx.grad(w.vehicle, cost, ter, dev(s[idx].T.copy()), dev(w.ctrl[:, idx]), w.dt, w.n_sub, ckpt,
                        objective=objective)
        torch.cuda.synchronize()
        return J.cpu().numpy(), G.cpu().numpy()

    J, G = grad(np.arange(64))
    good = np.setdiff1d(np.arange(64), [5, 6])
    assert np.all(np.isfinite(J[good])) and np.all(np.isfinite(G[:, good]))
    done = np.all(G[-1, good] == 0.0, axis=1)
    assert objective == "margin" or (0 < done.sum() < done.size)
    for n in (1, 63, 304, 305, 8192):
        idx = np.arange(n) % 64
        Jn, Gn = grad(idx)
        assert np.array_equal(Jn, J[idx], equal_nan=True)
        assert np.array_equal(Gn, G[:, idx], equal_nan=True)
