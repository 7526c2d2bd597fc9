"""A small plan in every layout: the default's eight threads per candidate beside
one, two and four, over formats, FP64 cost, a costmap, odd numbers of Euler
steps, candidates that reach the goal and degenerate starts.  Every output the
same bits (a NaN equal to a NaN)."""
import numpy as np
import pytest

import gen
from test_gpu_layouts import ctx, dev, plan, same          # noqa: F401  (ctx is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 15, 17, 900])
@pytest.mark.parametrize("fmt,acc64,n_sub,costmap", [(0, 0, 3, True), (0, 1, 4, False), (1, 0, 1, True), (1, 1, 5, False)])
def test_every_layout(ctx, N, fmt, acc64, n_sub, costmap):          # noqa: F811
    w = gen.workload_plain(0, N=N, H=40)
    w.n_sub = n_sub
    w.cost = gen.cost_default(17.0, 25.6)
    s = np.repeat(w.x0[None, :], N, 0)
    s[:, 6] = (2.0 + 10.0 * gen.uniform(3, 5, N)).astype(np.float32)
    bad = [(3, -2.4e5), (4, 1.4e5), (5, 3e6), (12, 5e5), (0, -3.0), (1, 60.0), (0, 1e20), (9, 1e6), (2, np.nan),
           (6, np.inf), (4, np.nan), (1, np.nan)]
    for i, (q, v) in enumerate(bad):
        if 3 + 5 * i < N:
            s[3 + 5 * i, q] = v
    cm = dev(gen.uniform(4, 6, 256 * 256).reshape(256, 256).astype(np.float32) * 50.0) if costmap else None
    x0 = dev(s.T.copy())
    one = plan(ctx, w, x0, 1, fmt, acc64, cm)
    assert N < 900 or 0 < np.sum((one["flags"] & 2) != 0) < N
    for lanes in (0, 2, 4):
        same(plan(ctx, w, x0, lanes, fmt, acc64, cm), one)
