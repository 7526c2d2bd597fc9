"""Perimeters with a vertex at infinity, at NaN or very far off: their open or
endless outlines, and the rounding of their edges, change the inside test and
the distance far from every other edge, so the costmap with tiles left out has to be, bit for
bit, the one with every perimeter evaluated at every node (as it is when the
signed distances are wanted too)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf, 1e25, 3e8, -1e7])
@pytest.mark.parametrize("n", [40, 20000])            # edges kept between the kernels, or made on use
def test_unbounded_perimeters_are_never_left_out(kind, value, n):
    from paper_2603_20525_gb300 import atp
    ctx = atp.Context(0)
    a = 2.0 * np.pi * np.arange(n) / n
    ring = np.stack([20.0 + 14.0 * np.cos(a), 16.0 + 12.0 * np.sin(a)], 1)
    for vertex, axis in ((n // 8, 0), (n // 6, 1)):
        bad = ring.copy()
        bad[vertex, axis] = value
        polys = [(np.array([[8.0, 8.0], [10.0, 8.0], [10.0, 11.0], [8.0, 11.0]]), 0), (bad, kind)]
        full, _ = ctx.costmap(polys, 205, 163, 0.2, want_sdist=True)
        skip = ctx.costmap(polys, 205, 163, 0.2)
        torch.cuda.synchronize()
        assert np.array_equal(skip.cpu().numpy(), full.cpu().numpy(), equal_nan=True)
    ctx.close()
