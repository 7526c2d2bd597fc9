"""The map kernels where their variants meet: level of detail on aligned and
misaligned maps (the same bits) and at the radii where the window changes and
ends, against the FP64 oracle; the costmap with more edges than are kept
between its kernels and with ragged, nested path boundaries, skipping against
full evaluation (the same bits); texels of odd maps on their borders."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

U = 2.0 ** -24


@pytest.fixture(scope="module")
def ctx():
    from paper_2603_20525_gb300 import atp
    c = atp.Context(0)
    yield c
    c.close()


def field(ny, nx, seed=0):
    return np.random.default_rng(seed).normal(0.0, 1.0, (ny, nx)).astype(np.float32)


# radius in cells: 0, the ends of the narrow window, the wide one, the largest
@pytest.mark.parametrize("r", [0, 1, 15, 16, 61, 512])
@pytest.mark.parametrize("ny,nx", [(1, 64), (131, 260), (66, 1030), (257, 33)])
def test_lod_alignment_and_radii(ctx, r, ny, nx):
    f = field(ny, nx, r)
    sigma = 0.0 if r == 0 else 0.1 * r / 4.0
    a = ctx.lod_smooth(torch.as_tensor(f).cuda(), 0.1, sigma)
    flat = torch.zeros(ny * nx + 1, dtype=torch.float32, device="cuda")
    flat[1:] = torch.as_tensor(f).cuda().reshape(-1)
    out = torch.zeros(ny * nx + 1, dtype=torch.float32, device="cuda")
    b = ctx.lod_smooth(flat[1:].view(ny, nx), 0.1, sigma, out=out[1:].view(ny, nx))
    torch.cuda.synchronize()
    assert torch.equal(a, b) and float(out[0]) == 0.0
    o = oracle.lod_smooth(f, 0.1, sigma)
    assert np.abs(a.cpu().numpy() - o).max() <= 2 * (2 * r + 4) * U * np.abs(f).max()


def test_lod_keeps_non_finite_values_within_the_radius(ctx):
    f = field(40, 72)
    f[20, 30], f[5, 60] = np.inf, np.nan
    for sigma, r in ((0.3, 12), (0.4, 16)):
        g = ctx.lod_smooth(torch.as_tensor(f).cuda(), 0.1, sigma).cpu().numpy()
        bad = np.zeros(f.shape, bool)
        for j, i in ((20, 30), (5, 60)):
            bad[max(0, j - r):j + r + 1, max(0, i - r):i + r + 1] = True
        assert np.array_equal(~np.isfinite(g), bad)


def star(cx, cy, r, n, wob):
    a = 2.0 * np.pi * np.arange(n) / n
    q = r * (1.0 + wob * np.sin(7.0 * a))
    return np.stack([cx + q * np.cos(a), cy + q * np.sin(a)], 1)


@pytest.mark.parametrize("n_edge", [40, 20000])
def test_costmap_boundaries_and_many_edges(ctx, n_edge):
    nx, ny, cell = 205, 163, 0.2
    polys = [(star(20.0, 16.0, 3.0, 9, 0.3), 0), (star(20.0, 16.0, 14.0, n_edge, 0.2), 1),
             (star(30.0, 10.0, 1.0, 5, 0.0), 0), (star(21.0, 17.0, 12.0, 11, 0.1), 1)]
    full, sd = ctx.costmap(polys, nx, ny, cell, want_sdist=True)
    skip = ctx.costmap(polys, nx, ny, cell)
    torch.cuda.synchronize()
    assert torch.equal(full, skip)
    _, so = oracle.costmap(polys, nx, ny, cell, 0.0, 0.0)
    assert np.abs(sd.cpu().numpy() - so).max() <= 16 * U * nx * cell
    assert 0.05 < np.mean(full.cpu().numpy() == 0.0) < 0.95


@pytest.mark.parametrize("ny,nx", [(3, 3), (33, 31), (9, 70), (64, 5)])
def test_texels_of_odd_maps(ctx, ny, nx):
    f, cm = field(ny, nx, 3), field(ny, nx, 4)
    t = ctx.terrain_prepare(torch.as_tensor(f).cuda(), 0.25, costmap=torch.as_tensor(cm).cuda()).texels
    t = t.cpu().numpy().reshape(ny, nx, 4)
    gx, gy = np.empty_like(f), np.empty_like(f)      # exact scales: cell is a power of two
    gx[:, 1:-1] = (f[:, 2:] - f[:, :-2]) * np.float32(2.0)
    gx[:, 0], gx[:, -1] = (f[:, 1] - f[:, 0]) * np.float32(4.0), (f[:, -1] - f[:, -2]) * np.float32(4.0)
    gy[1:-1] = (f[2:] - f[:-2]) * np.float32(2.0)
    gy[0], gy[-1] = (f[1] - f[0]) * np.float32(4.0), (f[-1] - f[-2]) * np.float32(4.0)
    assert np.array_equal(t, np.stack([f, gx, gy, cm], -1))


def test_costmap_refuses_a_capture(ctx):
    """The vertices' copy reads host memory that does not outlive the call, so
    a graph that held it would read whatever lies there at its replay: refused
    before anything is enqueued, with the context and the capture intact."""
    box = np.array([[1.0, 1.0], [2.0, 1.0], [2.0, 2.0], [1.0, 2.0]])
    want = ctx.costmap([(box, 0)], 40, 40, 0.1)
    one = torch.zeros(1, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        one += 1
        with pytest.raises(RuntimeError):
            ctx.costmap([(box, 0)], 40, 40, 0.1)
    g.replay()
    again = ctx.costmap([(box, 0)], 40, 40, 0.1)
    torch.cuda.synchronize()
    assert one.item() == 1
    assert torch.equal(again, want) and (want > 0).any()
