"""costmap() on a stream that is being captured while another one is current:
the launches go into the graph, so the vertices they read have to live as long
as its replays do, whatever the allocator hands out in between."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_captured_launches_keep_their_vertices():
    from paper_2603_20525_gb300 import atp
    ctx = atp.Context(0)
    box = np.array([[1.0, 1.0], [2.0, 1.0], [2.0, 2.0], [1.0, 2.0]])
    polys = [(box, 0), (box + 0.7, 0)]
    want = ctx.costmap(polys, 40, 40, 0.1)
    torch.cuda.synchronize()
    s, o, g = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
        with torch.cuda.stream(o):
            cm = ctx.costmap(polys, 40, 40, 0.1, stream=s)
    # blocks of the vertices' size, on every stream a freed one could go back to
    for q in (o, s, torch.cuda.default_stream()):
        with torch.cuda.stream(q):
            junk = [torch.full((16,), 1.5, dtype=torch.float64, device="cuda") for _ in range(64)]
    torch.cuda.synchronize()
    other = ctx.costmap([(box + 0.3, 0)], 40, 40, 0.1)
    for _ in range(2):
        cm.zero_()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(cm, want) and not torch.equal(cm, other)
    del junk, g
    ctx.close()
