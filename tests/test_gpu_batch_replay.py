"""Both forms of the batched build under CUDA-graph replay, with other points in the same buffers before each replay: a
work queue, a counter or a look-back word left from the capture or an earlier replay would show."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2601_05347_gb300 import gen  # noqa: E402

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_05347_gb300 import psi

SIZES = [0, 1, 33, 70001, 4097, 0, 12345, 40]


@pytest.mark.parametrize("threads", [0, 512])
def test_replays_with_other_points(threads):
    off = np.concatenate([[0], np.cumsum(SIZES)])
    n, nq, k = int(off[-1]), 3000, 10
    sets = [torch.from_numpy(p).to("cuda") for p in (gen.varden(n, 2, 30, 1), gen.varden(n, 2, 30, 2),
                                                     gen.uniform(n, 2, 30, 3))]
    pts, ids = sets[0].clone(), torch.arange(n, dtype=torch.int32, device="cuda")
    q = torch.empty((nq, 2), dtype=torch.int32, device="cuda")
    qoff = torch.linspace(0, nq, len(SIZES) + 1, device="cuda").long()
    at = torch.randint(0, n, (nq,), device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    oi = torch.empty((nq, k), dtype=torch.int32, device="cuda")
    od = torch.empty((nq, k), dtype=torch.int64, device="cuda")
    b = psi.Batch(off, dim=2, kind="spac_h", threads=threads)
    b.reserve(nq)
    q.copy_(pts[at])
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        n0 = psi.launch_count()
        b.build(pts, ids)
        launches = psi.launch_count() - n0
        b.knn(q, qoff, k, oi, od)
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda.synchronize()
    assert (launches == 1) == (threads == 512)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        b.build(pts, ids)
        b.knn(q, qoff, k, oi, od)
    fresh = psi.Batch(off, dim=2, kind="spac_h", threads=512 - threads)  # the other form, outside a graph
    for s in (1, 2, 0):
        pts.copy_(sets[s])
        q.copy_(pts[at])
        g.replay()
        fresh.build(pts, ids)
        wi, wd = fresh.knn(q, qoff, k)
        torch.cuda.synchronize()
        b.sync()
        fresh.sync()
        assert torch.equal(oi, wi) and torch.equal(od, wd)
        for i in range(len(SIZES)):
            x, y = b.leaves(i), fresh.leaves(i)
            assert all(torch.equal(x[f], y[f]) for f in x)
