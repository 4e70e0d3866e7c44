"""A few of many queries stand on a pile of duplicate points of a P-Orth tree: the pile is left to the warp-per-query
kernel, not walked by one thread first."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2601_05347_gb300 import gen  # noqa: E402

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_05347_gb300 import psi


def best_ms(f, runs=4):
    best = float("inf")
    for _ in range(runs):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        r = f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best, r


@pytest.mark.parametrize("dim,bits", [(2, 30), (3, 21)])
def test_queries_on_a_large_pile(dim, bits):
    n, pile = 1 << 20, 1 << 19
    pts = gen.uniform(n, dim, bits, 1)
    pts[:pile] = pts[0]
    pts = torch.from_numpy(pts).to("cuda")
    ix = psi.Index(pts, torch.arange(n, dtype=torch.int32, device="cuda"), kind="porth")
    nq = torch.cuda.get_device_properties(0).multi_processor_count * 1024 * 4 + 77
    q = pts[torch.randint(pile, n, (nq,), device="cuda", generator=torch.Generator("cuda").manual_seed(2))].contiguous()
    q[::nq // 30] = pts[0]
    few, got = best_ms(lambda: ix.knn(q, 1))
    warps, want = best_ms(lambda: ix.knn_stats(q, 1)[:2])  # a warp (or half a warp) per query, counters included
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    # with one thread walking the pile first: 34 against 6.6 ms (2D); without that, both calls scan it once
    assert few < 2 * warps, (few, warps)
