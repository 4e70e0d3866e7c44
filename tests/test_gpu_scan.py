"""The device scans at the lengths where their form changes (one block; block sums added up by each block; block sums
scanned), through the calls that use them."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_05347_gb300 import psi

EDGES = [1, 4095, 4097, 16384, 16385, 2048 * 4096, 2048 * 4096 + 1]


@pytest.mark.parametrize("q", EDGES)
def test_report_offsets(q):
    g = torch.Generator(device="cuda").manual_seed(q)
    pts = torch.randint(0, 1 << 10, (200, 2), dtype=torch.int32, device="cuda", generator=g)
    ix = psi.Index(pts, torch.arange(200, dtype=torch.int32, device="cuda"), kind="spac_h", coord_bits=10)
    lo = torch.randint(0, 1 << 10, (q, 2), dtype=torch.int32, device="cuda", generator=g)
    boxes = torch.cat([lo, lo + 30], 1).contiguous()
    off, ids = ix.range_report(boxes)
    want = torch.cumsum(ix.range_count(boxes), 0)
    assert off[0] == 0 and torch.equal(off[1:], want) and ids.numel() == int(want[-1])


@pytest.mark.parametrize("n", EDGES)
def test_orth_leaves_cover_the_points(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    pts = torch.randint(0, 1 << 21, (n, 3), dtype=torch.int32, device="cuda", generator=g)
    ix = psi.Index(pts, torch.arange(n, dtype=torch.int32, device="cuda"), kind="porth")
    p, lv = ix.points(), ix.leaves()
    assert int(lv["count"].sum()) == n and int(lv["count"].min()) >= 1 and int(lv["count"].max()) <= 32
    assert torch.equal(p["pts"], pts[p["ids"].long()])
    assert torch.equal(p["ids"].sort().values, torch.arange(n, dtype=torch.int32, device="cuda"))
    assert bool((p["keys"][1:] >= p["keys"][:-1]).all())
    start = torch.cumsum(lv["count"], 0) - lv["count"]
    assert torch.equal(p["leaf"][start], torch.arange(lv["count"].numel(), dtype=torch.int32, device="cuda"))
