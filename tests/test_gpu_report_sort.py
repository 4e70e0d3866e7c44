"""Range report with sorted ids at the lengths where the segment sort changes its form."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_05347_gb300 import psi

EDGES = [0, 1, 2, 31, 32, 33, 63, 64, 65, 128, 129, 255, 256, 257, 511, 512, 513, 1024, 1025, 2047, 2048, 2049, 4095,
         4096, 4097, 8192, 8193, 16384, 16385, 20000]


@pytest.mark.parametrize("kind", ["spac_h", "porth"])
def test_sorted_report_of_every_segment_length(kind):
    n = 40000
    x = np.arange(n, dtype=np.int32)
    pts = np.stack([x, np.zeros(n, np.int32)], 1)  # a line: the box [a, a + len) holds exactly len points
    ids = (np.arange(n, dtype=np.uint64) * 2654435761 % (1 << 32)).astype(np.uint32)
    ids[7] = 0xFFFFFFFF
    lens = np.array(EDGES + EDGES[::-1] + [n], np.int64)
    lo = (np.arange(len(lens)) * 977) % (n - np.minimum(lens, n - 1))
    lo[-1] = 0
    boxes = np.stack([lo, np.zeros_like(lo), lo + lens - 1, np.zeros_like(lo)], 1).astype(np.int32)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).to("cuda")
    off, got = psi.Index(T(pts), T(ids), kind=kind).range_report(T(boxes), sort=True)
    off, got = off.cpu().numpy(), got.cpu().numpy().view(np.uint32)
    assert (np.diff(off) == lens).all()
    for i, (a, m) in enumerate(zip(lo, lens)):
        assert (got[off[i]:off[i + 1]] == np.sort(ids[a:a + m])).all(), (i, m)
