"""Sorted range lists of few boxes, and those of more than 16384 ids: a block of 1024 threads sorts each; lists of every
length beside the kernels of many boxes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_05347_gb300 import psi

LENGTHS = [0, 1, 2, 32, 33, 64, 65, 255, 256, 257, 1023, 1024, 1025, 4095, 4096, 4097, 16383, 16384, 16385, 40000]


@pytest.mark.parametrize("boxes,kernel,others", [(len(LENGTHS), True, False), (1, True, False), (1500, True, True)])
def test_lists_of_every_length(boxes, kernel, others):
    n = 50000
    x = np.arange(n, dtype=np.int32)
    pts = np.stack([x, np.zeros(n, np.int32)], 1)  # a line: the box [a, a + len) holds exactly len points
    ids = (np.arange(n, dtype=np.uint64) * 2654435761 % (1 << 32)).astype(np.uint32)
    ids[11] = 0xFFFFFFFF
    lens = np.resize(np.array(LENGTHS[::-1], np.int64), boxes)
    lo = (np.arange(boxes) * 977) % (n - lens)
    box = np.stack([lo, np.zeros_like(lo), lo + lens - 1, np.zeros_like(lo)], 1).astype(np.int32)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).to("cuda")
    ix = psi.Index(T(pts), T(ids))
    psi.profile_enable(True)
    psi.profile_reset()
    try:
        off, got = ix.range_report(T(box), capacity=int(lens.sum()), sort=True)
        names = psi.profile_dump()
    finally:
        psi.profile_enable(False)
    assert ("k_sort_seg_any" in names) == kernel and ("k_sort_seg_warp" in names) == others
    off, got = off.cpu().numpy(), got.cpu().numpy().view(np.uint32)
    assert (np.diff(off) == lens).all()
    for i, (a, m) in enumerate(zip(lo, lens)):
        assert (got[off[i]:off[i + 1]] == np.sort(ids[a:a + m])).all(), (i, m)
