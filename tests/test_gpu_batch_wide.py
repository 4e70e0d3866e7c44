"""Batches with a few large indexes, built by device-wide sorts when the block's form is left open: the same layout,
points and results as a block per index gives (and, through it, the oracle)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2601_05347_gb300 import gen  # noqa: E402

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_05347_gb300 import psi


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).to("cuda")


@pytest.mark.parametrize("kind,dim,bits,phi,sizes,shape", [
    ("spac_h", 2, 30, 32, [0, 5, 60000, 60000, 0, 33, 1, 20000, 0], "same"),
    ("spac_z", 3, 21, 16, [60000, 32, 31, 40000], "piles"),
    ("spac_h", 3, 21, 64, [80001], "uniform"),
    ("spac_z", 2, 31, 7, [3, 70000, 2], "uniform"),
    ("spac_h", 2, 3, 32, [50000, 49, 50000], "uniform"),  # 6-bit keys: runs of about 800 equal points
    ("spac_h", 2, 30, 32, [70000] + [20] * 300, "walks"),  # index numbers of 9 bits
])
def test_layout_and_results_of_a_device_wide_build(kind, dim, bits, phi, sizes, shape):
    off = np.concatenate([[0], np.cumsum(sizes)])
    parts = []
    for i, n in enumerate(sizes):
        seed = 3 if shape == "same" else 3 + i  # "same": neighbouring indexes begin with the same points
        p = gen.varden(n, dim, bits, seed) if shape == "walks" else gen.uniform(n, dim, bits, seed)
        if shape == "piles":
            p = (p >> (bits - 2)).astype(np.int32)
            p[: n // 8] = p[:1]  # one pile of thousands
        if shape == "same" and n:
            p[-(n // 3 + 1):] = (1 << bits) - 1  # the last key of each index is a pile too
            p[: n // 3] = p[-1]
        parts.append(p)
    pts = T(np.concatenate(parts).astype(np.int32))
    ids = T((np.arange(off[-1], dtype=np.uint64) * 2654435761 % (1 << 32)).astype(np.uint32))
    q = pts[torch.randint(0, int(off[-1]), (3000,), device="cuda", generator=torch.Generator("cuda").manual_seed(1))]
    qoff = torch.linspace(0, 3000, len(sizes) + 1, device="cuda").long()
    got = []
    for threads in (0, 512):
        b = psi.Batch(off, dim=dim, kind=kind, leaf_size=phi, coord_bits=bits, threads=threads)
        n0 = psi.launch_count()
        b.build(pts, ids)
        launches = psi.launch_count() - n0
        assert launches == 1 if threads else launches > 1  # the device-wide form ran
        r = [b.leaves(i) for i in range(len(sizes))], b.knn(q.contiguous(), qoff, 40), b.knn(q.contiguous(), qoff, 1)
        b.sync()
        got.append(r)
    for x, y in zip(got[0][0], got[1][0]):
        assert all(torch.equal(x[f], y[f]) for f in ("count", "lo", "hi"))
    for x, y in zip(got[0][1] + got[0][2], got[1][1] + got[1][2]):
        assert torch.equal(x, y)


def test_out_of_range_coordinates_are_reported():
    pts = T(gen.uniform(70000, 2, 30, 1))
    pts[123, 1] = -5
    b = psi.Batch([0, 70000], dim=2, kind="spac_h")
    b.build(pts, torch.arange(70000, dtype=torch.int32, device="cuda"))
    with pytest.raises(psi.PsiError) as e:
        b.sync()
    assert e.value.status == psi.ERR_RANGE
