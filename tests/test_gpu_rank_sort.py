"""Small encoding sorts (tiles sorted in registers, then ranked) against the digit passes: the same index, point by
point, at the lengths where tiles begin and where the form ends."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_05347_gb300 import psi


@pytest.mark.parametrize("n", [1, 2, 255, 1023, 1024, 1025, 4096, 5000, 81919, 81920, 81921])
@pytest.mark.parametrize("kind,dim,bits", [("spac_h", 2, 30), ("spac_z", 3, 21), ("porth", 2, 31), ("spac_h", 3, 4),
                                           ("spac_z", 2, 1)])
def test_same_index_as_the_digit_passes(n, kind, dim, bits):
    g = torch.Generator(device="cuda").manual_seed(n + bits)
    pts = torch.randint(0, (1 << bits) - 1 if bits > 30 else 1 << bits, (n, dim), dtype=torch.int32, device="cuda", generator=g)
    pts[: n // 3] = pts[0].clone()  # a pile of equal keys across tiles
    ids = torch.randperm(n, device="cuda", generator=g).int()
    a, b = (psi.Index(pts, ids, kind=kind, coord_bits=bits, radix_bits=r) for r in (0, 8))
    m = n // 2 + 1
    new = torch.randint(0, 1 << min(bits, 30), (m, dim), dtype=torch.int32, device="cuda", generator=g)
    nid = torch.arange(n, n + m, dtype=torch.int32, device="cuda")
    gone = torch.randint(0, n, (m,), device="cuda", generator=g)  # with repeated entries
    count = [torch.zeros(1, dtype=torch.int64, device="cuda") for _ in range(2)]
    for ix, c in ((a, count[0]), (b, count[1])):
        ix.insert(new, nid)
        ix.delete(pts[gone].contiguous(), ids[gone].contiguous(), c)
        ix.sync()
    assert int(count[0]) == int(count[1]) == gone.unique().numel()
    pa, pb = a.points(), b.points()
    assert all(torch.equal(pa[k], pb[k]) for k in pa)


def test_query_order_and_range_errors():
    g = torch.Generator(device="cuda").manual_seed(3)
    pts = torch.randint(0, 1 << 30, (9000, 2), dtype=torch.int32, device="cuda", generator=g)
    ids = torch.arange(9000, dtype=torch.int32, device="cuda")
    a, b = (psi.Index(pts, ids, kind="spac_h", radix_bits=r) for r in (0, 8))
    q = torch.randint(0, 1 << 30, (6001, 2), dtype=torch.int32, device="cuda", generator=g)
    assert all(torch.equal(x, y) for x, y in zip(a.knn(q, 7), b.knn(q, 7)))
    pts[5], ids[5] = -1, -1  # the highest key that coordinates out of range can give, and the highest id
    with pytest.raises(psi.PsiError) as e:
        ix = psi.Index(pts, ids, kind="spac_z")
        ix.sync()
    assert e.value.status == psi.ERR_RANGE
