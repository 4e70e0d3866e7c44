"""k-NN of many queries that the one-query-per-thread kernels leave to the others: all of them (taken in curve order),
half of them (taken from the list), and few, on trees deep enough for long walks; results against the warp kernels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2601_05347_gb300 import gen  # noqa: E402

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_05347_gb300 import psi


def enough(waves):
    return int(torch.cuda.get_device_properties(0).multi_processor_count * 1024 * waves) + 77


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


@pytest.mark.parametrize("share", [1.0, 0.74, 0.5, 0.01])
@pytest.mark.parametrize("kind,dim,bits,k,waves", [("spac_h", 2, 30, 1, 1), ("spac_z", 3, 21, 10, 1.2),
                                                   ("porth", 2, 30, 8, 1), ("porth", 3, 21, 16, 2)])
def test_far_queries_of_any_share(kind, dim, bits, k, waves, share):
    n, nq = 30011, enough(waves)
    pts = gen.uniform(n, dim, bits - 9, 1)  # a corner of the grid
    q = pts[gen.sample_with_replacement(n, nq, 2)].copy()
    far = np.arange(nq) % 100 < 100 * share
    q[far] = gen.uniform(int(far.sum()), dim, bits, 3)
    ix = psi.Index(T(pts), torch.arange(n, dtype=torch.int32, device="cuda"), kind=kind)
    got, want = ix.knn(T(q), k), ix.knn_stats(T(q), k)[:2]
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("kind,dim,bits,k,shape", [("spac_h", 2, 30, 10, "walks"), ("spac_z", 3, 21, 16, "walks"),
                                                   ("porth", 2, 30, 16, "walks"), ("porth", 3, 21, 13, "walks"),
                                                   ("porth", 3, 21, 10, "uniform"), ("spac_h", 3, 21, 10, "uniform")])
def test_millions_of_points(kind, dim, bits, k, shape):
    n, nq = 3_000_017, enough(2.6)
    pts = T(gen.varden(n, dim, bits, 1) if shape == "walks" else gen.uniform(n, dim, bits, 1))
    g = torch.Generator("cuda").manual_seed(4)
    q = pts[torch.randint(0, n, (nq,), device="cuda", generator=g)]
    q[::7] = torch.randint(0, 1 << bits, q[::7].shape, dtype=torch.int32, device="cuda", generator=g)
    ix = psi.Index(pts, torch.arange(n, dtype=torch.int32, device="cuda"), kind=kind)
    got, want = ix.knn(q, k), ix.knn_stats(q, k)[:2]
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("share", [1.0, 0.5])
def test_batch_with_far_queries(share):
    sizes = [9000, 0, 20001, 1]
    off = np.concatenate([[0], np.cumsum(sizes)])
    nq = enough(3)
    pts = T(gen.uniform(int(off[-1]), 2, 21, 5))
    g = torch.Generator("cuda").manual_seed(6)
    q = pts[torch.randint(0, len(pts), (nq,), device="cuda", generator=g)]
    far = torch.rand(nq, device="cuda", generator=g) < share
    q[far] = torch.randint(0, 1 << 30, (int(far.sum()), 2), dtype=torch.int32, device="cuda", generator=g)
    b = psi.Batch(off, dim=2, kind="spac_h")
    b.build(pts, torch.arange(len(pts), dtype=torch.int32, device="cuda"))
    qoff = torch.linspace(0, nq, len(sizes) + 1, device="cuda").long()
    got, want = b.knn(q, qoff, 10), b.knn_stats(q, qoff, 10)[:2]
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


@pytest.mark.parametrize("dim,k,share", [(2, 1, 1.0), (3, 10, 1.0), (3, 16, 0.5), (5, 10, 1.0)])
def test_float_tree(dim, k, share):
    n, nq = 20011, enough(1.6)
    g = torch.Generator("cuda").manual_seed(7)
    pts = torch.rand((n, dim), device="cuda", generator=g) * 0.002
    q = pts[torch.randint(0, n, (nq,), device="cuda", generator=g)]
    far = torch.rand(nq, device="cuda", generator=g) < share
    q[far] = torch.rand((int(far.sum()), dim), device="cuda", generator=g)
    ix = psi.FOrth(pts, torch.arange(n, dtype=torch.int32, device="cuda"), [0.0] * dim, [1.0] * dim)
    got = ix.knn(q, k)
    parts = [ix.knn(x, k) for x in q.split(enough(0.4))]  # too few for one query per thread
    for a, b in zip(got, zip(*parts)):
        assert torch.equal(a, torch.cat(b))
