"""k-NN of many queries (the one-query-per-thread kernel and the queries it leaves to the others): all results
against the instrumented warp-per-query kernels, a sample against the oracle, bit-exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_2601_05347_gb300 import gen  # noqa: E402

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_05347_gb300 import psi


def T(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).to("cuda")


def enough(waves):
    """More queries than `waves` times what fills the chip, and not a multiple of a block."""
    return int(torch.cuda.get_device_properties(0).multi_processor_count * 1024 * waves) + 77


def shaped(shape, n, dim, bits, seed):
    if shape == "uniform":
        return gen.uniform(n, dim, bits, seed)
    if shape == "walks":
        return gen.varden(n, dim, bits, seed, clusters=7)
    if shape == "piles":  # 32 values per axis: piles of duplicates, equal distances everywhere
        return (gen.uniform(n, dim, bits, seed) >> (bits - 5)).astype(np.int32)
    # two far corners: the curve jumps between them
    p = gen.uniform(n, dim, bits - 8, seed)
    p[n // 2:] += (1 << bits) - (1 << (bits - 8))
    return p


@pytest.mark.parametrize("kind,dim,bits,n,phi,k,waves,shape", [
    ("spac_h", 2, 30, 30000, 32, 1, 1, "walks"), ("spac_z", 2, 30, 30001, 31, 5, 1, "corners"),
    ("spac_h", 2, 31, 30002, 32, 10, 1.5, "uniform"), ("spac_h", 2, 30, 20000, 33, 16, 2, "piles"),
    ("spac_z", 3, 21, 30000, 32, 10, 1.5, "walks"), ("spac_h", 3, 21, 25000, 7, 9, 1.5, "corners"),
    ("spac_z", 3, 21, 20000, 64, 16, 3, "uniform"), ("porth", 2, 30, 30000, 32, 10, 2, "walks"),
    ("porth", 2, 30, 20001, 8, 16, 4, "corners"), ("porth", 3, 21, 30000, 32, 10, 4, "uniform"),
    ("porth", 3, 21, 20000, 32, 4, 2.5, "piles"), ("porth", 2, 30, 20000, 32, 1, 1, "uniform"),
    ("spac_h", 2, 30, 7, 32, 10, 1.5, "uniform"), ("porth", 3, 21, 40, 32, 5, 2.5, "walks"),
    ("spac_z", 2, 30, 1, 32, 1, 1, "uniform"),
])
def test_many_queries_match_the_warp_kernels_and_the_oracle(kind, dim, bits, n, phi, k, waves, shape):
    p = shaped(shape, n, dim, bits, 5)
    ids = (np.arange(n, dtype=np.uint64) * 2654435761 % (1 << 32)).astype(np.uint32)
    nq = enough(waves)
    q = p[gen.sample_with_replacement(n, nq, 6)].copy()
    q[: nq // 4] = gen.uniform(nq // 4, dim, bits, 7)  # away from the data
    jitter = gen.uniform(nq // 4, dim, 4, 8)
    q[-(nq // 4):] = np.minimum(q[-(nq // 4):] + jitter, (1 << bits) - 1)
    ix = psi.Index(T(p), T(ids), kind=kind, leaf_size=phi, coord_bits=bits)
    new = shaped(shape, n // 3, dim, bits, 9)  # leaves of other sizes than a fresh build's
    nid = (ids[: n // 3] + np.uint32(1)).astype(np.uint32)
    if n > 100:
        ix.insert(T(new), T(nid))
        ix.delete(T(p[: n // 5]), T(ids[: n // 5]))
    gi, gd = ix.knn(T(q), k)
    wi, wd, _ = ix.knn_stats(T(q), k)
    ix.sync()
    assert torch.equal(gi, wi) and torch.equal(gd, wd)
    o = O.Index(p, ids, dim=dim, kind={"spac_z": O.SPAC_Z, "spac_h": O.SPAC_H, "porth": O.PORTH}[kind], phi=phi, bits=bits)
    if n > 100:
        o.insert(new, nid)
        o.delete(p[: n // 5], ids[: n // 5])
    at = gen.sample_with_replacement(nq, 300, 10)
    oi, od = o.knn(q[at], k)
    assert (gi.cpu().numpy().view(np.uint32)[at] == oi).all() and (gd.cpu().numpy()[at] == od).all()


@pytest.mark.parametrize("kind,dim,k", [("spac_h", 2, 10), ("spac_z", 3, 1)])
def test_many_queries_of_many_indexes(kind, dim, k):
    bits = 30 if dim == 2 else 21
    sizes = [0, 1, 31, 700, 5000, 3, 20000, 0, 90] + [40] * 60
    off = np.concatenate([[0], np.cumsum(sizes)])
    pts = np.concatenate([shaped(("uniform", "walks", "corners", "piles")[i % 4], s, dim, bits, 20 + i)
                          for i, s in enumerate(sizes)]).astype(np.int32)
    b = psi.Batch(off, dim=dim, kind=kind)
    b.build(T(pts), T(np.arange(off[-1], dtype=np.uint32)))
    per = enough(1.5) // len(sizes) + 1
    qoff = torch.arange(len(sizes) + 1, dtype=torch.int64, device="cuda") * per
    q = np.concatenate([np.concatenate([pts[off[i] + gen.sample_with_replacement(s, per - per // 3, 50 + i)] if s else
                                        gen.uniform(per - per // 3, dim, bits, 50 + i),
                                        gen.uniform(per // 3, dim, bits, 90 + i)]) for i, s in enumerate(sizes)])
    gi, gd = b.knn(T(q), qoff, k)
    wi, wd, _ = b.knn_stats(T(q), qoff, k)
    b.sync()
    assert torch.equal(gi, wi) and torch.equal(gd, wd)
