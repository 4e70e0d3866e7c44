"""Float P-Orth k-NN of many queries (the one-query-per-thread kernel and the queries it leaves to the other) against
calls small enough to take the warp-per-query kernel, and a sample against the oracle, bit-exact."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_05347_gb300 import psi


@pytest.mark.parametrize("dim,k,n,phi,shape", [(2, 10, 20001, 32, "uniform"), (3, 10, 30000, 32, "clusters"),
                                               (3, 16, 20000, 7, "piles"), (4, 1, 20000, 32, "uniform"),
                                               (5, 10, 20000, 32, "clusters"), (2, 3, 25, 32, "uniform"),
                                               (2, 16, 9, 4, "uniform"), (5, 16, 15000, 16, "piles"),
                                               (3, 10, 20000, 32, "tiny")])
def test_many_queries(dim, k, n, phi, shape):
    rng = np.random.default_rng(dim * 100 + k)
    p = rng.random((n, dim))
    if shape == "clusters":
        p = rng.random((9, dim))[rng.integers(0, 9, n)] + rng.normal(0, 1e-3, (n, dim))
    elif shape == "piles":  # few distinct points, equal distances everywhere, one pile longer than any leaf
        p = np.floor(p * 6) / 6
        p[:2000] = p[0]
    elif shape == "tiny":  # squared distances below the smallest normal float
        p = p * 1e-20
    p = np.clip(p, 0, np.nextafter(np.float32(1), np.float32(0))).astype(np.float32)
    ids = (rng.permutation(n) * 3 + 1).astype(np.uint32)
    nq = int(torch.cuda.get_device_properties(0).multi_processor_count * 1024 * 2) + 77
    q = p[rng.integers(0, n, nq)].copy()
    q[: nq // 3] = rng.random((nq // 3, dim)) * 3 - 1
    q[nq // 2:] += rng.normal(0, 1e-4 if shape != "tiny" else 1e-22, q[nq // 2:].shape).astype(np.float32)
    q[5], q[6], q[7] = np.nan, np.inf, 3e30
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda")
    f = psi.FOrth(T(p), T(ids.view(np.int32)), [0.0] * dim, [1.0] * dim, leaf_size=phi)
    gi, gd = f.knn(T(q), k)
    f.sync()
    part = [f.knn(T(q[a: a + 4000]), k) for a in list(range(0, nq, 4000))[::5]]
    for j, a in enumerate(list(range(0, nq, 4000))[::5]):
        assert torch.equal(gi[a: a + 4000], part[j][0])
        assert torch.equal(gd[a: a + 4000].view(torch.int64), part[j][1].view(torch.int64))
    o = O.FOrth(p, ids, [0.0] * dim, [1.0] * dim, phi=phi)
    at = rng.integers(8, nq, 200)
    oi, od = o.knn(q[at], k)
    assert (gi.cpu().numpy().view(np.uint32)[at] == oi).all() and (gd.cpu().numpy()[at] == od).all()
