"""k-NN of few queries on a P-Orth tree (several nodes expanded at once when the list is full): lists longer than the
tree, piles of duplicates, queries at and away from the data; results against the instrumented kernel."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2601_05347_gb300 import gen  # noqa: E402

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_05347_gb300 import psi


@pytest.mark.parametrize("dim,bits", [(2, 30), (3, 21)])
@pytest.mark.parametrize("n,leaf,shape", [(3, 32, "uniform"), (31, 1, "uniform"), (20000, 32, "walks"),
                                          (20000, 1, "uniform"), (20000, 16, "piles")])
@pytest.mark.parametrize("k", [1, 2, 32])
def test_few_queries(dim, bits, n, leaf, shape, k):
    pts = gen.varden(n, dim, bits, 1) if shape == "walks" else gen.uniform(n, dim, bits, 1)
    if shape == "piles":
        pts = (pts >> (bits - 4)).astype(np.int32)
    q = gen.uniform(700, dim, bits, 2)
    q[:400] = pts[gen.sample_with_replacement(n, 400, 3)]
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda")
    ix = psi.Index(T(pts), torch.arange(n, dtype=torch.int32, device="cuda"), kind="porth", leaf_size=leaf)
    for nq in (1, 700):
        got, want = ix.knn(T(q[:nq]), k), ix.knn_stats(T(q[:nq]), k)[:2]
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
