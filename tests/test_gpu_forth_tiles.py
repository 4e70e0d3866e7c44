"""Float P-Orth builds around the tiles that count in shared memory (256 points per item, 1024 counters; several items
per thread from about three hundred thousand points on): the tree is the oracle's, node for node."""
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from test_gpu_forth import T, check_tree, points  # noqa: E402

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_05347_gb300 import psi


@pytest.mark.parametrize("dim,phi,n,clustered,dup", [
    (2, 32, 33, False, 0), (3, 1, 255, False, 0), (3, 1, 256, False, 0), (3, 1, 257, True, 0),
    (2, 1, 1025, False, 0), (4, 1, 4099, False, 0), (5, 1, 8193, False, 0),   # small segments: counters do not fit
    (5, 31, 8192, True, 700), (3, 32, 319487, False, 0),                        # one or two points per thread
    (3, 32, 700001, True, 3000), (2, 8, 1300003, False, 0), (5, 32, 1245184, False, 0)])
def test_tree_matches_oracle_around_the_tiles(dim, phi, n, clustered, dup):
    p, ids = points(n, dim, 13 * dim + n % 97, clustered=clustered, dup=dup)
    f = psi.FOrth(T(p), T(ids), [0] * dim, [1] * dim, leaf_size=phi)
    o = O.FOrth(p, ids, [0] * dim, [1] * dim, phi=phi)
    check_tree(f, o)
    f.close()
