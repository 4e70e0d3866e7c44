"""The key sort at the lengths where its tiles change size, against a stable sort."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2601_05347_gb300 import psi


@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 33000, 79999, 80000, 80001, 90000])
@pytest.mark.parametrize("bits", [1, 20, 64])
def test_sort_pairs(n, bits):
    g = torch.Generator(device="cuda").manual_seed(n + bits)
    k = torch.randint(-(1 << 62), 1 << 62, (n,), device="cuda", generator=g)
    if bits < 64:
        k &= (1 << bits) - 1
    v = torch.arange(n, dtype=torch.int32, device="cuda")
    flip = k ^ (-(1 << 63))  # unsigned order
    order = torch.sort(flip, stable=True).indices
    a, b = psi.sort_pairs(k.clone(), v.clone(), key_bits=bits)
    assert torch.equal(a, k[order]) and torch.equal(b, order.int())
