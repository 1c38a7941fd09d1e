"""Accumulation chains of the three-part BF16x3 product end after K = 2048: the MMAs
lose toward zero with every add, the more the longer the chain."""
import pytest

torch = pytest.importorskip("torch")

from paper_2110_01011_gb300 import rqlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("trans", [0, 1])
def test_a_long_product_loses_what_its_slices_lose(trans):
    """Values of one sign, whose sums grow evenly. With one 128-row tile per SM
    no chain ends anywhere else, so K = 10240 consists of the same chains as five
    products of 2048 and loses the same but for the rounding of four adds (chains
    of 2560 lose a quarter more)."""
    M = 128 * torch.cuda.get_device_properties(0).multi_processor_count
    K, d, S = 10240, 64, 2048
    g = torch.Generator(device="cuda").manual_seed(6)
    A = torch.rand(K, M, generator=g, device="cuda") if trans else torch.rand(M, K, generator=g, device="cuda")
    X = torch.rand(K, d, generator=g, device="cuda")

    def product(k0, k1):
        part = A[k0:k1] if trans else A[:, k0:k1]
        return rqlp.sketch(part, X[k0:k1], trans, precision=rqlp.PREC_BF16X3, parts=3)[0].double()

    ref = (A.T if trans else A).double() @ X.double()
    whole = float((1 - product(0, K) / ref).mean())
    slices = float((1 - sum(product(k, k + S) for k in range(0, K, S)) / ref).mean())
    assert abs(whole - slices) <= 0.1 * abs(slices), (whole, slices)
