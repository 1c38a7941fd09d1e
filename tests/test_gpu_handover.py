"""A stage of A must not be refilled while lanes still read it. With every entry
of unit u of K (32 wide) equal to u and X the 0/1 matrix that sums unit u into
column u, every result is 32 u exactly, and a value read from a refilled stage
shows as a multiple of the ring's length. Rows enough for every CTA pair to pass
several row tiles: where a tile ends, the lanes' reads queue behind the stores
of the result."""
import pytest

from paper_2110_01011_gb300 import rqlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pad", [0, 1], ids=["aligned", "unaligned"])
@pytest.mark.parametrize("prec,parts", [(rqlp.PREC_BF16X3, 2), (rqlp.PREC_BF16X3, 3), (rqlp.PREC_FP32, 0)],
                         ids=["two", "three", "fp32"])
@pytest.mark.parametrize("trans", [0, 1])
@pytest.mark.parametrize("units", [200, 90])
def test_every_unit_lands_in_its_column(units, trans, prec, parts, pad):
    import torch
    K, M = 32 * units, 20000
    u = torch.arange(K, device="cuda") // 32
    rows = (K, M) if trans else (M, K)
    A = torch.empty(rows[0], rows[1] + pad, device="cuda")[:, :rows[1]]
    A.copy_((u[:, None] if trans else u[None, :]).float().expand(rows))
    X = torch.zeros(K, units, device="cuda")
    X[torch.arange(K, device="cuda"), u] = 1
    want = (32 * torch.arange(units, device="cuda")).float().expand(M, units)
    for _ in range(4):
        Y, _ = rqlp.sketch(A, X, trans, precision=prec, parts=parts)
        torch.cuda.synchronize()
        assert torch.equal(Y, want), (Y - want).abs().max()
