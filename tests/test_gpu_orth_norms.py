"""Column norms of an FP32 orthonormalisation: rounding may move them either
way, but not all of them the same way."""
import pytest

torch = pytest.importorskip("torch")

from paper_2110_01011_gb300 import rqlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,d", [(20000, 210), (5000, 60), (100000, 120)])
def test_column_norms_are_not_short(m, d):
    """Mean of |q_j|^2 - 1 within 4e-8, two thirds of the 2^-24 by which one
    rounding below 1 is off. A root's reciprocal that is 5e-8 low next to 1 takes
    twice that off every |q_j|^2."""
    g = torch.Generator(device="cuda").manual_seed(m + d)
    X = torch.randn(m, d, generator=g, device="cuda") * torch.exp(-3 * torch.arange(d, device="cuda") / d)
    Q, _, info, _ = rqlp.orth(X)
    assert int(info[0]) == 0
    short = float((Q.double().square().sum(0) - 1).mean())
    assert abs(short) <= 4e-8, short
