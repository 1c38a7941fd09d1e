"""FP32 products with very small entries: values that BF16 parts hold only when
scaled take the tensor-core form like any other, with the accuracy of FP32."""
import pytest

torch = pytest.importorskip("torch")

from paper_2110_01011_gb300 import rqlp

pytestmark = pytest.mark.gpu
M, N, D = 4099, 2500, 96
TINY = [1e-30, 1.3e-35, -1.2e-38, 1e-41, 2.0 ** -149]


def _randn(*shape, seed):
    return torch.randn(*shape, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda")


@pytest.mark.parametrize("trans", [0, 1])
@pytest.mark.parametrize("where", ["A", "X"])
def test_small_entries_among_others_change_nothing(where, trans):
    """Far below an ulp of every sum, so the results are those with zeros in
    their place, bit for bit: both came the same way."""
    A, X = _randn(M, N, seed=1), _randn(M if trans else N, D, seed=2)
    t = A if where == "A" else X
    at = torch.rand(t.shape, generator=torch.Generator(device="cuda").manual_seed(3), device="cuda") < 0.01
    t[at] = 0
    base = rqlp.sketch(A, X, trans, precision=rqlp.PREC_FP32)[0].clone()
    t[at] = torch.tensor(TINY, device="cuda").repeat(int(at.sum()))[:int(at.sum())]
    Y, _ = rqlp.sketch(A, X, trans, precision=rqlp.PREC_FP32)
    assert torch.equal(Y, base)


@pytest.mark.parametrize("trans", [0, 1])
@pytest.mark.parametrize("scale", [1e-30, 1e-37, 1e-39, 1e-44])
def test_rows_of_small_values(scale, trans):
    """Rows of the result that consist of small values only. 4e-6 of |A| |X| as for
    every FP32 product; below the normal floats a sum of t terms is off by at most
    t + 1 halves of the smallest one (K slices and partial sums: t = 200)."""
    A, X = _randn(M, N, seed=4), _randn(M if trans else N, D, seed=5)
    (A[:, ::3] if trans else A[::3]).mul_(scale)
    Y, _ = rqlp.sketch(A, X, trans, precision=rqlp.PREC_FP32)
    op = (A.T if trans else A).double()
    err = (Y.double() - op @ X.double()).abs() - 100 * 2.0 ** -149
    assert bool((err <= 4e-6 * (op.abs() @ X.double().abs())).all())


def test_basis_of_small_values():
    """Columns of X far below the range of the parts."""
    A, X = _randn(M, N, seed=6), _randn(N, D, seed=7)
    X[:, 5].mul_(1e-37)
    X[:, 9].mul_(1e-42)
    Y, _ = rqlp.sketch(A, X, 0, precision=rqlp.PREC_FP32)
    err = (Y.double() - A.double() @ X.double()).abs() - 100 * 2.0 ** -149
    assert bool((err <= 4e-6 * (A.double().abs() @ X.double().abs())).all())


def test_batch_keeps_small_entries():
    """The grouped form: small entries leave the factors as they are with zeros."""
    def run(value):
        As, Os = [], []
        for i in range(12):
            A = _randn(900 + i, 800 - i, seed=20 + i) * 0.9 ** torch.arange(800 - i, device="cuda")
            A[i::7, i::11] = value
            As.append(A)
            Os.append(_randn(900 + i, 45, seed=50 + i))
        b = rqlp.Batch(As, Os, [40] * 12, [5] * 12, 1, precision=0)
        b.launch()
        torch.cuda.synchronize()
        assert not bool(b.info.any())
        return [x.clone() for x in b.L]
    for a, b in zip(run(0.0), run(1e-35)):
        assert torch.equal(a, b)


@pytest.mark.parametrize("scale_a,scale_x", [(1e20, 1.0), (1e30, 1.0), (1.0, 1e30), (1e18, 1e18), (1e33, 1e-33)])
def test_large_values(scale_a, scale_x):
    """Sums and values that overflow in the scaled form come from the FMA units,
    the others from the tensor cores; either way they are FP32's."""
    A, X = _randn(M, N, seed=8) * scale_a, _randn(N, D, seed=9) * scale_x
    Y, _ = rqlp.sketch(A, X, 0, precision=rqlp.PREC_FP32)
    ref = A.double() @ X.double()
    assert bool(Y.isfinite().all())
    assert bool(((Y.double() - ref).abs() <= 4e-6 * (A.double().abs() @ X.double().abs())).all())
