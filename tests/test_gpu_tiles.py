"""Edges of the tiled kernels: the split product (256-row tiles of CTA pairs,
32 of K per unit, one tensor map per row class where rows of A are not
16-byte aligned, columns in halves above 208 / 224), the Gram of a long X
(one 8 x 8 block per thread, clusters sharing the rows) and the Cholesky on a
cluster (32-column panels). Against the product, QR identities and the oracle
in float64.

Tolerances. Products: |Y - Y_ref| <= tol (|A|^T |X|) elementwise, tol = 4e-6
for FP32 (the FMA product's bound: K = 256 terms per running sum) and 1e-4 for
BF16x3 (two parts keep 16 bits per operand), as for the passes in
test_gpu_sketch. Orthonormalisation: CholeskyQR2 leaves |Q^T Q - I| at
rounding level, at most 4 d u + 16 u per entry (u = 2^-24: Gram sums in chains
of at most 256, then a d-term triangular product), and Q R reproduces X's rows
to 2 (d + 8) u |X|."""
import numpy as np
import pytest

from oracle import rqlp_oracle as orc
from paper_2110_01011_gb300 import rqlp

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


def _randn(rows, cols, seed, pad=0, shift=0):
    """rows x cols, row stride cols + pad, first value `shift` floats into a buffer."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    ld = cols + pad
    flat = torch.randn(rows * ld + shift, generator=g, device="cuda")
    return flat[shift:shift + rows * ld].view(rows, ld)[:, :cols]


def _check(A, X, trans, prec, tol):
    import torch
    Y, _ = rqlp.sketch(A, X, trans, precision=prec)
    torch.cuda.synchronize()
    A64, X64 = A.double(), X.double()
    A64 = A64.T if trans else A64
    ratio = ((Y.double() - A64 @ X64).abs() / (A64.abs() @ X64.abs())).max()
    assert float(ratio) <= tol, float(ratio)


# (m, n, d, row padding, offset of the first value): both sides of 256-row
# tiles and of 32-wide units, N at 16, 208, 224 and above, every row class;
# all of at least 2e8 multiply-adds, where FP32 takes the split product too.
PRODUCTS = [(2560, 5120, 16, 0, 0), (2561, 5121, 17, 0, 1), (1279, 1025, 208, 2, 3), (1281, 1023, 209, 3, 0),
            (1024, 1056, 224, 0, 0), (1025, 1057, 225, 1, 2), (1500, 1400, 256, 0, 2), (270, 70001, 33, 0, 0),
            (70001, 270, 33, 1, 1)]


@pytest.mark.parametrize("prec,tol", [(rqlp.PREC_FP32, 4e-6), (rqlp.PREC_BF16X3, 1e-4)], ids=["fp32", "bf16x3"])
@pytest.mark.parametrize("trans", [1, 0])
@pytest.mark.parametrize("m,n,d,pad,shift", PRODUCTS)
def test_product_edges(m, n, d, pad, shift, trans, prec, tol):
    A = _randn(m, n, m + n, pad, shift)
    _check(A, _randn(m if trans else n, d, d, shift % 2, shift), trans, prec, tol)


@pytest.mark.parametrize("value", [1e-35, -3e38, 2e-45, float("inf"), float("nan")])
@pytest.mark.parametrize("where", ["A", "X"])
def test_values_outside_the_parts_range(where, value):
    """BF16 parts represent neither the smallest nor the largest floats: the
    product is then that of the FMA form."""
    import torch
    m, n, d = 2049, 2047, 64
    A, X = _randn(m, n, 1), _randn(n, d, 2) * 2.0 ** -20
    (A if where == "A" else X)[5, 7] = value
    if abs(value) < 1e-30:   # a row or column in which nothing hides the value
        (A[5] if where == "A" else X[:, 7]).mul_(0)
        (A if where == "A" else X)[5, 7] = value
    Y, _ = rqlp.sketch(A, X, 0, precision=rqlp.PREC_FP32)
    torch.cuda.synchronize()
    ref = A.double() @ X.double()
    # Finite where a float32 is (products of 3e38 overflow); where it is not, the
    # compensated sum over K slices leaves inf or NaN in the FMA form as well.
    finite = ref.float().isfinite()
    assert bool((Y.isfinite() == finite).all())
    bound = A.double().abs() @ X.double().abs()
    # A result below the normal floats is exact to the smallest float's half.
    err = (Y.double() - ref).abs() - 2.0 ** -149
    assert bool((err[finite] <= 4e-6 * bound[finite]).all())


# d around panels and clusters of the Cholesky, rows on both sides of the long
# Gram's line (50000 rows, or rows d^2 = 3.2e8), stride and base off 16 bytes.
ORTHS = [(300, 1, 0, 0), (1000, 15, 1, 0), (1000, 16, 0, 0), (1000, 17, 0, 0), (1000, 31, 0, 3), (1000, 32, 0, 0),
         (1000, 33, 0, 0), (2000, 224, 0, 0), (2000, 225, 0, 0), (2000, 256, 0, 0), (50001, 8, 0, 0), (50000, 20, 0, 0),
         (49999, 20, 0, 0), (60001, 65, 1, 1), (20001, 129, 0, 0), (7003, 248, 0, 0), (6001, 249, 0, 2), (5001, 256, 0, 0)]


@pytest.mark.parametrize("rows,d,pad,shift", ORTHS)
def test_orth_edges(rows, d, pad, shift):
    import torch
    X = _randn(rows, d, rows + d, pad, shift)
    X64 = X.double()
    Q, R, info, _ = rqlp.orth(X)
    torch.cuda.synchronize()
    assert int(info[0]) == 0
    Q64, R64 = Q.double(), R.double()
    assert float((Q64.T @ Q64 - torch.eye(d, device="cuda")).abs().max()) <= 4 * d * U + 16 * U
    assert float(torch.tril(R64, -1).abs().max()) == 0.0
    assert float((Q64 @ R64 - X64).norm()) <= 2 * (d + 8) * U * float(X64.norm())


def test_batch_redoes_one_problem_outside_the_range():
    """FP32 batches on the tensor cores: a problem with a value that the parts
    do not represent is redone by FMAs, one with a NaN reports it, and neither
    changes the others."""
    import torch
    g = np.random.default_rng(3)
    sizes = [(int(g.integers(700, 1100)), int(g.integers(600, 900))) for _ in range(24)]
    k, p, q, u = 40, 5, 1, U
    As = [_randn(m, n, 10 + i, i % 3, i % 4) for i, (m, n) in enumerate(sizes)]
    for A in As:   # decaying columns: the leading values are well separated
        A.mul_(0.9 ** torch.arange(A.shape[1], device="cuda"))
    Os = [_randn(m, k + p, 900 + i) for i, (m, n) in enumerate(sizes)]

    def run():
        b = rqlp.Batch(As, Os, [k] * 24, [p] * 24, q, precision=0)
        b.launch()
        torch.cuda.synchronize()
        return [x.clone() for x in b.L], [x.clone() for x in b.P], b.info.cpu().numpy()

    base = run()
    As[3][4, 5] = 1e-35
    As[7][100, 3] = float("nan")
    L, P, info = run()
    assert np.all(base[2][:, 0] == 0) and info[7, 0] != 0 and np.all(np.delete(info[:, 0], 7) == 0)
    for i in range(24):
        if i not in (3, 7):
            assert torch.equal(L[i], base[0][i]) and torch.equal(P[i], base[1][i]), i
    ref = orc.rand_qlp(As[3].double().cpu().numpy(), Os[3].double().cpu().numpy(), q)
    lr = np.abs(np.diag(ref.L)[:k])
    err = np.abs(np.diag(L[3].double().cpu().numpy())[:k] - lr)
    assert np.all(err <= np.maximum(1e-4 * lr, 16 * u * lr[0]))


def test_sparse_columns_of_every_length():
    """The transpose's column sort: columns of up to 32 entries by a warp, up
    to 2048 in shared memory, longer ones in place, several entries of one
    place among them. Two calls agree bitwise, and the dense FP32 form of the
    same matrix gives L to 1e-5 of its largest entry (FP32 rounding of both)."""
    import torch
    m, k, p, q = 6000, 16, 8, 1
    lengths = [0, 1, 2, 31, 32, 33, 64, 65, 500, 2047, 2048, 2049, 3000, 6000] + [int(x) for x in range(3, 300, 3)]
    g = np.random.default_rng(8)
    rows = np.concatenate([g.choice(m, L, replace=False) for L in lengths])
    cols = np.repeat(np.arange(len(lengths)), lengths)
    rows, cols = np.append(rows, rows[-400:]), np.append(cols, cols[-400:])   # places given twice
    vals = (g.standard_normal(rows.size) / (1.0 + cols)).astype(np.float32)
    order = np.argsort(rows, kind="stable")
    rows, cols, vals = rows[order], cols[order], vals[order]
    ptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=m))]).astype(np.int64)
    n = len(lengths)
    dense = np.zeros((m, n))
    np.add.at(dense, (rows, cols), vals.astype(np.float64))
    dev = [torch.from_numpy(x).cuda() for x in (ptr, cols.astype(np.int32), vals)]
    Om = _randn(m, k + p, 4)
    a = rqlp.factor_sparse(*dev, m, n, k, p, q, Om)
    b = rqlp.factor_sparse(*dev, m, n, k, p, q, Om)
    ref = rqlp.factor(torch.from_numpy(dense.astype(np.float32)).cuda(), k, p, q, Om)
    torch.cuda.synchronize()
    assert int(a[3][0]) == 0
    for x, y in zip(a[:3], b[:3]):
        assert torch.equal(x, y)
    assert float((a[1] - ref[1]).abs().max()) <= 1e-5 * float(ref[1].abs().max())
