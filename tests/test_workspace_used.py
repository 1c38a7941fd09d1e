"""Scratch sizes hold what a call uses (host only: no device pointer is read)."""
from paper_2110_01011_gb300 import rqlp


def test_sparse_plans_have_no_room_for_dense_products():
    """A sparse factorisation never runs the split product, whose image of X and
    partial tiles are the larger part of a dense plan's scratch at this size."""
    fake, n, k, p = 0x1000, 7320, 100, 10
    nnz = 13 * n
    dense = rqlp.rqlp_workspace_bytes(n, n, k, p, 1)
    sparse = rqlp.rqlp_sparse_workspace_bytes(rqlp.Csr(n, n, nnz, fake, fake, fake), k, p, 1)
    transposed = 8 * (n + 1) + 8 * nnz + 4 * n
    image = 3 * 2 * n * 112   # of X in three BF16 parts, 110 columns
    assert transposed < sparse <= dense + transposed - image
