"""A bounded wait of the split product that runs out (a stage that is withheld,
no GPU fault): rqlp_sketch has no status word, so an FP32 pass must still be
right (it is redone without waits), and a BF16x3 pass must show what it lost."""
import ctypes

import pytest

from paper_2110_01011_gb300 import rqlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [rqlp.PREC_FP32, rqlp.PREC_BF16X3], ids=["fp32", "bf16x3"])
def test_withheld_stage_leaves_no_silent_result(prec):
    import torch
    m, n, d = 6000, 4000, 48
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    A, X = torch.randn(m, n, generator=g, device="cuda"), torch.randn(n, d, generator=g, device="cuda")
    ref, bound = A.double() @ X.double(), A.double().abs() @ X.double().abs()
    opts = rqlp._opts(prec)
    nb = rqlp.rqlp_sketch_workspace_bytes(0, m, n, d, opts)
    buf, ws = rqlp._workspace(nb, A.device)
    Y = torch.zeros(m, d, device="cuda")
    stalled = rqlp.load().rqlp_test_sketch_stalled
    stalled.argtypes = rqlp.load().rqlp_sketch.argtypes
    tol = 4e-6 if prec == rqlp.PREC_FP32 else 1e-4   # as for the passes in test_gpu_tiles

    def run(call):
        assert call(0, A.data_ptr(), m, n, n, X.data_ptr(), d, d, Y.data_ptr(), d, ws, nb, ctypes.byref(opts),
                    rqlp._stream()) == 0
        torch.cuda.synchronize()
        return (Y.double() - ref).abs() <= tol * bound, Y.isnan()

    right, lost = run(stalled)
    if prec == rqlp.PREC_FP32:
        assert bool(right.all())
    else:
        assert bool(lost.any()) and bool((right | lost).all())
    right, lost = run(rqlp.load().rqlp_sketch)   # the context and the workspace are as good as before
    assert bool(right.all())
