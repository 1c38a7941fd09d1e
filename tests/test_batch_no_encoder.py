"""Without the tensor-map encoder (no GPU here) an FP32 batch of any size takes
the FMA passes, as one FP32 matrix does, and is not refused at creation: its
layout then holds no tensor-core scratch."""

import pytest

from paper_2110_01011_gb300 import build, rqlp


def test_large_fp32_batch_is_laid_out_for_fma_passes():
    import torch
    if torch.cuda.is_available():
        pytest.skip("the encoder is there")
    build.build()
    one = rqlp.Problem(0x1000, 1000, 1000, 1000, 0x1000, 50, 45, 5, 0x1000, 50, 0x1000, 50, 0x1000, 50)

    def size(count):   # 5e7 multiply-adds a problem and pass: six make 3e8
        return rqlp.rqlp_batch_workspace_bytes(count, (rqlp.Problem * count)(*[one] * count), 1)

    step = size(4) - size(3)
    scratch = 6 * 1024 * 64 * 3 * 2   # X's parts of six problems
    assert abs((size(6) - size(5)) - step) < scratch // 4
    assert abs((size(12) - size(11)) - step) < scratch // 4
