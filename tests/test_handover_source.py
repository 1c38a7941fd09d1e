"""Hand-overs between the warps of the split products, from the source. A stage
of shared memory that lanes have read goes back to the copy warp behind a proxy
fence and a releasing arrive; both CTAs' halves of X complete on the barrier
that the pair's MMAs wait for; waits acquire. Relaxed arrivals are left for
barriers whose hand-over lies in tensor memory, which the tcgen05 fences order.
A missing order need not show in any one build (the compiler's schedule can hide
it), so it is checked where it is written."""
import os
import re

import pytest

from paper_2110_01011_gb300 import build


def _read(name):
    return re.sub(r"//[^\n]*", "", open(os.path.join(build.CSRC, name)).read())


def _body(text, name):
    at = text.index(name + "(")
    depth, i = 0, text.index("{", at)
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j]
    raise AssertionError(name)


def test_shared_memory_goes_with_release_and_acquire():
    text = _read("split_device.cuh") + _read("tc_ptx.cuh")
    assert "wait.parity.relaxed" not in text
    assert text.count("arrive.relaxed") == 1 and "arrive.relaxed" in _body(text, "void arrive_remote")
    read = _body(text, "void arrive_read")
    assert read.index("fence.proxy.async") < read.index("__syncwarp") < read.index("mbar_arrive(")
    assert "cta_group::2" in _body(text, "void load_image")


@pytest.mark.parametrize("name", ["split_gemm.cu", "split_grouped.cu"])
def test_relaxed_arrivals_are_for_tensor_memory(name):
    text = _read(name)
    used = re.findall(r"arrive_(?:remote|leader)\(&?(\w+)", text)
    assert used and set(used) <= {"afull0", "acce", "corre"}
    assert "arrive_read(&fempty[" in text
    assert re.search(r"uint32_t xfull0 = leader_addr\(xfull\)", text)   # the peer's copies complete on the leader's
    assert re.search(r"load_image\([^;]*xfull0 \+ 8 \* r\.s", text)
