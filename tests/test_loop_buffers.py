"""CPU check of the loop buffers of pipelined flows: two stages' loops run on two streams at a time, each into its own FP32
buffer, so the split two-band flow k-sum must not write the one FP64 loop buffer (nothing reads it there)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_08830_gb300", "csrc")


def _function(name, file):
    with open(os.path.join(CSRC, file), encoding="utf-8") as fh:
        src = fh.read()
    start = src.index("\n{", src.index(name + "(")) + 1
    depth = 0
    for i in range(start, len(src)):
        depth += (src[i] == "{") - (src[i] == "}")
        if depth == 0:
            return src[start:i + 1]
    raise AssertionError(name)


def test_flow_stages_write_only_their_own_loop_buffer():
    body = _function("cudaError_t launch_loops_flow", "k_loops2.cu")
    assert "d_Lc32" in body and not re.search(r"\bd_Lc\b", body)
    # the stages take turns on the FP32 buffers
    stage = _function("tufrg_status enqueue_attempt", "api.cu")
    assert "d_Lc32B" in stage and "launch_loops_flow" not in stage
