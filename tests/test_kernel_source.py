"""Properties of the kernels' source that no run can be made to show without a GPU fault."""

import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_15039_gb300", "csrc")


def test_every_drain_arrival_is_waited_for():
    """A tcgen05.commit arrives on its barrier some time later: where a kernel commits to its drain barrier it waits
    for it under the same condition, before the CTA leaves its shared memory to another."""
    found = 0
    for name in ("gemm_tc.cu", "gemm_pair.cuh", "gemm_f64.cuh"):
        with open(os.path.join(CSRC, name)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"pdl_trigger\(\);\s*if \((leader|!ok)\) \{(.*?)mbar_wait\(drain_bar", text, re.S):
            body = m.group(2)
            assert len(re.findall(r"mma_commit(?:_pair)?\(drain_bar\)", body)) == 1
            guarded = re.search(r"if \(!ok\)\s*$", body) is not None  # the wait alone is conditional
            assert not guarded, name
            found += 1
        assert len(re.findall(r"mma_commit(?:_pair)?\(drain_bar\)", text)) == len(
            re.findall(r"mbar_wait\(drain_bar", text)), name
    assert found == 4
