"""Waits that can give up, followed by warp-collective instructions (source check,
on the CPU: the failure it excludes would be a hang).

In the prompt kernels a failed wait ends its role's loop.  tcgen05.ld / .st, votes
and shuffles of the rest of the loop need every lane of the warp, so whether a wait
failed is decided by the warp as a whole: each mb_wait sits inside __all_sync.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2309_08168_gb300", "csrc")


@pytest.mark.parametrize("name", ["tc_gemm.cuh", "prefill.cu"])
def test_waits_are_decided_by_the_warp(name):
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    calls = [m.start() for m in re.finditer(r"\bmb_wait\(", src) if not src[:m.start()].endswith("bool ")]
    assert len(calls) >= 4
    for at in calls:
        before = src[max(0, at - 64):at].replace("tc::", "")
        assert before.endswith("__all_sync(0xffffffffu, "), src[max(0, at - 40):at + 60]
