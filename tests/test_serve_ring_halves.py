"""The serving ring's entry is read as the two 8-byte halves that it is written as: a half read by
two accesses can pair the new sequence number with the previous lap's value (the model shows it),
so the kernel reads an entry by 64-bit accesses only."""
import os
import re

import pytest

from oracle import model_check as mc

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("hi_first", [False, True])
def test_half_read_by_two_accesses_is_caught(hi_first):
    r = mc.check(mc.RingPublish(hi_first=hi_first, broken="torn_half"), 2, 3)
    assert not r.ok and "taken with" in r.violation


def test_kernel_reads_whole_halves():
    src = open(os.path.join(ROOT, "paper_1110_4623_gb300", "csrc", "serve.cu")).read()
    code = re.sub(r"//[^\n]*", "", src)
    assert "v4.u32" not in code and "ld_acquire_v4" not in code
    assert re.search(r"ld\.acquire\.sys\.global\.(v2\.u64|b128)", code)
