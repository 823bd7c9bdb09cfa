"""The serving slot's claim word: a claim and the chunk count that it is judged by come from one
64-bit access.  The model with the word in one access is safe and live, also where workers keep
their request; with its halves read or published by two accesses it is not; and the kernel reads,
adds to and publishes the word in 64-bit accesses only."""
import os
import re

import pytest

from oracle import model_check as mc

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("nch,nproc", [((1, 2), 4), ((2, 1), 4), ((3, 2), 3), ((2, 1, 2), 3)])
def test_kept_claims_are_safe_and_live(nch, nproc):
    r = mc.check(mc.ServeSlot(nch=nch, keep=True), nproc, 1)
    assert r.ok, r.violation


@pytest.mark.parametrize("broken", ["torn_publish", "torn_look"])
@pytest.mark.parametrize("nch", [(1, 2), (2, 1)])
def test_word_in_two_accesses_is_caught(broken, nch):
    r = mc.check(mc.ServeSlot(nch=nch, broken=broken), 3, 1)
    assert not r.ok and r.violation


def test_kernel_accesses_the_word_whole():
    src = open(os.path.join(ROOT, "paper_1110_4623_gb300", "csrc", "serve.cu")).read()
    code = re.sub(r"//[^\n]*", "", src)
    assert re.search(r"uint64_t claim;", code)
    uses = re.findall(r"[^\n]*->\s*claim\b[^\n]*", code)
    assert len(uses) >= 4
    for line in uses:
        assert re.search(r"(ld_relaxed|atom_add_acquire|atom_add_relaxed|st_release)_u64\(&\w+->claim\b", line), line
