"""The barrier workload's full fold, put together one round late: over any pattern of failed crossings
(a cluster's blocks go on after one) no half is read while the other warps write it, because the
pending round is put together at the failed crossing."""
import itertools
import os
import re

import pytest

from oracle import model_check as mc

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("warps", [1, 2, 3])
def test_every_pattern_of_failures_is_safe(warps):
    for ok in itertools.product((0, 1), repeat=5):
        r = mc.check(mc.FullFold(ok=ok), warps, 1)
        assert r.ok, (ok, r.violation)


@pytest.mark.parametrize("ok", [(1, 0, 1), (1, 1, 0, 1, 1), (0, 1, 0, 1)])
def test_pending_round_kept_over_a_failure_is_caught(ok):
    r = mc.check(mc.FullFold(ok=ok, broken="kept_pending"), 2, 1)
    assert not r.ok and "put together" in r.violation


def test_kernel_folds_at_the_failed_crossing():
    src = open(os.path.join(ROOT, "paper_1110_4623_gb300", "csrc", "bench_barrier.cu")).read()
    code = re.sub(r"//[^\n]*", "", src)
    failed = re.search(r"if \(rc != GSYNC_OK\) \{.*?continue;", code, re.S).group(0)
    assert re.search(r"if \(FULL && pend\) fold_round\(\(uint32_t\)r - 1u\);", failed)
    assert re.search(r"pend = false;", failed)


def test_full_fold_kernels_stay_in_registers(tmp_path):
    # Every acquire empties L1, so that a spilled register is an L2 round trip in a crossing.
    import subprocess

    from paper_1110_4623_gb300 import build
    out = subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-c", os.path.join(build.CSRC, "bench_barrier.cu"),
                          "-o", str(tmp_path / "b.o")], capture_output=True, text=True, check=True, timeout=600)
    text = out.stdout + out.stderr
    full = re.findall(r"Function properties for \S*barrier_workload_kernelILi(\d+)ELb1ELb0E\S*\n\s*"
                      r"(\d+) bytes stack frame, (\d+) bytes spill stores", text)
    assert sorted(int(k) for k, _, _ in full) == list(range(9))
    assert all(spill == "0" for _, _, spill in full), full
