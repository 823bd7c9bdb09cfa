"""Group barriers of 256-thread blocks in clusters, whose state waits in shared memory between
crossings: groups of one cluster and of many, blocks in no group, no crossing at all, launches one
after another on one group state, and every block's slot checks against the oracle, also beside
blocks of 128 and 129 to 256 threads on the same state."""
import numpy as np
import pytest

from gpu_util import require_gpu
from oracle import calc
from paper_1110_4623_gb300 import autotune, inputs

pytestmark = pytest.mark.gpu

NKEYS = 300
POLICY = [("cluster_die_carry", 0, 0), ("cluster", 128, 4000), ("ticket_carry", 64, 2000)]


def check(run, keys, adds, rounds):
    got = run.run()
    want = calc.batched_final(keys, adds, NKEYS)
    assert got["rc"] == 0 and got["status"] == 0, got["status"]
    assert np.array_equal(got["sum"], want["sum"]) and np.array_equal(got["count"], want["count"])
    assert not got["bad"].any()
    for st, sz in zip(run.group_start, run.group_sizes):
        assert np.array_equal(got["mix"][st:st + sz], calc.barrier_sampled(int(sz), rounds)["mix"])
    assert not got["mix"][int(run.group_sizes.sum()):].any()


@pytest.mark.parametrize("cluster,sizes", [(2, [2, 6, 16]), (4, [8, 4, 12, 4]), (8, [8, 24])])
@pytest.mark.parametrize("rounds", [0, 1, 2, 7, 90])
@pytest.mark.parametrize("nacq", [17, 40 * 33])
def test_slot_checks_exact(cluster, sizes, rounds, nacq):
    from paper_1110_4623_gb300 import gsync as G, runner
    require_gpu()
    keys, adds, _ = inputs.batched_inputs(nacq, NKEYS, 0.9, seed=nacq + rounds)
    cls = autotune.classify_keys(keys, NKEYS, 40)
    state = None
    for threads in (256, 128, 160, 256):
        run = runner.BatchedRun(keys, adds, NKEYS, 40, np.array(sizes), rounds, cls, 3, block_threads=threads,
                                cluster=cluster)
        run.set_policy(POLICY)
        if state is None:
            state = run.group_state
        run.work.group_state = G.ptr(state)
        for _ in range(2):
            check(run, keys, adds, rounds)
