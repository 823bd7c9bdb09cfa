"""The batched kernel's staged acquisitions at the edges of a batch of 32: blocks with 0, 1, 31,
32, 33, 64 and 65 acquisitions, blocks of one warp (which stages for itself) and of more, without
and with clusters, crossings in between, and a key out of range."""
import numpy as np
import pytest

from gpu_util import require_gpu
from oracle import calc
from paper_1110_4623_gb300 import autotune, inputs

pytestmark = pytest.mark.gpu

NBLOCKS, NKEYS = 24, 50
POLICIES = {1: [("ticket", 0, 0), ("ticket_carry", 64, 2000), ("cas_spin", 0, 0)],
            8: [("cluster_die_carry", 0, 0), ("cluster", 128, 4000), ("ticket_carry", 0, 0)]}


def make(nacq, threads, cluster, keys=None):
    k, adds, _ = inputs.batched_inputs(nacq, NKEYS, 0.8, seed=nacq)
    keys = k if keys is None else keys
    run = autotune.make_run(keys, adds, NKEYS, NBLOCKS, 3, 7, cluster,
                            autotune.classify_keys(np.minimum(keys, NKEYS - 1), NKEYS, NBLOCKS), block_threads=threads)
    run.set_policy(POLICIES[cluster])
    return run, keys, adds


@pytest.mark.parametrize("cluster", [1, 8])
@pytest.mark.parametrize("threads", [32, 64, 256])
@pytest.mark.parametrize("nacq", [10, 24, 31 * 24, 32 * 24, 32 * 24 + 1, 33 * 24, 64 * 24 + 5, 65 * 24])
def test_batch_edges_exact(nacq, threads, cluster):
    require_gpu()
    run, keys, adds = make(nacq, threads, cluster)
    want = calc.batched_final(keys, adds, NKEYS)
    for _ in range(2):
        got = run.run()
        assert got["rc"] == 0 and got["status"] == 0, got["status"]
        assert np.array_equal(got["sum"], want["sum"]) and np.array_equal(got["count"], want["count"])
        assert not got["bad"].any()


@pytest.mark.parametrize("at", [0, 31 * 24, 40 * 24 + 3])
def test_key_out_of_range_is_reported(at):
    from paper_1110_4623_gb300 import gsync as G
    require_gpu()
    keys = inputs.batched_inputs(45 * 24, NKEYS, 0.8, seed=5)[0].copy()
    keys[at] = NKEYS
    run, _, _ = make(45 * 24, 64, 1, keys)
    got = run.run()
    assert got["rc"] == 0 and got["status"] & G.GSYNC_STATUS_VIOLATION


def test_group_state_serves_other_groups_and_cluster_launches():
    # One buffer of group barriers, never zeroed: launches with other group sizes and of the other
    # kind of group barrier, one after another.
    from paper_1110_4623_gb300 import gsync as G, runner
    require_gpu()
    keys, adds, _ = inputs.batched_inputs(40 * 32, NKEYS, 0.8, seed=11)
    cls = autotune.classify_keys(keys, NKEYS, 32)
    want = calc.batched_final(keys, adds, NKEYS)
    state = None
    for sizes, cluster in (([5, 9, 18], 1), ([8, 16, 8], 8), ([1, 30, 1], 1), ([16, 16], 1), ([24, 8], 8), ([7, 7, 7], 1)):
        run = runner.BatchedRun(keys, adds, NKEYS, 32, np.array(sizes), 13, cls, 3, block_threads=64, cluster=cluster)
        run.set_policy(POLICIES[1] if cluster == 1 else POLICIES[8])
        if state is None:
            state = run.group_state
        run.work.group_state = G.ptr(state)
        for _ in range(2):
            got = run.run()
            assert got["rc"] == 0 and got["status"] == 0, (sizes, got["status"])
            assert np.array_equal(got["sum"], want["sum"]) and np.array_equal(got["count"], want["count"])
            assert not got["bad"].any()
