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
