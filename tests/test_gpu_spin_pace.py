"""The CAS spin lock on both sides of the grid from which its attempts are paced, and the spin
semaphores whose posts fence before they swap: exact final state at the edges."""
import numpy as np
import pytest

from gpu_util import require_gpu
from oracle import calc
from paper_1110_4623_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nblocks,threads", [(1, 256), (660, 256), (679, 256), (680, 256), (699, 128), (1216, 256),
                                             (2400, 64)])
@pytest.mark.parametrize("cs_words", [0, 300])
def test_cas_spin_exact(nblocks, threads, cs_words):
    from paper_1110_4623_gb300 import runner
    require_gpu()
    delay, add = inputs.mutex_inputs(nblocks, 4, nblocks)
    got = runner.MutexRun("cas_spin", nblocks, threads, 4, cs_words, delay, add).run()
    want = calc.mutex_final(nblocks, 4, cs_words, add)
    assert got["rc"] == 0 and got["status"] == 0, got["status"]
    assert got["total"] == want["total"] and np.array_equal(got["data"], want["data"])
    assert calc.check_grant_log(got["log"], None, nblocks, 4, fifo=False) == []


@pytest.mark.parametrize("kind", ["spin", "spin_backoff"])
@pytest.mark.parametrize("nblocks,n", [(1, 1), (2, 1), (33, 1), (33, 2), (64, 64), (100, 99)])
def test_spin_semaphores_exact(kind, nblocks, n):
    from paper_1110_4623_gb300 import runner
    require_gpu()
    hold, add = inputs.sem_inputs(nblocks, 15, nblocks + n, 0, 900)
    bo = runner.backoff(min_ns=64, max_ns=4096) if kind == "spin_backoff" else None
    got = runner.SemRun(kind, nblocks, 64, 15, n, hold, add, bo=bo, timeout_ns=20_000_000_000).run()
    want = calc.sem_final(nblocks, 15, n, add)
    assert got["rc"] == 0 and got["status"] == 0, got["status"]
    assert np.array_equal(got["count"], want["count"]) and got["tally"] == want["tally"]
    assert got["occupancy"] == 0 and 1 <= got["max_occ"] <= n
    assert n > 1 or got["total"] == want["total"]
