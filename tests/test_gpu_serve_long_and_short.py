"""One long request and many short ones on few slots: the short ones go through the slots that are
left, and finish before the long one does.  (30,000 chunks of a few microseconds each on three
workers, against 200 requests of one chunk.)"""
import numpy as np
import pytest
import torch

from gpu_util import require_gpu
from oracle import calc

pytestmark = pytest.mark.gpu

CHUNK, LONG = 1024, 30_000 * 1024


@pytest.fixture(scope="module")
def pool():
    require_gpu()
    p = np.random.default_rng(3).integers(-1000, 1000, LONG + 4096, dtype=np.int32)
    return p, torch.from_numpy(p).cuda()


@pytest.mark.parametrize("nslots,admitters", [(7, 1), (7, 2), (4, 1), (2, 1), (7, 7), (3, 8)])
@pytest.mark.parametrize("at", [0, 1])
def test_short_requests_pass_a_long_one(pool, nslots, admitters, at):
    from paper_1110_4623_gb300 import runner
    p, dp = pool
    n = 200
    ln = np.full(n, CHUNK, dtype=np.int64)
    ln[at] = LONG
    off = np.arange(n, dtype=np.int64) * 7
    r = runner.ServeRun(off, ln, np.zeros(n, dtype=np.int64), dp, nslots=nslots, nblocks=admitters + 3,
                        admitters=admitters, chunk_elems=CHUNK, ring_slots=1024).run()
    assert r["rc"] == 0 and r["stats"][3] == 0, r["stats"]
    assert np.array_equal(r["res"], calc.serve_final(off, ln, p))
    lat = r["latency_ns"]
    assert np.delete(lat, at).max() < lat[at] / 2, (np.delete(lat, at).max(), lat[at])
