"""Workers and a long request when many slots are active: a worker leaves a request after a bounded
run of its chunks, so that the short requests beside a long one go on.  Results are exact around
the length of that run."""
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
    p = np.random.default_rng(4).integers(-1000, 1000, LONG + 4096, dtype=np.int32)
    return p, torch.from_numpy(p).cuda()


def serve(pool, ln, nslots, admitters, workers):
    from paper_1110_4623_gb300 import runner
    p, dp = pool
    n = len(ln)
    off = np.arange(n, dtype=np.int64) * 7 % 4096
    r = runner.ServeRun(off, ln, np.zeros(n, dtype=np.int64), dp, nslots=nslots, nblocks=admitters + workers,
                        admitters=admitters, chunk_elems=CHUNK, ring_slots=4096).run()
    assert r["rc"] == 0 and r["stats"][3] == 0, r["stats"]
    assert np.array_equal(r["res"], calc.serve_final(off, ln, p))
    assert r["stats"][1] == int((-(-ln // CHUNK)).sum())
    return r["latency_ns"]


@pytest.mark.parametrize("nslots,admitters,workers,n", [(16, 1, 3, 200), (64, 8, 3, 600), (64, 16, 16, 3000)])
def test_short_requests_pass_a_long_one(pool, nslots, admitters, workers, n):
    ln = np.full(n, CHUNK, dtype=np.int64)
    ln[0] = LONG
    lat = serve(pool, ln, nslots, admitters, workers)
    assert lat[1:].max() < lat[0] / 2, (lat[1:].max(), lat[0])


@pytest.mark.parametrize("chunks", [1, 2, 15, 16, 17, 31, 32, 33, 47, 48, 49])
@pytest.mark.parametrize("workers", [1, 5])
def test_runs_of_chunks_exact(pool, chunks, workers):
    serve(pool, np.full(150, chunks * CHUNK - 3, dtype=np.int64), 16, 2, workers)
