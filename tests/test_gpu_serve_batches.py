"""The serving loop where a batch of admissions can go wrong: fewer slots than admitters, slots
that do not divide among them, one lane and a lane per warp, request counts that leave a batch
unfilled, and a ring shorter than the indices taken ahead.  Results against the oracle."""
import numpy as np
import pytest
import torch

from gpu_util import require_gpu
from oracle import calc
from paper_1110_4623_gb300 import inputs

pytestmark = pytest.mark.gpu

POOL = 1 << 21


@pytest.fixture(scope="module")
def pool():
    require_gpu()
    off, ln, p = inputs.serve_inputs(3001, POOL, seed=91, len_hi=1 << 16)
    return off, ln, p, torch.from_numpy(p).cuda()


@pytest.mark.parametrize("nslots,admitters", [(1, 8), (2, 3), (5, 2), (16, 2), (63, 8), (64, 1), (64, 16)])
@pytest.mark.parametrize("nreq,ring_slots", [(1, 2), (131, 64), (3001, 4096)])
def test_backlog_exact(pool, nslots, admitters, nreq, ring_slots):
    from paper_1110_4623_gb300 import runner
    off, ln, p, dp = pool
    r = runner.ServeRun(off[:nreq], ln[:nreq], np.zeros(nreq, dtype=np.int64), dp, nslots=nslots, nblocks=80,
                        admitters=admitters, chunk_elems=1024, ring_slots=ring_slots, drain_timeout_s=10).run()
    assert r["rc"] == 0, r["stats"]
    assert np.array_equal(r["res"], calc.serve_final(off[:nreq], ln[:nreq], p))
    chunks = int((-(-ln[:nreq] // 1024)).sum())
    assert r["stats"] == [nreq, chunks, nreq, 0]


@pytest.mark.parametrize("first,then", [(3001, 40), (300, 299), (40, 3001)])
def test_ring_with_an_earlier_calls_entries(pool, first, then):
    # One ring for two calls: entries of the longer one past the shorter one's must not be taken.
    from paper_1110_4623_gb300 import runner
    off, ln, p, dp = pool
    ring = None
    for n, start in ((first, 0), (then, 5 if then < first else 0)):
        idx = (np.arange(n) + start) % len(off)
        r = runner.ServeRun(off[idx], ln[idx], np.zeros(n, dtype=np.int64), dp, nslots=64, nblocks=80, admitters=8,
                            chunk_elems=1024, ring_slots=4096, drain_timeout_s=10)
        ring = r.ring = ring if ring is not None else r.ring
        got = r.run()
        assert got["rc"] == 0, got["stats"]
        assert np.array_equal(got["res"], calc.serve_final(off[idx], ln[idx], p))
        assert got["stats"][0] == n and got["stats"][2] == n
