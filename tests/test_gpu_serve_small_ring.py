"""Bursts through rings shorter than what the producer would publish at once: the ring takes what it
has room for, and every result is exact."""
import numpy as np
import pytest
import torch

from gpu_util import require_gpu
from oracle import calc
from paper_1110_4623_gb300 import inputs

pytestmark = pytest.mark.gpu

POOL = 1 << 20


@pytest.mark.parametrize("ring_slots", [2, 4, 32, 64])
@pytest.mark.parametrize("nslots,admitters", [(1, 2), (64, 8), (64, 1), (6, 8)])
@pytest.mark.parametrize("nreq", [3, 65, 700])
def test_burst_exact(ring_slots, nslots, admitters, nreq):
    from paper_1110_4623_gb300 import runner
    require_gpu()
    off, ln, p = inputs.serve_inputs(nreq, POOL, seed=13, len_hi=1 << 14)
    r = runner.ServeRun(off, ln, np.zeros(nreq, dtype=np.int64), torch.from_numpy(p).cuda(), nslots=nslots, nblocks=40,
                        admitters=admitters, chunk_elems=1024, ring_slots=ring_slots, drain_timeout_s=10).run()
    assert r["rc"] == 0, r["stats"]
    assert np.array_equal(r["res"], calc.serve_final(off, ln, p))
    assert r["stats"][0] == nreq and r["stats"][2] == nreq
