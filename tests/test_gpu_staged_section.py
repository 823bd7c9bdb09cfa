"""Critical sections around the lines between the narrow, the wide and the staged kernel, and around
the staged one's passes, from data on and off a 16-byte boundary: exact final data."""
import numpy as np
import pytest
import torch

from gpu_util import require_gpu
from oracle import calc
from paper_1110_4623_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,cluster", [("ticket", 0), ("cluster_mcs", 8), ("cas_backoff", 0)])
@pytest.mark.parametrize("threads,cs_words", [(32, 256), (32, 257), (32, 511), (32, 512), (32, 513), (32, 1027),
                                              (64, 2050), (128, 1026), (256, 2049), (256, 9001)])
@pytest.mark.parametrize("shift", [0, 1])
def test_section_exact(kind, cluster, threads, cs_words, shift):
    from paper_1110_4623_gb300 import gsync as G, runner
    require_gpu()
    delay, add = inputs.mutex_inputs(24, 3, threads + cs_words, max_delay=200)
    run = runner.MutexRun(kind, 24, threads, 3, cs_words, delay, add, cluster=cluster)
    guard = torch.full((cs_words + 8,), 7, dtype=torch.int32, device="cuda")
    assert guard.data_ptr() % 16 == 0
    guard[shift:shift + cs_words] = 0
    run.work.data = guard.data_ptr() + 4 * shift
    run.reset()
    G.check("gsync_bench_mutex", run.launch())
    got = run.results()
    want = calc.mutex_final(24, 3, cs_words, add)
    assert got["status"] == 0 and got["total"] == want["total"]
    data = guard.cpu().numpy().view(np.uint32)
    assert np.array_equal(data[shift:shift + cs_words], want["data"])
    assert (data[:shift] == 7).all() and (data[shift + cs_words:] == 7).all()
