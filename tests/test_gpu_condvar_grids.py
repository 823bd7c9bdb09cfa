"""The condition-variable queue on the ticket lock, on both sides of the grid from which the compact
form of its kernel runs: every item taken once, the sums exact."""
import numpy as np
import pytest

from gpu_util import require_gpu
from paper_1110_4623_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("blocks,threads", [(16, 128), (1520, 128), (1536, 128), (2432, 128), (4864, 32)])
def test_ticket_queue_exact(blocks, threads):
    from paper_1110_4623_gb300 import runner
    require_gpu()
    half = blocks // 2
    value = inputs.condvar_inputs(half, blocks)
    got = runner.CondVarRun(half, half, 1, 32, value, block_threads=threads, bo=runner.backoff(min_ns=64, max_ns=2000),
                            mutex="ticket").run()
    assert got["rc"] == 0 and got["status"] == 0, got["status"]
    assert (got["seen"] == 1).all() and (got["count"] == 1).all()
    assert int(got["sum"].sum()) == int(value.view(np.int32).astype(np.int64).sum())
