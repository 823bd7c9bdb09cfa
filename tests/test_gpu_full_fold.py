"""The full fold at its edges: fewer slots than a block's threads, as many, one more, several a
thread with a remainder; no round, one, two (both parities of the shares) and three."""
import numpy as np
import pytest

from gpu_util import require_gpu
from oracle import calc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,param", [("count", 8), ("exchange", 0), ("flag", 0), ("cluster", 4)])
@pytest.mark.parametrize("nblocks,threads", [(4, 64), (32, 32), (36, 32), (64, 64), (100, 32), (128, 96), (260, 64)])
@pytest.mark.parametrize("rounds", [0, 1, 2, 3, 40])
def test_full_fold_exact(kind, param, nblocks, threads, rounds):
    from paper_1110_4623_gb300 import runner
    require_gpu()
    run = runner.BarrierRun(kind, nblocks, threads, rounds, True, param=param)
    if rounds == 0:  # run() has no chk to shape
        run.mix.fill_(7)
        assert run.launch() == 0 and int(run.status.item()) == 0
        assert not run.mix.any() and not run.bad.any()
        return
    for _ in range(2):
        got = run.run()
        assert got["rc"] == 0 and got["status"] == 0, got["status"]
        assert not got["bad"].any()
        want = calc.barrier_full(nblocks, rounds)
        assert np.array_equal(got["chk"], want["chk"]) and np.array_equal(got["mix"], want["mix"])
