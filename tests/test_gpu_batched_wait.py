"""Failure detection of batches with problems on the tensor cores: a task whose completion is
withheld -- the first and the last of the tensor-core steps, and one of the persistent launch beside
them -- makes the bounded waits run out, the run returns EGS_ERR_TIMEOUT, and the next ordinary run
of the same batch gives the values of the first."""
import time

import numpy as np
import pytest

import egs_inputs as ei

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,tile", [([2100, 300, 2500], 128), ([2100, 2500], 256), ([2100, 300], 512)])
def test_withheld_step_times_out_then_recovers(sizes, tile):
    import paper_1708_02835_gb300 as egs
    from gpu_util import locs_dev, dev
    th = np.array([(1.0, 0.08, 0.5)] * len(sizes))
    probs = [ei.Problem(n=n, theta=(1.0, 0.08, 0.5), seed=k) for k, n in enumerate(sizes)]
    dl, dz = [locs_dev(p.locations()) for p in probs], [dev(p.e()) for p in probs]
    B = egs.egs_batch(sizes, tile=tile)
    steps = sum(-(-n // tile) - 1 for n in sizes if n > 2048 or tile > 256)
    assert B.tasks >= steps > 0 and (B.tasks > steps) == (tile <= 256 and min(sizes) <= 2048)
    want, _ = B.run(dl, dz, th)
    for task in {0, B.tasks - steps, B.tasks - 1}:
        B.set_wait_limit(20_000_000, withhold_task=task)
        t0 = time.time()
        with pytest.raises(egs.EgsError) as e:
            B.run(dl, dz, th)
        assert e.value.status == egs.EGS_ERR_TIMEOUT and time.time() - t0 < 2.0
        B.set_wait_limit(10_000_000_000, withhold_task=-1)
        got, stat = B.run(dl, dz, th)
        assert np.all(stat == 0) and np.array_equal(got, want)
    with pytest.raises(egs.EgsError) as e:
        B.set_wait_limit(1_000_000, withhold_task=B.tasks)
    assert e.value.status == egs.EGS_ERR_ARG
    B.close()
