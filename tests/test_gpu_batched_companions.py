"""A problem's value in an FP64 batch does not depend on its companions: with tiles up to 256 every l
equals the single evaluation's with the same tile bit for bit, problems of more than 2,048 rows and
smaller ones in one batch, in a plan (run and replay) and in the one-call form, and a problem that is not positive definite
leaves the others alone on both routes."""
import numpy as np
import pytest

import egs_inputs as ei

pytestmark = pytest.mark.gpu

SIZES = [130, 2049, 1, 64, 700, 2500, 2048, 63]


@pytest.mark.parametrize("tile", [64, 128, 192, 256])
def test_every_value_equals_the_single_evaluation(tile):
    import paper_1708_02835_gb300 as egs
    from gpu_util import locs_dev, dev
    rng = np.random.default_rng(tile)
    probs = [ei.Problem(n=n, theta=(1.0, 0.08, 0.5), seed=70 + k, origin=(0.1, 0.2), side=0.7) for k, n in enumerate(SIZES)]
    th = np.array([(rng.uniform(0.5, 2.0), rng.uniform(0.03, 0.12), [0.5, 1.5, 0.8][k % 3]) for k in range(len(SIZES))])
    dl, dz = [locs_dev(p.locations()) for p in probs], [dev(p.e()) for p in probs]
    want = [egs.egs_loglik_ex(dl[i], dz[i], tuple(th[i]), n, "fp64", tile=tile)[0] for i, n in enumerate(SIZES)]
    B = egs.egs_batch(SIZES, tile=tile)
    assert B.tasks > 0
    for _ in range(2):
        out, stat = B.run(dl, dz, th)
        assert np.all(stat == 0) and list(out) == want
    for bad in (4, 5):
        t2 = th.copy()
        t2[bad] = (1.0, 5.0, 4.2)  # singular in FP64
        out, stat = B.run(dl, dz, t2)
        assert stat[bad] == egs.EGS_ERR_NOT_PD and np.isnan(out[bad])
        assert [v for i, v in enumerate(out) if i != bad] == [v for i, v in enumerate(want) if i != bad]
    B.close()
    if tile == 128:  # the default tile of a batch with a problem of more than 2,048 rows
        out, _ = egs.egs_loglik_batched(dl, dz, th, SIZES)
        assert list(out) == want
