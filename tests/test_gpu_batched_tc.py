"""Batches on the tensor cores: a batch whose largest problem has more than 2,048 rows factors
all its problems there, step by step, and so does the independent-blocks approximation.

Sizes of one row, of less than a tile, at the edges of tiles and with every number of tiles,
unsorted.  Every l against the oracle within the FP64 bar 1e-10; problems of more than 2,048
rows equal the single evaluation bit for bit (the same kernels on the same blocks); a replay
equals the first run; a problem that is not positive definite does not disturb the others."""
import numpy as np
import pytest

import egs_inputs as ei
import oracle

pytestmark = pytest.mark.gpu

SIZES = [130, 2049, 1, 64, 700, 2500, 257, 512, 63]


@pytest.fixture(scope="module")
def egs():
    import paper_1708_02835_gb300 as m
    m.load_library()
    return m


@pytest.mark.parametrize("tile", [64, 128, 192, 320, 512])
def test_tc_batch(egs, tile):
    from gpu_util import locs_dev, dev
    rng = np.random.default_rng(tile)
    probs = []
    for k, n in enumerate(SIZES):
        th = (float(rng.uniform(0.5, 2.0)), float(rng.uniform(0.03, 0.12)), [0.5, 1.5, 0.8][k % 3])
        p = ei.Problem(n=n, theta=th, seed=50 + k, origin=(0.1, 0.2), side=0.7)
        locs = p.locations()
        probs.append((n, th, locs, oracle.simulate_z(locs, th, p.e()) if n > 1 else p.e()))
    B = egs.egs_batch(SIZES, tile=tile)
    dl, dz = [locs_dev(p[2]) for p in probs], [dev(p[3]) for p in probs]
    thetas = np.array([p[1] for p in probs])
    out, stat = B.run(dl, dz, thetas)
    assert np.all(stat == 0)
    for i, (n, th, locs, z) in enumerate(probs):
        ref = oracle.loglik(locs, z, th)["loglik"]
        assert abs(out[i] - ref) <= 1e-10 * max(1.0, abs(ref)), (i, n, out[i], ref)
        if n > 2048:
            assert out[i] == egs.egs_loglik_ex(dl[i], dz[i], th, n, "fp64", tile=tile)[0]
    assert np.array_equal(B.run(dl, dz, thetas)[0], out)
    bad = thetas.copy()
    bad[5] = (1.0, 5.0, 4.2)  # singular in FP64
    got, stat = egs.egs_batch(SIZES, tile=tile).run(dl, dz, bad)
    assert stat[5] == egs.EGS_ERR_NOT_PD and np.isnan(got[5])
    keep = np.arange(len(SIZES)) != 5
    assert np.array_equal(got[keep], out[keep])
    B.close()


@pytest.mark.parametrize("n,tile,st", [(1000, 64, 1), (2111, 64, 3), (1500, 128, 8)])
def test_ind_blocks(egs, n, tile, st):
    from gpu_util import locs_dev, dev
    th = (1.2, 0.08, 0.7)
    p = ei.Problem(n=n, theta=th, seed=3)
    locs, z = p.locations(), p.e()
    ref = oracle.loglik_ind(locs, z, th, st * tile)["loglik"]
    dev_ll, _ = egs.egs_loglik_ind(locs_dev(locs), dev(z), th, n, tile=tile, super_tiles=st)
    host_ll, _ = egs.egs_loglik_ind(np.ascontiguousarray(locs.reshape(-1)), np.ascontiguousarray(z), th, n, tile=tile,
                                    super_tiles=st)
    assert abs(dev_ll - ref) <= 1e-10 * abs(ref) and host_ll == dev_ll
