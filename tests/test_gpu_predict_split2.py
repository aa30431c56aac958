"""Kriging on both sides of 2,432 new locations, where 32 threads per location take over from a CTA
per location, against the oracle: the bar of test_gpu_predict_split.py."""
import numpy as np
import pytest

import egs_inputs as ei
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("theta", [(1.0, 0.1, 0.5), (1.3, 0.05, 1.2)])
@pytest.mark.parametrize("m", [2431, 2432])
def test_predict_split(m, theta):
    import torch
    import paper_1708_02835_gb300 as egs
    from gpu_util import locs_dev, dev
    n = 300
    p = ei.Problem(n=n, theta=theta, seed=4)
    locs = p.locations()
    z = oracle.simulate_z(locs, theta, p.e())
    new = np.random.default_rng(m).uniform(0.0, 1.0, (2, m))
    new[:, -1] = locs[:, 7]
    ref = oracle.predict(locs, z, new, theta)
    out = torch.full((m,), float("nan"), dtype=torch.float64, device="cuda")
    egs.egs_predict(locs_dev(locs), dev(z), n, locs_dev(new), m, theta, out)
    assert np.max(np.abs(out.cpu().numpy() - ref)) <= 1e-9 * np.max(np.abs(z))
