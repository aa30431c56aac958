"""Kriging at the numbers of new locations where the split of the work changes (a CTA per
location up to 303, 32 threads up to 9,727, 8 beyond) and with the local polynomials of a
general smoothness, against the oracle: |z_gpu - z_oracle| <= 1e-9 max|Z| (the FP64 bar of
the kriging tests).  New locations on top of observed ones (r = 0) and far away (C = 0)."""
import numpy as np
import pytest

import egs_inputs as ei
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("theta", [(1.0, 0.1, 0.5), (1.3, 0.05, 1.2)])
@pytest.mark.parametrize("m", [1, 303, 304, 9727, 9728])
def test_predict_split(m, theta):
    import torch
    import paper_1708_02835_gb300 as egs
    from gpu_util import locs_dev, dev
    n = 300
    p = ei.Problem(n=n, theta=theta, seed=4)
    locs = p.locations()
    z = oracle.simulate_z(locs, theta, p.e())
    new = np.random.default_rng(m).uniform(0.0, 1.0, (2, m))
    new[:, 0] = locs[:, 7]
    new[:, m // 2] = 400.0 if m > 2 else new[:, m // 2]
    ref = oracle.predict(locs, z, new, theta)
    out = torch.full((m,), float("nan"), dtype=torch.float64, device="cuda")
    egs.egs_predict(locs_dev(locs), dev(z), n, locs_dev(new), m, theta, out)
    assert np.max(np.abs(out.cpu().numpy() - ref)) <= 1e-9 * np.max(np.abs(z))
