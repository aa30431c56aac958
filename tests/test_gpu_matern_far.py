"""Covariances at distances of hundreds of ranges and more (a short range, coordinates in other
units): both sides of x = r / theta2 = 640 and of 708, where e^-x leaves the normal doubles, far
beyond, and a squared distance that overflows.  Up to 708 against SciPy's scaled Bessel function:
1e-12 relative (x 2^-53 of x itself, 8e-14, twice, and SciPy's own error); from there 0, or at most
the smallest normal numbers.  Through egs_matern_tiles and egs_predict."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

XS = [1.0, 500.0, 639.0, 641.0, 700.0, 707.0, 709.0, 1279.0, 1281.0, 1e5, 1e150, 1e200]


def _want(x, theta):
    from scipy.special import gamma, kve
    th1, _, nu = theta
    x = np.asarray(x)
    lead = {0.5: 1.0 + 0 * x, 1.5: 1.0 + x, 2.5: 1.0 + x + x * x / 3.0}.get(nu)
    if lead is None:
        lead = 2.0 ** (1.0 - nu) / gamma(nu) * x ** nu * kve(nu, x)
    return th1 * lead * np.exp(-x)


@pytest.mark.parametrize("nu", [0.5, 0.8, 1.5, 1.3, 2.5])
def test_far_covariances(nu):
    import torch
    import paper_1708_02835_gb300 as egs
    from gpu_util import dev
    theta = (1.7, 0.001, nu)
    n, b = len(XS) + 1, 64
    xy = np.zeros((2, n))
    xy[0, 1:] = np.array(XS) * theta[1]
    tiles = torch.full((egs.egs_tiles_bytes(n, b) // 8,), float("nan"), dtype=torch.float64, device="cuda")
    egs.egs_matern_tiles(dev(xy.reshape(-1)), n, theta, b, tiles)
    got = tiles.cpu().numpy().reshape(b, b)[1:n, 0]
    x = np.abs(xy[0, 1:]) / theta[1]
    near = x < 708.0
    want = _want(x[near], theta)
    assert np.all(np.abs(got[near] - want) <= 1e-12 * want)
    assert np.all(got[~near] >= 0.0) and np.all(got[~near] <= 1e-300)

    # kriging: new locations that far from every observed one
    m = 64
    r = np.random.default_rng(1)
    obs = r.uniform(0.0, 1e-4, (2, m)) + np.arange(m) * 3e-3
    z = r.standard_normal(m)
    new = np.array([[1e3, 1e150, 1e200, obs[0, 0] - 0.66], [0.0, 0.0, 1e200, obs[1, 0]]])
    out = torch.full((4,), float("nan"), dtype=torch.float64, device="cuda")
    egs.egs_predict(dev(obs.reshape(-1)), dev(z), m, dev(new.reshape(-1)), 4, theta, out)
    got = out.cpu().numpy()
    assert np.all(np.isfinite(got)) and np.all(got[:3] == 0.0) and abs(got[3]) <= 1e-200
