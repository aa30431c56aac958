"""The FP64 band rows of a mixed factorisation: X L^T = A leaves no larger a residual than a
substitution in FP64 does (LAPACK's, on the same L and A), for rough and for smooth fields, whose
diagonal tiles are ill-conditioned.  The first step's tiles are read from the caller's workspace,
which begins with the FP64 band (position i band + (i - j)); residuals in extended precision on a
sample of rows."""
import numpy as np
import pytest

import egs_inputs as ei

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "tf32"])
@pytest.mark.parametrize("tile,band", [(256, 2), (512, 2), (256, 3)])
@pytest.mark.parametrize("theta", [(1.0, 0.1, 0.5), (1.0, 0.2, 1.3), (1.0, 0.1, 2.5)])
def test_band_rows_residual(prec, tile, band, theta):
    import scipy.linalg as sla
    import torch
    import paper_1708_02835_gb300 as egs
    from gpu_util import locs_dev, dev
    n = (band + 2) * tile + 77
    p = ei.Problem(n=n, theta=theta, seed=6)
    locs, z = locs_dev(p.locations()), dev(p.e())
    ws = torch.zeros(egs.egs_loglik_workspace_bytes(n, tile, prec, band), dtype=torch.uint8, device="cuda")
    try:
        egs.egs_loglik_ex(locs, z, theta, n, prec, tile=tile, band=band, workspace=ws)
    except (egs.NotPositiveDefinite, egs.MixedInaccurate):
        pass  # a later tile; the first step is there
    torch.cuda.synchronize()
    sig = torch.zeros(egs.egs_tiles_bytes(n, tile, prec, band), dtype=torch.uint8, device="cuda")
    egs.egs_matern_tiles(locs, n, theta, tile, sig, precision=prec, band=band)
    bb = tile * tile
    count = band * band * bb
    F = ws[:count * 8].view(torch.float64).cpu().numpy().reshape(-1, tile, tile)
    S = sig[:count * 8].view(torch.float64).cpu().numpy().reshape(-1, tile, tile)
    L = np.tril(F[0])
    LD = np.longdouble
    for i in range(1, band):
        rows = np.random.default_rng(i).choice(tile, 24, replace=False)
        X, A = F[i * band + i][rows], S[i * band + i][rows]
        want = sla.solve_triangular(L, A.T, lower=True).T

        def rms(x):
            r = x.astype(LD) @ L.T.astype(LD) - A.astype(LD)
            return float(np.sqrt((r * r).mean()))

        got, sub = rms(X), rms(want)
        print("%s tile %d row %d theta %s: residual %.2e, substitution %.2e" % (prec, tile, i, theta, got, sub))
        assert 0.0 < got <= sub
