"""FP64 evaluations at the limit of their workspace: with exactly egs_loglik_workspace_bytes the
tensor-core update runs; with less, but enough for the matrix, the call takes the DFMA update and
gives the same value to rounding (two FP64 factorisations: |dl| <= 1e-10 |l|, the FP64 bar); with
less than that it is refused.  Sizes: the smallest problem that takes the tensor cores, a ragged
one with several tiles, one that never takes them (no smaller route)."""
import pytest

import egs_inputs as ei

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tile", [(2049, 256), (2500, 320), (1000, 128)])
def test_fp64_workspace_limits(n, tile):
    import torch
    import paper_1708_02835_gb300 as egs
    from gpu_util import locs_dev, dev
    theta = (1.0, 0.1, 0.8)
    p = ei.Problem(n=n, theta=theta, seed=2)
    locs, z = locs_dev(p.locations()), dev(p.e())
    need = egs.egs_loglik_workspace_bytes(n, tile, "fp64", 2)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    full, _ = egs.egs_loglik_ex(locs, z, theta, n, "fp64", tile=tile, workspace=ws)
    assert full == egs.egs_loglik_ex(locs, z, theta, n, "fp64", tile=tile)[0]
    less = torch.empty(need - 256, dtype=torch.uint8, device="cuda")
    if n > 2048:
        ll, _ = egs.egs_loglik_ex(locs, z, theta, n, "fp64", tile=tile, workspace=less)
        assert abs(ll - full) <= 1e-10 * abs(full)
    else:
        with pytest.raises(egs.EgsError) as e:
            egs.egs_loglik_ex(locs, z, theta, n, "fp64", tile=tile, workspace=less)
        assert e.value.status == egs.EGS_ERR_ARG
    tiny = torch.empty(need // 4, dtype=torch.uint8, device="cuda")
    with pytest.raises(egs.EgsError) as e:
        egs.egs_loglik_ex(locs, z, theta, n, "fp64", tile=tile, workspace=tiny)
    assert e.value.status == egs.EGS_ERR_ARG
