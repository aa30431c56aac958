"""An infinite, NaN, zero or negative pivot is reported as a failed one in its own row, wherever it
stands in a block, a tile or the matrix, on both sides of the tensor cores' rule."""
import pytest

import egs_inputs as ei

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,b", [(100, 64), (500, 128), (2100, 128), (1500, 320)])
@pytest.mark.parametrize("what", [float("inf"), float("-inf"), float("nan"), 0.0, -1.0])
def test_failed_pivot(n, b, what):
    import torch
    import paper_1708_02835_gb300 as egs
    from gpu_util import locs_dev
    locs = locs_dev(ei.jittered_grid(n, seed=1))
    for pos in (0, 3, 4, 63, 64, n - 1):
        t = torch.zeros(egs.egs_tiles_bytes(n, b) // 8, dtype=torch.float64, device="cuda")
        egs.egs_matern_tiles(locs, n, (1.0, 0.05, 0.5), b, t)
        i, r = divmod(pos, b)
        t.view(-1, b, b)[i * (i + 3) // 2, r, r] = what
        with pytest.raises(egs.NotPositiveDefinite) as e:
            egs.egs_potrf_tiles(t, n, b)
        assert str(e.value).endswith("at row %d" % pos), (pos, str(e.value))
