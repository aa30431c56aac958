"""The independent-blocks approximation with one block is the exact FP64 evaluation with that tile, bit
for bit at every tile and on both sides of the tensor cores' rule, with the same diagnostics (band:
the super tile), and a matrix that is not positive definite is reported with its row."""
import pytest

import egs_inputs as ei

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tile,st", [(700, 128, 6), (700, 320, 3), (1900, 512, 4), (900, 1024, 1), (2300, 320, 8),
                                       (2100, 128, 17)])
def test_one_block_is_the_exact_evaluation(n, tile, st):
    import paper_1708_02835_gb300 as egs
    from gpu_util import locs_dev, dev
    theta = (1.1, 0.07, 0.8)
    p = ei.Problem(n=n, theta=theta, seed=n)
    locs, z = locs_dev(p.locations()), dev(p.e())
    one, info = egs.egs_loglik_ind(locs, z, theta, n, tile=tile, super_tiles=st)
    exact, want = egs.egs_loglik_ex(locs, z, theta, n, "fp64", tile=tile)
    assert one == exact
    assert info == dict(want, band=st)
    with pytest.raises(egs.NotPositiveDefinite) as e:
        egs.egs_loglik_ind(locs, z, (1.0, 5.0, 4.2), n, tile=tile, super_tiles=st)
    assert "egs_loglik_ind" in str(e.value) and "row" in str(e.value)
