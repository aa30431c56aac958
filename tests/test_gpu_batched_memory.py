"""A batch plan that fits the device only without the tensor-core update's slices is made without
them, as the other calls do; its values agree with single evaluations to the FP64 bar 1e-10.  The
device is filled by an ordinary allocation up to a little less than the plan with slices needs."""
import numpy as np
import pytest

import egs_inputs as ei

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [128, 320])
def test_plan_without_room_for_the_slices(tile):
    import torch
    import paper_1708_02835_gb300 as egs
    from gpu_util import locs_dev, dev
    ns, th = [6000, 500, 6000, 4000], (1.0, 0.05, 0.5)
    probs = [ei.Problem(n=n, theta=th, seed=k) for k, n in enumerate(ns)]
    dl, dz = [locs_dev(p.locations()) for p in probs], [dev(p.e()) for p in probs]
    want = [egs.egs_loglik_ex(l, z, th, n, "fp64", tile=tile)[0] for l, z, n in zip(dl, dz, ns)]
    B = egs.egs_batch(ns, tile=tile)
    full = B.workspace_bytes
    B.close()
    egs.egs_set_allocator(None, None)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - full + (20 << 20), dtype=torch.uint8, device="cuda")
    try:
        assert torch.cuda.mem_get_info()[0] < full
        B = egs.egs_batch(ns, tile=tile)
        assert B.workspace_bytes < full
        out, stat = B.run(dl, dz, np.array([th] * len(ns)))
        B.close()
    finally:
        del hog
        torch.cuda.empty_cache()
    assert np.all(stat == 0)
    for v, w in zip(out, want):
        assert abs(v - w) <= 1e-10 * abs(w)
