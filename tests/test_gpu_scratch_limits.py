"""FP64 calls on a device with room for the matrix but not for the tensor-core update's scratch: they
take the DFMA update and give the same results (1e-10, the FP64 bar; the factor as in
test_gpu_tc64.py).  The device is filled by an ordinary allocation."""
import numpy as np
import pytest

import egs_inputs as ei

pytestmark = pytest.mark.gpu


def test_calls_without_room_for_the_slices():
    import torch
    import paper_1708_02835_gb300 as egs
    from gpu_util import locs_dev, dev
    n, tile, m, theta = 6200, 1024, 50, (1.0, 0.05, 0.5)
    p = ei.Problem(n=n, theta=theta, seed=3)
    locs, z = locs_dev(p.locations()), dev(p.e())
    new = dev(np.random.default_rng(0).uniform(0, 1, 2 * m))
    tiles = torch.empty(egs.egs_tiles_bytes(n, tile) // 8, dtype=torch.float64, device="cuda")

    def run():
        out = {"l": egs.egs_loglik_ex(locs, z, theta, n, "fp64", tile=tile)[0]}
        zs, pr, y = torch.empty_like(z), torch.empty(m, dtype=torch.float64, device="cuda"), torch.empty_like(z)
        egs.egs_simulate(locs, z, theta, n, zs, tile=tile)
        egs.egs_predict(locs, z, n, new, m, theta, pr, tile=tile)
        egs.egs_matern_tiles(locs, n, theta, tile, tiles)
        egs.egs_potrf_tiles(tiles, n, tile)
        out["logdet"], out["quad"] = egs.egs_trsv_tiles(tiles, n, tile, z, y)
        return out, zs, pr

    need = egs.egs_loglik_workspace_bytes(n, tile, "fp64", 2)
    T = -(-n // tile)
    slices = 14 * (T - 1) * tile * tile
    want, zs0, pr0 = run()
    for room in (need - slices // 2, slices // 2):  # the whole call; the factorisation's own scratch
        egs.egs_set_allocator(None, None)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        hog = torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda")
        try:
            if room > slices:
                got, zs, pr = run()
            else:
                egs.egs_matern_tiles(locs, n, theta, tile, tiles)
                egs.egs_potrf_tiles(tiles, n, tile)
                y = torch.empty_like(z)
                got = dict(zip(("logdet", "quad"), egs.egs_trsv_tiles(tiles, n, tile, z, y)))
        finally:
            del hog
            torch.cuda.empty_cache()
        for k in got:
            assert abs(got[k] - want[k]) <= 1e-10 * abs(want[k]), (k, room)
        if room > slices:
            assert float((zs - zs0).abs().max()) <= 1e-10 * float(zs0.abs().max())
            assert float((pr - pr0).abs().max()) <= 1e-9 * float(z.abs().max())
