"""Tiles and workspaces of a caller that start 8 bytes past a 16-byte boundary: the factor and the
value are those of aligned memory -- bit for bit where the same kernels run (n <= 2,048), to
rounding where the tensor-core update gives way to the DFMA one (the bars of test_gpu_tc64.py and
of the FP64 parity tests).  Sizes: one tile, several, and both sides of the tensor cores' rule."""
import pytest

import egs_inputs as ei

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tile", [(100, 128), (1000, 128), (2048, 320), (2049, 256), (2500, 192)])
def test_odd_double_offsets(n, tile):
    import torch
    import paper_1708_02835_gb300 as egs
    from gpu_util import locs_dev, dev
    theta = (1.0, 0.05, 0.5)
    p = ei.Problem(n=n, theta=theta, seed=2)
    locs, z = locs_dev(p.locations()), dev(p.e())
    count = egs.egs_tiles_bytes(n, tile) // 8
    ref = torch.empty(count, dtype=torch.float64, device="cuda")
    odd = torch.empty(count + 1, dtype=torch.float64, device="cuda")[1:]
    assert ref.data_ptr() % 16 == 0 and odd.data_ptr() % 16 == 8
    egs.egs_matern_tiles(locs, n, theta, tile, ref)
    egs.egs_matern_tiles(locs, n, theta, tile, odd)
    assert torch.equal(ref, odd)
    egs.egs_potrf_tiles(ref, n, tile)
    egs.egs_potrf_tiles(odd, n, tile)
    y = torch.empty_like(z)
    assert egs.egs_trsv_tiles(odd, n, tile, z, y)[0] == pytest.approx(egs.egs_trsv_tiles(ref, n, tile, z, y)[0], rel=1e-10)
    T = -(-n // tile)
    low = [t for i in range(T) for t in range(i * (i + 1) // 2, i * (i + 1) // 2 + i)]  # below the diagonal
    a, b = ref.view(-1, tile, tile), odd.view(-1, tile, tile)
    diag = [i * (i + 3) // 2 for i in range(T)]
    for x, w in ((a[low], b[low]), (torch.tril(a[diag]), torch.tril(b[diag]))):
        if n <= 2048:
            assert torch.equal(x, w)
        else:
            assert bool((torch.abs(x - w) <= 1e-12 * torch.abs(x).max() + 1e-10 * torch.abs(x)).all())
    need = egs.egs_loglik_workspace_bytes(n, tile, "fp64", 2)
    ws = torch.empty(need + 8, dtype=torch.uint8, device="cuda")[8:]
    assert ws.data_ptr() % 16 == 8
    want, _ = egs.egs_loglik_ex(locs, z, theta, n, "fp64", tile=tile)
    got, _ = egs.egs_loglik_ex(locs, z, theta, n, "fp64", tile=tile, workspace=ws)
    assert got == want if n <= 2048 else abs(got - want) <= 1e-10 * abs(want)
