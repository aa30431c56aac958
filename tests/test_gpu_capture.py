"""egs_matern_tiles, which is asynchronous, inside a CUDA graph capture: as the library's very first
call (nothing of it exists yet) and later, with the allocation of the polynomials' scratch (general
nu) and without, in both layouts; a replay equals the direct call bit for bit.  Each in a process of
its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = """
import sys, torch
sys.path.insert(0, %r)
import egs_inputs as ei, paper_1708_02835_gb300 as egs
egs.load_library()
n, tile = 1000, 256
locs = torch.as_tensor(ei.jittered_grid(n, seed=1).reshape(-1).copy()).cuda()
prec, nu = sys.argv[1], float(sys.argv[2])
out = torch.zeros(egs.egs_tiles_bytes(n, tile, prec, 2) // 8, dtype=torch.float64, device="cuda")
torch.cuda.synchronize()
""" % ROOT

CAPTURE = HEAD + """
for _ in range(2):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        egs.egs_matern_tiles(locs, n, (1.0, 0.1, nu), tile, out, precision=prec, band=2)
    out.zero_()
    g.replay()
    g.replay()
    torch.cuda.synchronize()
    got = out.clone()
    out.zero_()
    egs.egs_matern_tiles(locs, n, (1.0, 0.1, nu), tile, out, precision=prec, band=2)
    torch.cuda.synchronize()
    assert torch.equal(got, out) and float(out.abs().max()) == 1.0
print("fine")
"""

@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("nu", [0.8, 0.5])
def test_matern_tiles_under_capture(prec, nu):
    r = subprocess.run([sys.executable, "-c", CAPTURE, prec, str(nu)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("fine"), r.stderr[-2000:]
