"""The two streams of a mixed evaluation beside other work on the GPU: bands of one, two and three
tiles, evaluated alone and by three threads at once, give the same value bit for bit (every tile's
updates are ordered, whatever the streams' timing), and that value is within the modes' guards of
the oracle (5e-5 in the FP32 mode, 1e-3 in TF32 and BF16)."""
import threading

import pytest

import egs_inputs as ei
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,lim", [("fp32", 5e-5), ("tf32", 1e-3), ("bf16", 1e-3)])
@pytest.mark.parametrize("band", [1, 2, 3])
def test_same_value_alone_and_beside_others(prec, lim, band):
    import torch
    import paper_1708_02835_gb300 as egs
    from gpu_util import locs_dev, dev
    n, theta = 3100, (1.0, 0.03, 0.5)
    p = ei.Problem(n=n, theta=theta, seed=21)
    locs = p.locations()
    z = oracle.simulate_z(locs, theta, p.e())
    ref = oracle.loglik_lapack(locs, z, theta)["loglik"]
    dl, dz = locs_dev(locs), dev(z)

    def one(stream=0):
        return egs.egs_loglik_ex(dl, dz, theta, n, prec, tile=256, band=band, stream=stream)[0]

    alone = [one() for _ in range(3)]
    assert alone[0] == alone[1] == alone[2]
    assert abs(alone[0] - ref) <= lim * abs(ref)
    torch.cuda.synchronize()
    got = []

    def work():
        s = torch.cuda.Stream()
        for _ in range(4):
            got.append(one(s.cuda_stream))

    threads = [threading.Thread(target=work) for _ in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert got == [alone[0]] * 12
