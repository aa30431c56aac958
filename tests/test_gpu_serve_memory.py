"""Served requests whose workspace cannot be allocated, by an allocator hook that declines what is
above a limit: an FP64 request that fits without the tensor-core update's scratch is answered (the
FP64 bar 1e-10 against the direct call), one that does not fit at all fails with EGS_ERR_OOM in
bounded time, and the request behind it is served."""
import numpy as np
import pytest

import egs_inputs as ei

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("room", ["dfma", "nothing"])
def test_workspace_that_cannot_be_had(room):
    import torch
    import paper_1708_02835_gb300 as egs
    from gpu_util import locs_dev, dev
    big, small, tile, th = 2500, 500, 256, (1.0, 0.08, 0.6)
    probs = {n: ei.Problem(n=n, theta=th, seed=n) for n in (big, small)}
    want = {n: egs.egs_loglik_ex(locs_dev(p.locations()), dev(p.e()), th, n, "fp64", tile=tile)[0]
            for n, p in probs.items()}
    need = egs.egs_loglik_workspace_bytes(big, tile, "fp64", 2)
    limit = need - 256 if room == "dfma" else egs.egs_loglik_workspace_bytes(small, tile, "fp64", 2)
    live = {}

    def alloc(nbytes, stream):
        if nbytes > limit:
            return 0
        t = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        live[t.data_ptr()] = t
        return t.data_ptr()

    egs.egs_set_allocator(alloc, lambda p, n, s: live.pop(p))
    try:
        srv = egs.egs_server(8 << 30, max_inflight=2, tile=tile)
    finally:
        egs.egs_set_allocator(None, None)
    ids = {n: srv.add_field(np.ascontiguousarray(p.locations().reshape(-1)), p.e(), n) for n, p in probs.items()}
    tickets = [srv.submit(ids[n], th, "fp64") for n in (big, small)]
    if room == "dfma":
        assert abs(srv.wait(tickets[0], timeout_ms=20000)[0] - want[big]) <= 1e-10 * abs(want[big])
    else:
        with pytest.raises(egs.EgsError) as e:
            srv.wait(tickets[0], timeout_ms=20000)
        assert e.value.status == egs.EGS_ERR_OOM
    assert srv.wait(tickets[1], timeout_ms=20000)[0] == want[small]
    st = srv.stats()
    assert st["rejected"] == (0 if room == "dfma" else 1) and st["queued"] == 0
    srv.close()
    assert not live
