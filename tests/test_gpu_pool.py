"""The library's memory pool gives back what it keeps between calls on egs_set_allocator and when a
server ends."""
import pytest

import egs_inputs as ei

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.fixture()
def egs():
    import torch
    import paper_1708_02835_gb300 as m
    m.load_library()
    m.egs_set_allocator(None, None)
    torch.cuda.empty_cache()
    yield m
    m.egs_set_allocator(None, None)
    torch.cuda.empty_cache()


def _fill_pool(egs):
    from gpu_util import locs_dev, dev
    n, theta = 18000, (1.0, 0.05, 0.5)
    p = ei.Problem(n=n, theta=theta, seed=1)
    egs.egs_loglik_ex(locs_dev(p.locations()), dev(p.e()), theta, n, "fp64", tile=512)
    return egs.egs_loglik_workspace_bytes(n, 512, "fp64", 2)


def test_pool_is_given_back(egs):
    base = _free()
    kept = _fill_pool(egs)
    assert kept > 1200 * MB and _free() <= base - kept + 200 * MB
    egs.egs_set_allocator(None, None)
    assert _free() >= base - 200 * MB
    _fill_pool(egs)
    srv = egs.egs_server(1 << 30, max_inflight=1)
    srv.close()
    assert _free() >= base - 200 * MB
