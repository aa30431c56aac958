"""FP64 factorisations of matrices whose pivots lie near the ends of the doubles' range, or far apart
inside one 64 x 64 block: diagonal matrices against the square roots (each entry by itself, 4 ulp; a
subnormal pivot has only its own bits: 1e-10), coupled pairs of very different scale, and the whole
evaluation at theta1 from 2^-900 to 2^996, which shifts log|Sigma| by n log theta1 and leaves the
quadratic form of data scaled alike (1e-10 relative, the FP64 bar; n log theta1 is up to 700 n).
Further down the covariances themselves leave the normal doubles, where they are 0."""
import math

import numpy as np
import pytest

import egs_inputs as ei

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def egs():
    import paper_1708_02835_gb300 as m
    m.load_library()
    return m


def _factor(egs, A, b):
    import torch
    n = A.shape[0]
    T = -(-n // b)
    t = torch.zeros(T * (T + 1) // 2, b, b, dtype=torch.float64)
    k = 0
    for i in range(T):
        for j in range(i + 1):
            blk = torch.as_tensor(np.ascontiguousarray(A[i * b:(i + 1) * b, j * b:(j + 1) * b]))
            t[k, :blk.shape[0], :blk.shape[1]] = blk
            if i == j:
                for r in range(blk.shape[0], b):
                    t[k, r, r] = 1.0
            k += 1
    t = t.cuda()
    assert egs.egs_potrf_tiles(t, n, b) == -1
    L, k = np.zeros((T * b, T * b)), 0
    t = t.cpu().numpy()
    for i in range(T):
        for j in range(i + 1):
            L[i * b:(i + 1) * b, j * b:(j + 1) * b] = t[k]
            k += 1
    return np.tril(L)[:n, :n]


@pytest.mark.parametrize("n,b", [(64, 64), (200, 128), (2100, 128)])
def test_diagonal_matrices(egs, n, b):
    r = np.random.default_rng(n)
    for lo, hi in ((-300, 300), (-307, -300), (300, 308)):
        d = 10.0 ** r.uniform(lo, hi, n)
        d = np.where(np.isfinite(d), d, 1e308)
        L = _factor(egs, np.diag(d), b)
        assert np.all(np.abs(np.diag(L) - np.sqrt(d)) <= 4 * 2.0 ** -53 * np.sqrt(d)), (lo, hi)
        assert np.count_nonzero(L - np.diag(np.diag(L))) == 0
    d = np.ones(n)
    d[[10, 37, 63]] = 1e-310, 5e-320, 3e-309
    d[-1] = 1e-312
    L = _factor(egs, np.diag(d), b)
    assert np.all(np.abs(np.diag(L) - np.sqrt(d)) <= 1e-10 * np.sqrt(d))


@pytest.mark.parametrize("n", [150, 2100])
def test_coupled_scales_in_one_block(egs, n):
    """Correlation 0.45 between neighbours whose scales differ by up to 10^280."""
    r = np.random.default_rng(3)
    s = 10.0 ** r.uniform(-140, 140, n)
    C = np.eye(n) + 0.5 * (np.eye(n, k=1) + np.eye(n, k=-1)) * 0.9
    L = _factor(egs, C * s[:, None] * s[None, :], 128) / s[:, None]
    assert np.max(np.abs(L - np.linalg.cholesky(C))) <= 1e-13


@pytest.mark.parametrize("n", [700, 2500])
@pytest.mark.parametrize("nu", [0.5, 0.8])
def test_theta1_over_the_range_of_doubles(egs, n, nu):
    from gpu_util import locs_dev, dev
    p = ei.Problem(n=n, theta=(1.0, 0.05, nu), seed=1)
    locs, z = locs_dev(p.locations()), p.e()
    _, ref = egs.egs_loglik_ex(locs, dev(z), (1.0, 0.05, nu), n, "fp64")
    for e in (-900, -700, 640, 996):
        th1 = 2.0 ** e
        _, info = egs.egs_loglik_ex(locs, dev(z * 2.0 ** (e // 2)), (th1, 0.05, nu), n, "fp64")
        assert abs(info["quad"] - ref["quad"]) <= 1e-10 * ref["quad"], e
        want = ref["logdet"] + n * e * math.log(2.0)
        assert abs(info["logdet"] - want) <= 1e-10 * abs(want), e
