"""The FP64 factorisation on the tensor cores (n > 2048: BF16 slice products for
the trailing update), at the sizes where its blocks can go wrong: tiles of one
and of several K chunks, tiles that are not a multiple of the 128-row block, a
K that is not a multiple of the 256-column flush, the smallest problem that
takes the path and ragged tails.

Factor: |L - L_lapack| <= 1e-12 max|L| + 1e-10 |L_lapack| (two FP64 Cholesky
factorisations of the same matrix differ by rounding order only, about
n 2^-53 max|L| = 5e-13 here).  A NaN in Sigma is reported as a failed pivot in
the first row that holds it, as by a Cholesky without slicing."""
import numpy as np
import pytest

import egs_inputs as ei

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def egs():
    import paper_1708_02835_gb300 as m
    m.load_library()
    return m


def _tiles(S, b):
    n = S.shape[0]
    T = -(-n // b)
    out = np.zeros((T * (T + 1) // 2, b, b))
    t = 0
    for i in range(T):
        for j in range(i + 1):
            blk = S[i * b:(i + 1) * b, j * b:(j + 1) * b]
            out[t, :blk.shape[0], :blk.shape[1]] = blk
            if i == j:
                for r in range(blk.shape[0], b):
                    out[t, r, r] = 1.0
            t += 1
    return out


def _cov(n, th2, seed):
    locs = ei.jittered_grid(n, seed=seed)
    return np.exp(-np.hypot(locs[0][:, None] - locs[0], locs[1][:, None] - locs[1]) / th2)


@pytest.mark.parametrize("n,b", [(2049, 64), (2049, 1024), (2100, 128), (2111, 192), (2560, 320), (2700, 256),
                                 (3000, 448), (4097, 512)])
def test_factor_matches_lapack(egs, n, b):
    import scipy.linalg as sla
    import torch
    S = _cov(n, 0.05, n)
    buf = torch.as_tensor(_tiles(S, b).reshape(-1)).cuda()
    assert egs.egs_potrf_tiles(buf, n, b) == -1
    got = buf.cpu().numpy().reshape(-1, b, b)
    L = sla.cholesky(S, lower=True)
    want = _tiles(L, b)
    lim = 1e-12 * np.abs(L).max() + 1e-10 * np.abs(want)
    T, t = -(-n // b), 0
    for i in range(T):
        for j in range(i + 1):
            w = np.tril(want[t]) if i == j else want[t]
            assert np.all(np.abs(got[t] - w) <= lim[t]), (i, j)
            t += 1


def test_nan_is_a_failed_pivot(egs):
    import torch
    n, b, bad = 2304, 256, 1500
    S = _cov(n, 0.05, 7)
    S[bad, 10] = S[10, bad] = np.nan
    buf = torch.as_tensor(_tiles(S, b).reshape(-1)).cuda()
    with pytest.raises(egs.NotPositiveDefinite) as e:
        egs.egs_potrf_tiles(buf, n, b)
    assert "row %d" % bad in str(e.value)
