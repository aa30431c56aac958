"""The FP64 update by slice products on rows whose digits are all large and of one sign: the level
sums have to be exact whatever the data, not only for rows that look random.

Sigma = [[I, X'], [X, X X' + I]], so that L = [[I, 0], [X, I]].  X = f 2^-56 with base-256 digits of
f in 240 .. 255 (the first), 120 .. 127 (the next three) and 0 .. 15, so that 256 products of level 2
and 3 sum to more than 2^24 units.  X X' comes from exact integer products (three 19-bit pieces).
Errors: the rounding of Sigma and of the update (2^-53 b each, b the tile), the dropped products
(below b 2^-56) and the FP32 sums of the levels from 4 on (a few 2^-48): below 1e-12 for b <= 1,024.
One unit of level 2 lost is 2^-32."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _digits(rows, b, seed):
    r = np.random.default_rng(seed)
    f = r.integers(240, 256, (rows, b), dtype=np.int64)
    for lo, hi in ((120, 128), (120, 128), (120, 128), (0, 16), (0, 16)):
        f = f * 256 + r.integers(lo, hi, (rows, b), dtype=np.int64)
    return f * 256  # 56 bits, the last byte 0: exact doubles


def _gram(f):
    """f f' 2^-112 to long double."""
    p = [(f >> (19 * i) & (2 ** 19 - 1)).astype(np.float64) for i in range(3)]
    out = np.zeros((f.shape[0], f.shape[0]), dtype=np.longdouble)
    for i in range(3):
        for j in range(3):
            out += np.ldexp((p[i] @ p[j].T).astype(np.longdouble), 19 * (i + j) - 112)
    return out


@pytest.mark.parametrize("b,T,flip", [(256, 9, 0), (512, 5, 0), (576, 4, 1), (1024, 3, 1)])
def test_rows_in_phase(b, T, flip):
    import torch
    import paper_1708_02835_gb300 as egs
    n, m = b * T, b * (T - 1)
    f = _digits(m, b, b)
    if flip:
        f[::3] *= -1
        s = np.where(np.arange(m) % 3 == 0, -1.0, 1.0)
    else:
        s = np.ones(m)
    X = np.ldexp(f.astype(np.float64), -56)
    assert np.all(np.ldexp(X, 56).astype(np.int64) == f) and np.abs(X).max() < 1.0
    A = (_gram(np.abs(f)) * s[:, None] * s[None, :] + np.eye(m)).astype(np.float64)
    t = torch.zeros(T * (T + 1) // 2, b, b, dtype=torch.float64, device="cuda")
    k = 0
    for i in range(T):
        for j in range(i + 1):
            blk = np.eye(b) if i == 0 else (X[(i - 1) * b:i * b] if j == 0 else
                                            A[(i - 1) * b:i * b, (j - 1) * b:j * b])
            t[k] = torch.as_tensor(blk)
            k += 1
    assert egs.egs_potrf_tiles(t, n, b) == -1
    eye = torch.eye(b, dtype=torch.float64, device="cuda")
    k, worst = 0, 0.0
    for i in range(T):
        for j in range(i + 1):
            if j > 0:
                d = torch.tril(t[k]) - eye if i == j else t[k]
                worst = max(worst, float(d.abs().max()))
            k += 1
    print("b %d: worst |L - I| %.2e" % (b, worst))
    assert worst <= 1e-12
