"""Column sums of the Herman-Kluk spectrum (64-bit fixed point over a moving window of exponents)
against exactly rounded sums.

A summand is cut at 2^-54 of eight times the largest magnitude M seen (at most 2^-52 M), 64 at a time enter
an FP64 sum: the mean of n is off by at most 2^-52 M from the cuts and, the partial sums being at most n M,
by 2^-53 M for each of the n / 64 + 8 + 152 additions behind it at worst.  (4 + n / 64 / 2 + 80) 2^-52 M is the bound.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _columns(kind, n, K, rng):
    a = rng.normal(size=(n, K, 2))
    if kind == "spread":          # twenty orders of magnitude within a column
        a *= 10.0 ** rng.uniform(-20, 0, size=(n, K, 1))
    elif kind == "growing":       # the window moves all the time
        a *= 2.0 ** (0.9 * np.arange(n) * min(1.0, 900.0 / n))[:, None, None]
    elif kind == "positive":
        a = np.abs(a)
    elif kind == "tiny":          # denormals and the smallest normal numbers
        a *= 1e-308
    elif kind == "huge":
        a *= 1e300 / n
    elif kind == "zeros":
        a[: n // 2] = 0.0
    return a


@pytest.mark.parametrize("kind", ["plain", "spread", "growing", "positive", "tiny", "huge", "zeros"])
@pytest.mark.parametrize("n,K", [(1, 2), (7, 5), (8, 3), (64, 257), (71, 256), (1000, 300), (5000, 33)])
def test_column_sums(kind, n, K):
    import torch
    from paper_1312_4698_gb300 import scivr as G
    rng = np.random.default_rng(n + K)
    a = _columns(kind, n, K, rng)
    good = (rng.random(n) > 0.2).astype(np.uint8)
    good[0] = 1
    bad = np.flatnonzero(good == 0)
    if bad.size:
        a[bad[0], :, 0], a[bad[-1], :, 1] = np.nan, np.inf
    n_E = 5
    I = torch.empty(n_E, dtype=torch.float64, device="cuda")
    C = torch.empty((K, 2), dtype=torch.float64, device="cuda")
    ng = torch.zeros(1, dtype=torch.int64, device="cuda")
    G.scivr_spectrum_hk(torch.as_tensor(a, device="cuda"), K, torch.as_tensor(good, device="cuda"), n, K - 1, 10.0,
                        0.001, 0.05, n_E, I, C, ng)
    got = C.cpu().numpy()
    rows = a[good.astype(bool)]
    m = len(rows)
    assert int(ng.item()) == m
    for c in range(K):
        for part in range(2):
            ref = math.fsum(rows[:, c, part]) / m
            big = np.abs(rows[:, c]).max()
            assert abs(got[c, part] - ref) <= (84 + n / 128) * 2.0 ** -52 * big + 5e-324, (c, part)


def test_column_sums_pass_on_what_is_not_finite():
    import torch
    from paper_1312_4698_gb300 import scivr as G
    a = np.random.default_rng(5).normal(size=(100, 4, 2))
    a[40, 1, 0], a[99, 2, 1] = np.inf, np.nan
    I = torch.empty(3, dtype=torch.float64, device="cuda")
    C = torch.empty((4, 2), dtype=torch.float64, device="cuda")
    ng = torch.zeros(1, dtype=torch.int64, device="cuda")
    G.scivr_spectrum_hk(torch.as_tensor(a, device="cuda"), 4, torch.ones(100, dtype=torch.uint8, device="cuda"), 100, 3,
                        10.0, 0.001, 0.05, 3, I, C, ng)
    got = C.cpu().numpy()
    assert got[1, 0] == np.inf and np.isnan(got[2, 1])
    assert np.isfinite(got[[0, 3]]).all() and np.isfinite([got[1, 1], got[2, 0]]).all()
    assert np.allclose(got[[0, 3]], a.mean(0)[[0, 3]], rtol=0, atol=1e-15)
