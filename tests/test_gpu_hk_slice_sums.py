"""Column sums of the Herman-Kluk spectrum where a slice has many rows, and where one part of a
column is much smaller than the other.

Real and imaginary parts are summed apart.  The sum s of a slice's rows carries one rounding, at
most 2^-53 |s|, plus one for every time a summand 256 times the largest so far (or more) arrives, and a
thread adds every eighth slice before the eight threads' sums are added: a mean over n rows in at most
n / 16 slices is off by at most (n / 128 + 8 + 3) 2^-53 of the slices' moduli summed and divided by
the count, the last 3 for a slice's own rounding, the division and the reference's.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _spectrum(a, good):
    import torch
    from paper_1312_4698_gb300 import scivr as G
    n, K = a.shape[:2]
    I = torch.empty(3, dtype=torch.float64, device="cuda")
    C = torch.empty((K, 2), dtype=torch.float64, device="cuda")
    G.scivr_spectrum_hk(a, K, good, n, K - 1, 10.0, 0.001, 0.05, 3, I, C)
    return C


def _check(got, col, moduli, slices):
    """got: the mean of col; moduli: a bound on the sum of the slices' moduli."""
    ref = math.fsum(col) / len(col)
    assert abs(got - ref) <= (slices / 8 + 11) * 2.0 ** -53 * moduli / len(col) + 5e-324


@pytest.mark.parametrize("small", [1e-3, 1e-9, 1e-14, 1e-40, 1e-250])
@pytest.mark.parametrize("n,K", [(9, 3), (71, 256), (1000, 300)])
def test_a_small_part_keeps_its_own_precision(small, n, K):
    import torch
    rng = np.random.default_rng(n)
    a = rng.normal(size=(n, K, 2))
    a[:, ::2, 1] *= small
    a[:, 1::2, 0] *= small
    got = _spectrum(torch.as_tensor(a, device="cuda"), torch.ones(n, dtype=torch.uint8, device="cuda")).cpu().numpy()
    for c in range(K):
        for part in range(2):
            _check(got[c, part], a[:, c, part], np.abs(a[:, c, part]).sum(), n / 16)


# 40000 columns are 157 CTAs wide, 8 slices of 1024 rows: 128 rows each, of 1023: 127 and a remainder of 7
@pytest.mark.parametrize("n", [1024, 1023])
def test_slices_of_many_rows(n):
    import torch
    K, ld = 40000, 40000
    rng = np.random.default_rng(n)
    i = np.arange(n)
    cols = {
        "plain": rng.normal(size=n),
        "positive": np.abs(rng.normal(size=n)),
        "negative": -np.abs(rng.normal(size=n)),
        # the first summand opens a window of eight binades above it, the rest fill it to the top
        "top": np.where(i % (n // 8) == 0, 1.0, np.nextafter(512.0, 0.0)),
        "minus top": np.where(i % (n // 8) == 0, -1.0, -np.nextafter(512.0, 0.0)),
        "past the top": np.where(i % (n // 8) == 0, 1.0, 512.0),
        "growing": rng.normal(size=n) * 2.0 ** (i % 128 * 7.0),
        "shrinking": rng.normal(size=n) * 2.0 ** (-(i % 128) * 7.0),
        "spread": rng.normal(size=n) * 10.0 ** rng.uniform(-16, 0, n),
        "huge": np.abs(rng.normal(size=n)) * 1e300,
        "tiny": rng.normal(size=n) * 1e-300,
    }
    # pairs of rows that cancel but for their last bits (128 rows a slice: no pair is cut)
    big = rng.normal(size=n // 2) * 1e8
    pairs = np.zeros(n)
    pairs[: n // 2 * 2 : 2], pairs[1 : n // 2 * 2 : 2] = big, -big + rng.normal(size=n // 2)
    if n % 2 == 0:
        cols["cancelling"] = pairs
    a = torch.randn((n, ld, 2), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    places = [(k * (K - 1) // (len(cols) - 1), k % 2) for k in range(len(cols))]
    for (c, part), x in zip(places, cols.values()):
        a[:, c, part] = torch.as_tensor(x, device="cuda")
    got = _spectrum(a, torch.ones(n, dtype=torch.uint8, device="cuda")).cpu().numpy()
    for (c, part), (name, x) in zip(places, cols.items()):
        moduli = np.abs(x).sum() if name != "cancelling" else np.abs(x.reshape(-1, 2).sum(1)).sum()
        _check(got[c, part], x, moduli, 8)
    # bad rows, whatever they hold, leave the others' sums alone
    good = (np.arange(n) % 3 != 1)
    a[torch.as_tensor(~good, device="cuda")] = float("nan")
    got = _spectrum(a, torch.as_tensor(good.astype(np.uint8), device="cuda")).cpu().numpy()
    for (c, part), (name, x) in zip(places, cols.items()):
        _check(got[c, part], x[good], np.abs(x[good]).sum(), 8)
