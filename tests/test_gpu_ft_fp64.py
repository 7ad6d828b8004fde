"""The direct FP64 Fourier step at its tile and block edges against 64-bit sums in numpy.

Blocks are 33 samples, tiles 8 or 32 rows by 32 energies (32 rows from 608 such tiles on).  A sum of K terms
of size ~1 carries at most ~K eps of rounding, its phases E t < 40 rad another 40 eps: 1e-12 of the largest
intensity bounds both with room for K = 1000.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_steps,n_E,f32", [
    (1, 1, 2, False), (3, 32, 33, False), (8, 33, 32, True), (9, 65, 31, False), (31, 66, 100, False),
    (640, 98, 960, False),    # 600 tiles of 32 rows: still 8-row tiles
    (641, 99, 961, False),    # 651: 32-row tiles, one row and one energy over
    (700, 1000, 900, True)])
def test_direct_sum_tiles_and_blocks(n, n_steps, n_E, f32):
    import torch
    from paper_1312_4698_gb300 import scivr as G
    rng = np.random.default_rng(n * 7 + n_steps)
    K, ld = n_steps + 1, n_steps + 4
    amp = rng.normal(size=(n, ld, 2)) * 0.5
    if f32:
        amp = amp.astype(np.float32)
    w, good = rng.uniform(0.5, 2.0, n), (rng.random(n) > 0.1).astype(np.uint8)
    good[0] = 1
    bad = np.flatnonzero(good == 0)
    if bad.size:
        amp[bad[0], K // 2] = np.nan   # a bad row does not reach the others
    dt, E0, E1 = 5.0, 0.001, 0.008
    I = torch.empty(n_E, dtype=torch.float64, device="cuda")
    ng = torch.zeros(1, dtype=torch.int64, device="cuda")
    G.scivr_spectrum(torch.as_tensor(amp, device="cuda"), ld, torch.as_tensor(w, device="cuda"),
                     torch.as_tensor(good, device="cuda"), n, n_steps, dt, E0, E1, n_E, I, ng, ft_mode=G.SCIVR_FT_FP64)
    g = good.astype(bool)
    a = amp[g, :K].astype(np.float64)
    ph = np.exp(1j * np.outer(np.arange(K) * dt, np.linspace(E0, E1, n_E)))
    ref = (w[g, None] * np.abs((a[..., 0] + 1j * a[..., 1]) @ ph) ** 2).sum(0) * dt * dt / (2 * np.pi * n_steps * dt * g.sum())
    assert int(ng.item()) == g.sum()
    assert np.abs(I.cpu().numpy() - ref).max() <= 1e-12 * ref.max()
