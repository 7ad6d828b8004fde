"""Phases of the FP64 Fourier steps that sum blocks of samples around shared centres, against
sums in extended precision.

The energies are exact in FP64 and phases reach 1.2e5 radians, whose own rounding (7e-12) would be
some 500 times the bounds if a block's samples shared it.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DT, E_MIN, N_E = 997.3, 2.0 ** -6, 65
E_MAX = E_MIN + (N_E - 1) * 2.0 ** -12


def _series(K, kind, dt=DT):
    c = np.arange(K)
    if kind == "line":       # one frequency, decaying: a peak in the window
        return np.exp(-c / (0.3 * K)) * np.exp(-1j * ((0.0251 * dt * c) % (2 * np.pi)))
    return np.exp(-1j * 0.4 * c / K) * (1.0 + 0.2 * np.cos(0.01 * c))


def _exact(a, K, dt=DT):
    """sum_c a_c exp(i E_k c dt) for every energy."""
    L = np.longdouble
    assert np.finfo(L).eps < 1e-18
    ph = (L(E_MIN) + np.arange(N_E).astype(L) * L(2.0 ** -12))[:, None] * (np.arange(K).astype(L) * L(dt))
    co, sn = np.cos(ph), np.sin(ph)
    re, im = a.real.astype(L), a.imag.astype(L)
    return (re * co - im * sn).sum(1), (re * sn + im * co).sum(1)


@pytest.mark.parametrize("kind", ["line", "flat"])
@pytest.mark.parametrize("K", [64, 505, 4001])
def test_herman_kluk_transform(K, kind):
    """A term passes up to 7 products for its place in the block and 7 for the block (a complex
    product and its factor: 5 roundings), the factors' own 6, 62 multiply-adds in the block and at most
    K / 504 + 8 behind it: (5 * 14 + 6 + 62 + 16) 2^-53 of the sum of moduli, 2^-45.7."""
    import torch
    from paper_1312_4698_gb300 import scivr as G
    a = _series(K, kind)
    dev = torch.as_tensor(np.stack([a.real, a.imag], -1)[None].copy(), device="cuda")
    I = torch.empty(N_E, dtype=torch.float64, device="cuda")
    G.scivr_spectrum_hk(dev, K, torch.ones(1, dtype=torch.uint8, device="cuda"), 1, K - 1, DT, E_MIN, E_MAX, N_E, I)
    half = a.copy()
    half[0] *= 0.5
    ref = np.asarray(_exact(half, K)[0] * np.longdouble(DT) / np.pi, dtype=np.longdouble)
    err = np.abs(I.cpu().numpy().astype(np.longdouble) - ref).max()
    print(f"K={K} {kind}: {float(err / (DT / np.pi * np.abs(a).sum())):.2e} of the sum of moduli")
    assert err <= 2.0 ** -45.7 * DT / np.pi * np.abs(a).sum()


@pytest.mark.parametrize("kind", ["line", "flat"])
@pytest.mark.parametrize("K", [17, 331, 4001])
def test_direct_step(K, kind):
    """Phases to 2e6 radians.  A term carries its two factors' roundings (11 with their product), 64
    multiply-adds in its block and two for every later block of 33 samples: X is off by at most
    d = (75 + 2 K / 33) 2^-53 of the sum of moduli, |X|^2 by (2 |X| + d) d."""
    import torch
    from paper_1312_4698_gb300 import scivr as G
    dt = 16 * DT
    a = _series(K, kind, dt)
    dev = torch.as_tensor(np.stack([a.real, a.imag], -1)[None].copy(), device="cuda")
    one = torch.ones(1, dtype=torch.float64, device="cuda")
    I = torch.empty(N_E, dtype=torch.float64, device="cuda")
    G.scivr_spectrum(dev, K, one, one.to(torch.uint8), 1, K - 1, dt, E_MIN, E_MAX, N_E, I, ft_mode=G.SCIVR_FT_FP64)
    re, im = _exact(a, K, dt)
    scale = dt * dt / (2 * np.pi * (K - 1) * dt)
    d = (75 + 2 * K / 33) * 2.0 ** -53 * np.abs(a).sum()
    X2 = re * re + im * im
    err = np.abs(I.cpu().numpy().astype(np.longdouble) / scale - X2)
    print(f"K={K} {kind}: {float((err / ((2 * np.sqrt(X2) + d) * d)).max()):.2e} of the bound")
    assert np.all(err <= (2 * np.sqrt(X2) + d) * d + 4 * 2.0 ** -53 * X2)
