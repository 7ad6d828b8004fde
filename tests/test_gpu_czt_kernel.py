"""Accuracy of the chirp-z step's convolution against sums in extended precision.

Model of the rounding errors: every butterfly stage and product gives each component two roundings of
standard deviation 2^-53 / sqrt(3) of its size, independent of each other.  Three transforms of log2 L stages, two
chirps and two products: a relative error of sqrt((3 log2 L + 6) 2 / 3) 2^-53 in the two-norm, which
spreads over the outputs, so that X has a root mean square error of that times the two-norm of
the amplitudes, and |X|, which the spectrum shows, 1 / sqrt(2) of it.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,n_E,log2L,log2dE", [
    (512, 500, 10, -15), (1000, 25, 10, -15), (200, 1025, 11, -20), (2049, 2000, 12, -18), (4001, 2000, 13, -15),
])
def test_convolution_error(K, n_E, log2L, log2dE):
    import torch
    from paper_1312_4698_gb300 import scivr as G
    L = np.longdouble
    assert np.finfo(L).eps < 1e-18
    rng = np.random.default_rng(K)
    a = rng.normal(size=K) + 1j * rng.normal(size=K)
    dt, E_min, dE = 8.0, 2.0 ** -8, 2.0 ** log2dE     # every phase E_k c dt exact in FP64
    dev = torch.as_tensor(np.stack([a.real, a.imag], -1)[None].copy(), device="cuda")
    one = torch.ones(1, dtype=torch.float64, device="cuda")
    I = torch.empty(n_E, dtype=torch.float64, device="cuda")
    G.scivr_spectrum(dev, K, one, one.to(torch.uint8), 1, K - 1, dt, E_min, E_min + (n_E - 1) * dE, n_E, I,
                     ft_mode=G.SCIVR_FT_CZT64)
    got = np.sqrt(I.cpu().numpy().astype(L) * L(2.0) * L("3.14159265358979323846264338327950288") * L(K - 1) / L(dt))
    ks = np.unique(np.linspace(0, n_E - 1, 80).astype(int))
    ph = (L(E_min) + ks.astype(L) * L(dE))[:, None] * (np.arange(K).astype(L) * L(dt))
    co, sn = np.cos(ph), np.sin(ph)
    ref = np.hypot((a.real * co - a.imag * sn).sum(1), (a.real * sn + a.imag * co).sum(1))
    rms = float(np.sqrt(np.mean((got[ks] - ref) ** 2)) / np.linalg.norm(a))
    print(f"K={K} n_E={n_E}: {rms * 2.0 ** 53:.2f} of 2^-53")
    assert rms <= np.sqrt((3 * log2L + 6) / 3) * 2.0 ** -53
