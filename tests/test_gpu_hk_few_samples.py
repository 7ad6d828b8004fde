"""Herman-Kluk transform of few samples, on both sides of the change from a sine and cosine per term to
blocks of samples, against sums in extended precision."""
import numpy as np
import pytest

from tests.test_gpu_ft_phases import DT, _series

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,n_E", [(2, 65), (3, 65), (8, 65), (9, 65), (33, 65), (127, 65), (128, 65), (129, 65),
                                   (128, 4864), (80, 4865), (81, 4865), (128, 4865)])
def test_few_samples(K, n_E):
    """A term has its factor's 6 roundings, the multiply-adds of up to 16 terms and 8 more for the sum over
    warps; in blocks up to 14 products of 5, the factors' 6, 62 multiply-adds and 16 behind the block: 154
    times 2^-53 of the sum of moduli covers both."""
    import torch
    from paper_1312_4698_gb300 import scivr as G
    L = np.longdouble
    assert np.finfo(L).eps < 1e-18
    a = _series(K, "flat")
    E_min, dE = 2.0 ** -6, 2.0 ** -12       # energies exact in FP64
    dev = torch.as_tensor(np.stack([a.real, a.imag], -1)[None].copy(), device="cuda")
    I = torch.empty(n_E, dtype=torch.float64, device="cuda")
    G.scivr_spectrum_hk(dev, K, torch.ones(1, dtype=torch.uint8, device="cuda"), 1, K - 1, DT, E_min,
                        E_min + (n_E - 1) * dE, n_E, I)
    ks = np.unique(np.linspace(0, n_E - 1, 65).astype(int))
    ph = (L(E_min) + ks.astype(L) * L(dE))[:, None] * (np.arange(K).astype(L) * L(DT))
    half = a.copy()
    half[0] *= 0.5
    ref = (half.real.astype(L) * np.cos(ph) - half.imag.astype(L) * np.sin(ph)).sum(1) * L(DT) / np.pi
    err = np.abs(I.cpu().numpy()[ks].astype(L) - ref).max()
    print(f"K={K} n_E={n_E}: {float(err / (DT / np.pi * np.abs(a).sum())):.2e} of the sum of moduli")
    assert err <= 154 * 2.0 ** -53 * DT / np.pi * np.abs(a).sum()
