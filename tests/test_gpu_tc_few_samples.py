"""Tensor-core Fourier step of up to a few hundred samples, whose amplitudes are split in short blocks:
around the ends of one to five of them, with ragged rows, bad trajectories and both row types."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

TOL = {2: 2e-4, 3: 2e-4}   # as for the other tests of these modes against the oracle


@pytest.mark.parametrize("mode", [2, 3])
@pytest.mark.parametrize("K", [2, 9, 55, 56, 57, 63, 64, 111, 112, 113, 119, 168, 169, 223, 224, 225])
def test_tc_amplitudes_at_block_edges(K, mode):
    import torch
    from paper_1312_4698_gb300 import scivr as G
    rng = np.random.default_rng(K)
    n, n_E = 131, 70
    amp = rng.normal(size=(n, K)) + 1j * rng.normal(size=(n, K))
    w = rng.uniform(0.2, 5.0, n)
    good = (rng.uniform(size=n) > 0.2).astype(np.uint8)
    good[0], good[-1], good[7] = 1, 1, 0
    amp[7, K // 2] = np.nan
    for f32 in (False, True):
        a = amp.astype(np.complex64) if f32 else amp
        dev = torch.as_tensor(np.stack([a.real, a.imag], -1).copy(), device="cuda")
        I = torch.empty(n_E, dtype=torch.float64, device="cuda")
        ng = torch.zeros(1, dtype=torch.int64, device="cuda")
        G.scivr_spectrum(dev, K, torch.as_tensor(w, device="cuda"), torch.as_tensor(good, device="cuda"), n, K - 1,
                         10.0, 0.002, 0.06, n_E, I, ng, ft_mode=mode)
        ref, rng_ = oracle.spectrum(a.astype(complex), w, good, K - 1, 10.0, 0.002, 0.06, n_E)
        assert int(ng.item()) == rng_
        assert np.max(np.abs(I.cpu().numpy() - ref)) <= TOL[mode] * np.max(ref)
