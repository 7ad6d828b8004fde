"""Chirp-z spectra from several host threads whose energy grids need different amounts of shared memory."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,grids,calls", [(100, (900, 300), 4000), (2000, (2090, 1100), 2000)])
def test_threads_with_different_grids(K, grids, calls):
    """Both grids take transforms of the same length (1024 points at K = 100, 4096 at 2000), hence the same
    kernel, whose limit of shared memory all threads share: no call may be refused, and every spectrum
    equals, bit for bit, the one computed alone."""
    import torch
    from paper_1312_4698_gb300 import scivr as G
    rng = np.random.default_rng(K)
    a = torch.as_tensor(rng.normal(size=(1, K, 2)), device="cuda")
    w = torch.ones(1, dtype=torch.float64, device="cuda")
    good = torch.ones(1, dtype=torch.uint8, device="cuda")

    def spectrum(n_E, out, stream):
        G.scivr_spectrum(a, K, w, good, 1, K - 1, 10.0, 0.01, 0.05, n_E, out, ft_mode=G.SCIVR_FT_CZT64, stream=stream)

    alone = [torch.empty(n_E, dtype=torch.float64, device="cuda") for n_E in grids]
    for n_E, out in zip(grids, alone):
        spectrum(n_E, out, 0)
    torch.cuda.synchronize()
    threads_of = (0, 0, 0, 1, 1, 1)
    outs = [torch.empty_like(alone[i]) for i in threads_of]
    streams = [torch.cuda.Stream() for _ in threads_of]
    torch.cuda.synchronize()
    refused = []
    start = threading.Barrier(len(threads_of))

    def work(t):
        start.wait()
        for c in range(calls):
            try:
                spectrum(grids[threads_of[t]], outs[t], streams[t].cuda_stream)
            except Exception as e:
                refused.append(str(e))
            if c % 100 == 99:
                streams[t].synchronize()

    threads = [threading.Thread(target=work, args=(t,)) for t in range(len(threads_of))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not refused, f"{len(refused)} of {calls * len(threads_of)} calls refused: {refused[0]}"
    assert all(torch.equal(outs[t], alone[i]) for t, i in enumerate(threads_of))
