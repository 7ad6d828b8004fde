"""The library's choice between the FP64 schedules where a surface has no couplings: its results are, bit
for bit, those of the schedule it names on each side of the lines."""
import numpy as np
import pytest

import oracle
from paper_1312_4698_gb300 import workloads as wl
from tests.test_gpu_parity import gpu_propagate

pytestmark = pytest.mark.gpu

THREAD, GROUP = 1, 2


@pytest.mark.parametrize("F,coupled,n,kernel", [
    (3, False, 14592, GROUP), (3, False, 14593, THREAD), (3, False, 19456, THREAD), (3, False, 19457, GROUP),
    (5, False, 14593, THREAD), (5, False, 19456, THREAD), (4, False, 16384, GROUP), (3, True, 16384, GROUP),
])
def test_auto_takes_the_named_schedule(F, coupled, n, kernel):
    import torch
    from paper_1312_4698_gb300 import scivr as G
    assert torch.cuda.is_available()
    w8 = (wl.config_generic(F, F, n, 4) if coupled else wl.uncoupled_morse(F)).with_(n_traj=n, n_steps=4)
    p0, q0, _ = oracle.sample_initial(w8.gamma, w8.p_eq, w8.q_eq, n, 11)
    auto, named = (gpu_propagate(G, w8, p0, q0, kernel=k) for k in (0, kernel))
    other = gpu_propagate(G, w8, p0, q0, kernel=THREAD + GROUP - kernel)
    assert np.array_equal(auto["amp"], named["amp"]) and np.array_equal(auto["good"], named["good"])
    assert not np.array_equal(auto["amp"], other["amp"])
