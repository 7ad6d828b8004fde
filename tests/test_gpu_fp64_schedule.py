"""The library's choice between the FP64 schedules: its results are, bit for bit, those of the schedule it
names on each side of the lines."""
import numpy as np
import pytest

import oracle
from paper_1312_4698_gb300 import workloads as wl
from tests.test_gpu_parity import gpu_propagate

pytestmark = pytest.mark.gpu

THREAD, GROUP = 1, 2


@pytest.mark.parametrize("F,form,n,steps,kernel", [
    (3, "", 14592, 4, GROUP), (3, "", 14593, 4, THREAD), (3, "", 19456, 4, THREAD), (3, "", 19457, 4, GROUP),
    (5, "", 14593, 4, THREAD), (5, "", 19456, 4, THREAD), (4, "", 16384, 4, GROUP), (3, "34", 16384, 4, THREAD),
    (3, "3", 16384, 4, GROUP), (3, "4", 16384, 4, GROUP), (5, "34", 16384, 4, GROUP),
    (6, "34", 9728, 1, GROUP), (6, "34", 9729, 1, THREAD), (9, "34", 14592, 1, GROUP), (9, "34", 14593, 1, THREAD),
    (7, "34", 14592, 2, GROUP), (7, "34", 14593, 2, THREAD), (8, "34", 14593, 2, GROUP), (7, "34", 14593, 3, GROUP),
])
def test_auto_takes_the_named_schedule(F, form, n, steps, kernel):
    import torch
    from paper_1312_4698_gb300 import scivr as G
    assert torch.cuda.is_available()
    w8 = wl.config_generic(F, F, n, steps)
    p = w8.pes
    c3 = (p.idx3, p.c3) if "3" in form else (np.zeros((0, 3)), np.zeros(0))
    c4 = (p.idx4, p.c4) if "4" in form else (np.zeros((0, 4)), np.zeros(0))
    w8 = w8.with_(pes=wl.PesDesc(F, p.diag_kind, p.omega, p.D, p.a, *c3, *c4))
    p0, q0, _ = oracle.sample_initial(w8.gamma, w8.p_eq, w8.q_eq, n, 11)
    auto, named = (gpu_propagate(G, w8, p0, q0, kernel=k) for k in (0, kernel))
    other = gpu_propagate(G, w8, p0, q0, kernel=THREAD + GROUP - kernel)
    assert np.array_equal(auto["amp"], named["amp"]) and np.array_equal(auto["good"], named["good"])
    assert not np.array_equal(auto["amp"], other["amp"])
