"""FP64 lane groups with more reference states than one: every group size of F = 1 and more states than
lanes, against the thread-per-trajectory schedule, whose records a lane forms alone."""
import numpy as np
import pytest

from paper_1312_4698_gb300 import workloads as wl
from tests.test_gpu_group_fp64 import _propagate

pytestmark = pytest.mark.gpu


# F = 1: 8, 4 and 2 lanes by the number of trajectories (4864 lanes a round with a recording warp)
@pytest.mark.parametrize("F,n,n_chi", [(1, 1, 8), (1, 5, 2), (1, 607, 8), (1, 609, 8), (1, 1217, 8), (1, 2437, 3),
                                       (1, 4867, 8), (2, 37, 8), (2, 2437, 5), (3, 609, 8), (6, 4867, 5), (9, 70, 8)])
@pytest.mark.parametrize("amplitude", [0, 1])
def test_states_agree_with_the_thread_schedule(F, n, n_chi, amplitude):
    """FP64 with other summation orders: 1e-9 of each row's largest amplitude, as between the schedules
    with one state."""
    from paper_1312_4698_gb300 import scivr as G
    rng = np.random.default_rng(10 * F + n_chi)
    w8 = wl.config_generic(F, F, n, 21)
    gam = np.asarray(w8.gamma)
    pe = np.asarray(w8.p_eq)[0] * rng.uniform(0.8, 1.2, (n_chi, F))
    qe = np.asarray(w8.q_eq)[0] + rng.normal(size=(n_chi, F)) * 0.3 / np.sqrt(gam)
    w8 = w8.with_(p_eq=pe, q_eq=qe)
    q0 = qe[0][:, None] + rng.standard_normal((F, n)) / np.sqrt(gam)[:, None]
    p0 = pe[0][:, None] + rng.standard_normal((F, n)) * np.sqrt(gam)[:, None]
    a, ga, fa = _propagate(G, w8, p0, q0, 2, amplitude)
    b, gb, fb = _propagate(G, w8, p0, q0, 1, amplitude)
    assert a.shape[0] == n_chi and np.array_equal(ga, gb)
    sel = gb.astype(bool)
    za, zb = a[..., 0] + 1j * a[..., 1], b[..., 0] + 1j * b[..., 1]
    err = np.abs(za - zb)[:, sel] / np.abs(zb)[:, sel].max(-1, keepdims=True)
    assert np.isfinite(za[:, sel]).all() and err.max() < 1e-9
    assert np.abs(fa["theta"] - fb["theta"])[sel].max() < 1e-8
