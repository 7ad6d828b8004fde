"""F = 24 without quartic terms: its own kernel beyond 608 trajectories and without couplings, the shared
Hessian's below: the same steps, sums and chunks, so the same bits, also as the general kernels give with a
quartic term of coefficient zero."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_cubic_schedule import G, _surface  # noqa: F401
from tests.test_gpu_parity import MIXED_STAB_TOL, gpu_propagate

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["cubic", "morse", "harmonic"])
@pytest.mark.parametrize("n", [1, 608, 611, 1221])
def test_f24_gives_the_general_kernels_bits(G, form, n):  # noqa: F811
    w8 = _surface(24, form).with_(n_traj=n, n_steps=6)
    ref8 = _surface(24, form, general=True).with_(n_traj=n, n_steps=6)
    p0, q0, _ = oracle.sample_initial(w8.gamma, w8.p_eq, w8.q_eq, n, 7)
    a = gpu_propagate(G, w8, p0, q0, precision=1, stab_tol=MIXED_STAB_TOL, fin=True)
    b = gpu_propagate(G, ref8, p0, q0, precision=1, stab_tol=MIXED_STAB_TOL, fin=True)
    for k in a:
        assert np.array_equal(a[k], b[k], equal_nan=True), k
