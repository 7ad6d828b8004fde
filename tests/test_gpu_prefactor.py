"""det A of the mixed path: the double-FP32 elimination shared by 1 to 32 lanes of a warp, at every
number of modes, against the FP64 determinant of the prefactor matrix built from the exported
monodromy (whose FP32 values it starts from)."""
import numpy as np
import pytest

import oracle
from paper_1312_4698_gb300 import workloads as wl
from tests.test_gpu_parity import MIXED_STAB_TOL, gpu_propagate

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    from paper_1312_4698_gb300 import scivr
    assert torch.cuda.is_available()
    return scivr


@pytest.mark.parametrize("F", list(range(1, 25)))
def test_det_a_is_the_determinant_of_its_matrix(G, F):
    """Bound: the entries of A are formed in FP32, three roundings each, so |d det / det| <=
    |tr(A^-1 dA)| <= ||A^-1|| ||dA||, ||dA|| at most 3 2^-24 of the norm of the terms' moduli; the
    elimination's own 2^-46 is far below.  The last step falls inside a chunk and on its end."""
    w8 = wl.config_f3() if F == 3 else wl.config_generic(F, seed=F, n_traj=1, n_steps=1)
    rg = np.sqrt(w8.gamma)
    a, b = rg[:, None], rg[None, :]
    for n_steps in (19, 64):
        w = w8.with_(n_traj=37, n_steps=n_steps)
        p0, q0, _ = oracle.sample_initial(w.gamma, w.p_eq, w.q_eq, 37, 3)
        g = gpu_propagate(G, w, p0, q0, precision=1, stab_tol=MIXED_STAB_TOL, fin=True)
        M = g["M"].reshape(37, 2 * F, 2 * F)
        pp, pq, qp, qq = M[:, :F, :F], M[:, :F, F:], M[:, F:, :F], M[:, F:, F:]
        A = 0.5 * ((a / b) * qq + (b / a) * pp + 1j * (-(a * b) * qp + pq / (a * b)))
        size = 0.5 * np.sqrt(((np.abs(a / b * qq) + np.abs(b / a * pp)) ** 2
                              + (np.abs(a * b * qp) + np.abs(pq / (a * b))) ** 2).sum((1, 2)))
        det = np.linalg.det(A)
        got = g["detA"][:, 0] + 1j * g["detA"][:, 1]
        bound = 3 * 2.0 ** -24 * size * np.linalg.norm(np.linalg.inv(A), axis=(1, 2)) + 1e-12
        assert np.all(np.abs(got - det) <= bound * np.abs(det))
        # and its argument is the phase's, modulo 2 pi
        turn = (g["theta"] - np.angle(got)) / (2 * np.pi)
        assert np.max(np.abs(turn - np.rint(turn))) <= 1e-9
