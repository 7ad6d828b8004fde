"""Mixed propagation above F = 13, where the warps of a CTA form the Hessians of two, four or
eight trajectories together: every number of trajectories per CTA, ragged last CTAs, staged and
streamed tensors, surfaces without one or both kinds of couplings."""
import numpy as np
import pytest

import oracle
from paper_1312_4698_gb300 import workloads as wl
from tests.test_gpu_parity import MIXED_STAB_TOL, amp_err, gpu_propagate

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    from paper_1312_4698_gb300 import scivr
    assert torch.cuda.is_available()
    return scivr


def _surface(F, form):
    w8 = wl.config_generic(F, seed=F, n_traj=1, n_steps=18)
    p = w8.pes
    none3, none4 = (np.zeros((0, 3)), np.zeros(0)), (np.zeros((0, 4)), np.zeros(0))
    c3 = (p.idx3, p.c3) if "3" in form else none3
    c4 = (p.idx4, p.c4) if "4" in form else none4
    kind = wl.DIAG_HARMONIC if form == "harmonic" else p.diag_kind
    return w8.with_(pes=wl.PesDesc(F, kind, p.omega, p.D, p.a, *c3, *c4))


@pytest.mark.parametrize("F,form", [(14, "34"), (15, "34"), (16, "34"), (17, "34"), (20, "34"), (22, "34"), (23, "34"),
                                    (24, "34"), (15, "3"), (15, "4"), (15, "none"), (24, "3"), (24, "4"),
                                    (24, "none"), (16, "harmonic"), (24, "harmonic")])
def test_trajectories_per_cta_give_the_same_trajectories(G, F, form):
    """Each entry's sum keeps its order whatever the tile, so a trajectory's amplitudes are the
    same bits in launches of 1, 303 (two per CTA), 605 (four) and 1221 (eight) trajectories; the
    first eight against the FP64 oracle.  Bound: 18 steps of an FP32 force and monodromy, about
    100 roundings of 2^-24 on phases of order 10, 1e-3 with room for the determinant's growth."""
    w8 = _surface(F, form)
    p0, q0, w = oracle.sample_initial(w8.gamma, w8.p_eq, w8.q_eq, 1221, 5)
    full = gpu_propagate(G, w8.with_(n_traj=1221), p0, q0, precision=1, stab_tol=MIXED_STAB_TOL)
    for n in (1, 303, 605):
        part = gpu_propagate(G, w8.with_(n_traj=n), np.ascontiguousarray(p0[:, :n]), np.ascontiguousarray(q0[:, :n]),
                             precision=1, stab_tol=MIXED_STAB_TOL)
        assert np.array_equal(part["amp"], full["amp"][:, :n], equal_nan=True)
        assert np.array_equal(part["good"], full["good"][:n])
    ra, rg = oracle.propagate(w8.pes, w8.gamma, w8.p_eq, w8.q_eq, w8.dt, w8.n_steps,
                              np.ascontiguousarray(p0[:, :8]), np.ascontiguousarray(q0[:, :8]))
    assert amp_err(full["amp"][:, :8], ra, rg) < 1e-3
