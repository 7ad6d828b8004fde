"""The split-step kernels of the learned-residual path, with a network whose output is scaled to nothing
(1e-30), against the FP64 thread schedule on the analytic surface alone.

Positions, momenta and the action are FP64 on both sides: they agree to 1e-10 of their largest value.  The
monodromy is FP32 on the learned path: 7 sub-flows a step of up to F rounded terms each, 23 steps x 63 x 2^-24 =
9e-5 at F = 9 if all errors added up; 1e-4 of the largest entry bounds M, and with it det A and the phase
(whose amplitudes rotate by half of it).
"""
import numpy as np
import pytest

from paper_1312_4698_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _run(G, w8, p0, q0, precision, kernel, amplitude):
    import torch
    F, n = p0.shape
    K = w8.n_steps + 1
    f64 = dict(dtype=torch.float64, device="cuda")
    amp = torch.full((w8.n_chi, n, K, 2), float("nan"), **f64)
    good = torch.empty(n, dtype=torch.uint8, device="cuda")
    fin = dict(p=torch.empty((F, n), **f64), q=torch.empty((F, n), **f64), S=torch.empty(n, **f64),
               theta=torch.empty(n, **f64), detM=torch.empty(n, **f64), detA=torch.empty((n, 2), **f64),
               M=torch.empty((n, 2 * F, 2 * F), **f64), stab=torch.empty(n, **f64))
    G.scivr_propagate(G.scivr_create_pes(w8.pes), w8.dt, w8.n_steps, w8.gamma, w8.p_eq, w8.q_eq, n,
                      torch.as_tensor(p0, device="cuda"), torch.as_tensor(q0, device="cuda"), amp, K, good,
                      precision=precision, stab_tol=1e-6 * 2.0 ** 29, fin=fin, kernel=kernel, amplitude=amplitude)
    torch.cuda.synchronize()
    return amp.cpu().numpy(), good.cpu().numpy(), {k: v.cpu().numpy() for k, v in fin.items()}


@pytest.mark.parametrize("F,n,steps,coupled,diag,amplitude", [
    (1, 1, 23, False, "morse", 0), (2, 33, 1, True, "morse", 1), (3, 32, 23, True, "harmonic", 0),
    (5, 31, 23, True, "morse", 0), (6, 70, 7, False, "harmonic", 1), (8, 33, 23, True, "morse", 1),
    (9, 33, 23, False, "morse", 0), (9, 65, 23, True, "morse", 0)])
def test_stages_with_a_vanishing_network(F, n, steps, coupled, diag, amplitude):
    from paper_1312_4698_gb300 import scivr as G
    w8 = {3: wl.config_f3, 6: wl.config_f6, 9: wl.config_f9}.get(F, lambda: wl.config_generic(F, F, 1, 1))()
    pes = w8.pes
    kind = wl.DIAG_HARMONIC if diag == "harmonic" else pes.diag_kind
    c = (pes.idx3, pes.c3, pes.idx4, pes.c4) if coupled else (np.zeros((0, 3)), np.zeros(0), np.zeros((0, 4)), np.zeros(0))
    w8 = w8.with_(pes=wl.PesDesc(F, kind, pes.omega, pes.D, pes.a, *c), n_traj=n, n_steps=steps)
    rng = np.random.default_rng(31 * F + n)
    gam = np.asarray(w8.gamma)[:, None]
    q0 = np.asarray(w8.q_eq)[0][:, None] + rng.standard_normal((F, n)) / np.sqrt(gam)
    p0 = np.asarray(w8.p_eq)[0][:, None] + rng.standard_normal((F, n)) * np.sqrt(gam)
    if n > 1:
        q0[:, n // 2] = -1e100   # leaves the numbers' range: flagged, and alone in that
    a, ga, fa = _run(G, w8, p0, q0, G.SCIVR_FP64, G.SCIVR_KERNEL_THREAD, amplitude)
    w8.pes.mlp = wl.init_mlp(F, 256, 3, s_in=np.sqrt(pes.omega), s_out=1e-30)
    b, gb, fb = _run(G, w8, p0, q0, G.SCIVR_MIXED, G.SCIVR_KERNEL_AUTO, amplitude)
    rows = np.ones(n, bool)
    if n > 1:
        rows[n // 2] = False
        assert gb[n // 2] == 0 or diag == "harmonic"
    assert ga[rows].all() and gb[rows].all()
    for k, tol in (("p", 1e-10), ("q", 1e-10), ("S", 1e-10), ("M", 1e-4), ("theta", 1e-4), ("detA", 1e-4)):
        x, y = (fa[k][:, rows], fb[k][:, rows]) if k in ("p", "q") else (fa[k][rows], fb[k][rows])
        assert np.abs(x - y).max() <= tol * max(np.abs(x).max(), 1e-3 if k in ("p", "q", "S") else 1.0), k
    assert np.abs(fb["detM"][rows] - 1.0).max() <= 1e-4 * F
    assert np.abs(a[:, rows] - b[:, rows]).max() <= 1e-4 * np.abs(a[:, rows]).max()
