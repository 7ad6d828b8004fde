"""FP64 lane groups of every size (chosen by the number of trajectories) against the
thread-per-trajectory schedule on the same inputs.

Both are FP64 with other summation orders, so they differ by rounding: amplitudes, final states and
determinants to 1e-9 relative, the bound the schedules have against the oracle; flags equal.
"""
import numpy as np
import pytest

from paper_1312_4698_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _propagate(G, w8, p0, q0, kernel, amplitude):
    import torch
    F, n = p0.shape
    K = w8.n_steps + 1
    f64 = dict(dtype=torch.float64, device="cuda")
    pes = G.scivr_create_pes(w8.pes)
    amp = torch.full((w8.n_chi, n, K, 2), float("nan"), **f64)
    good = torch.empty(n, dtype=torch.uint8, device="cuda")
    fin = dict(p=torch.empty((F, n), **f64), q=torch.empty((F, n), **f64), S=torch.empty(n, **f64),
               theta=torch.empty(n, **f64), detM=torch.empty(n, **f64), detA=torch.empty((n, 2), **f64),
               M=torch.empty((n, 2 * F, 2 * F), **f64), stab=torch.empty(n, **f64))
    G.scivr_propagate(pes, w8.dt, w8.n_steps, w8.gamma, w8.p_eq, w8.q_eq, n, torch.as_tensor(p0, device="cuda"),
                      torch.as_tensor(q0, device="cuda"), amp, K, good, precision=0, stab_tol=w8.stab_tol, fin=fin,
                      kernel=kernel, amplitude=amplitude)
    torch.cuda.synchronize()
    return amp.cpu().numpy(), good.cpu().numpy(), {k: v.cpu().numpy() for k, v in fin.items()}


def _surface(F, kind):
    w8 = {3: wl.config_f3, 6: wl.config_f6, 9: wl.config_f9}.get(F, lambda: wl.config_generic(F, F, 1, 1))()
    pes = w8.pes
    no3, no4 = (np.zeros((0, 3)), np.zeros(0)), (np.zeros((0, 4)), np.zeros(0))
    i3, c3 = no3 if kind in ("diagonal", "quartic", "harmonic") else (pes.idx3, pes.c3)
    i4, c4 = no4 if kind in ("diagonal", "cubic", "harmonic") else (pes.idx4, pes.c4)
    diag = wl.DIAG_HARMONIC if kind == "harmonic" else pes.diag_kind
    return w8.with_(pes=wl.PesDesc(F, diag, pes.omega, pes.D, pes.a, i3, c3, i4, c4))


# sizes: one trajectory; around 608 warps of 32-, 16- and 8-lane groups; 4-lane groups (8 at F >= 7)
# with a ragged last warp; step counts: one step, part of a chunk, several chunks with a rest
@pytest.mark.parametrize("F,n,steps,kind,amplitude", [
    *[(F, n, 37, "full", 0) for F in range(1, 10) for n in (1, 609, 1217, 2437)],
    (1, 4867, 5, "full", 0), (3, 4867, 37, "full", 1), (6, 4867, 1, "full", 0), (9, 2437, 3, "full", 1),
    (6, 609, 33, "full", 1), (9, 17, 31, "full", 1),
    # a second warp makes the records: one and two sets of trajectories per CTA, 1, 2 and 3 steps in its two slots
    (6, 150, 1, "full", 0), (6, 303, 2, "full", 0), (6, 305, 3, "full", 1), (9, 300, 33, "full", 0), (5, 305, 18, "full", 0),
    *[(6, 1217, 9, kind, 0) for kind in ("diagonal", "cubic", "quartic", "harmonic")],
])
def test_group_sizes_agree_with_the_thread_schedule(F, n, steps, kind, amplitude):
    from paper_1312_4698_gb300 import scivr as G
    w8 = _surface(F, kind).with_(n_traj=n, n_steps=steps)
    rng = np.random.default_rng(100 * F + n)
    gam = np.asarray(w8.gamma)[:, None]
    q0 = np.asarray(w8.q_eq)[0][:, None] + rng.standard_normal((F, n)) / np.sqrt(gam)
    p0 = np.asarray(w8.p_eq)[0][:, None] + rng.standard_normal((F, n)) * np.sqrt(gam)
    if n > 1:
        q0[:, n // 2] = -1e100   # one trajectory leaves the numbers' range; its neighbours must not notice
    a, ga, fa = _propagate(G, w8, p0, q0, G.SCIVR_KERNEL_THREAD, amplitude)
    b, gb, fb = _propagate(G, w8, p0, q0, G.SCIVR_KERNEL_GROUP, amplitude)
    assert np.array_equal(ga, gb)
    rows = ga.astype(bool)
    if n > 1:
        rows[n // 2] = False
    assert rows.sum() >= n // 2
    assert np.abs(a[:, rows] - b[:, rows]).max() <= 1e-9 * np.abs(a[:, rows]).max()
    for k in fa:
        x, y = (fa[k][:, rows], fb[k][:, rows]) if k in ("p", "q") else (fa[k][rows], fb[k][rows])
        tol = 1e-9 * max(np.abs(x).max(), 1.0) if k != "stab" else 1e-9
        assert np.abs(x - y).max() <= tol, k
