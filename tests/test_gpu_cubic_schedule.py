"""Mixed propagation at F = 14..23 of surfaces without quartic terms, which has kernels of its own:
against the kernels of the general surface, which a quartic term of coefficient zero selects."""
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


def _surface(F, form, general=False):
    w8 = wl.config_generic(F, seed=F, n_traj=1, n_steps=1)
    p = w8.pes
    c3 = (p.idx3, p.c3) if form == "cubic" else (np.zeros((0, 3)), np.zeros(0))
    c4 = (np.array([[0, 0, 1, 1]]), np.zeros(1)) if general else (np.zeros((0, 4)), np.zeros(0))
    kind = wl.DIAG_HARMONIC if form == "harmonic" else p.diag_kind
    return w8.with_(pes=wl.PesDesc(F, kind, p.omega, p.D, p.a, *c3, *c4))


@pytest.mark.parametrize("F,form,n,steps", [
    *[(F, form, 37, 19) for F in (14, 16, 17, 20, 23) for form in ("cubic", "morse", "harmonic")],
    (15, "cubic", 1, 1), (17, "cubic", 1, 2), (18, "cubic", 5, 33), (19, "morse", 4, 16), (21, "cubic", 611, 5),
    (22, "cubic", 1221, 4),
])
def test_agrees_with_the_general_kernels(G, F, form, n, steps):
    """Forces and Hessians are the same multiply-adds, above F = 16 and without couplings in the same
    order, so that positions, momenta and M are the same bits there; with cubic terms at F <= 16 the
    general kernel adds four partial sums.  Bound for all the rest, as for the trajectories of those
    kernels against the oracle: 1e-3 of a row's largest amplitude after up to 33 steps in FP32, and
    3 2^-24 of the entries of A, with room for their number, on det A."""
    w8 = _surface(F, form).with_(n_traj=n, n_steps=steps)
    ref8 = _surface(F, form, general=True).with_(n_traj=n, n_steps=steps)
    p0, q0, _ = oracle.sample_initial(w8.gamma, w8.p_eq, w8.q_eq, n, 7)
    a = gpu_propagate(G, w8, p0, q0, precision=1, stab_tol=MIXED_STAB_TOL, fin=True)
    b = gpu_propagate(G, ref8, p0, q0, precision=1, stab_tol=MIXED_STAB_TOL, fin=True)
    assert np.array_equal(a["good"], b["good"])
    if F > 16 or form != "cubic":
        for k in ("p", "q", "M", "detM"):
            assert np.array_equal(a[k], b[k], equal_nan=True), k
    assert amp_err(a["amp"], b["amp"], b["good"]) < 1e-3
    za, zb = a["detA"] @ [1, 1j], b["detA"] @ [1, 1j]
    assert np.max(np.abs(za - zb) / np.abs(zb)) < 1e-3
    m = min(n, 6)
    ra, rg = oracle.propagate(w8.pes, w8.gamma, w8.p_eq, w8.q_eq, w8.dt, steps, np.ascontiguousarray(p0[:, :m]),
                              np.ascontiguousarray(q0[:, :m]))
    assert amp_err(a["amp"][:, :m], ra, rg) < 1e-3


@pytest.mark.parametrize("schedule", ["per-class", "one"])
def test_batch_of_surfaces_with_and_without_quartic_terms(G, monkeypatch, schedule):
    """Molecules of one F with and without quartic terms make two groups of the plan, and every molecule
    equals its own call bit for bit; the one-launch schedule runs the general body for all (F = 15:
    1e-5 of a row's largest amplitude, as for the molecules of that schedule)."""
    import torch
    monkeypatch.setenv("SCIVR_BATCH_SCHEDULE", schedule)
    Fs = (15, 17, 15, 17) if schedule == "per-class" else (15, 9, 15, 24)
    entries = []
    for i, F in enumerate(Fs):
        w8 = wl.config_generic(F, seed=F, n_traj=70 + 9 * i, n_steps=21 + 5 * i, n_E=100)
        if i < 2:
            w8 = _surface(F, "cubic").with_(n_traj=w8.n_traj, n_steps=w8.n_steps, n_E=100)
        pes, b = G.scivr_create_pes(w8.pes), G.alloc_buffers(w8)
        G.scivr_sample_initial(pes, w8.gamma, w8.p_eq[0], w8.q_eq[0], w8.n_traj, 3, b.p0, b.q0, b.w)
        entries.append(dict(pes=pes, wl=w8, bufs=b, precision=1, stab_tol=MIXED_STAB_TOL))
    plan = G.scivr_batch_create(entries, ft_mode=2)
    if schedule == "per-class":
        assert sorted(F for F, _, _ in plan.groups()) == [15, 15, 17, 17]
    else:
        assert plan.one_launch()
    G.scivr_batch_launch(plan)
    torch.cuda.synchronize()
    for e in entries:
        w8, b = e["wl"], e["bufs"]
        amp, good = torch.empty_like(b.amp), torch.empty_like(b.good)
        G.scivr_propagate(e["pes"], w8.dt, w8.n_steps, w8.gamma, w8.p_eq, w8.q_eq, w8.n_traj, b.p0, b.q0, amp,
                          w8.n_steps + 1, good, precision=1, stab_tol=MIXED_STAB_TOL)
        assert torch.equal(b.good, good)
        if schedule == "per-class" or w8.F in (9, 24):
            assert torch.equal(b.amp, amp)
        else:
            d = (b.amp - amp).square().sum(-1).sqrt().amax(-1) / amp.square().sum(-1).sqrt().amax(-1)
            assert float(d[..., good.bool()].max()) < 1e-5
