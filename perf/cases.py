"""What a user of this framework has it compute, as timed cases.

Each case is one pass through public entry points of ``paper_1312_4698_gb300.scivr``:

* ``path``       sample -> propagate -> spectrum, the whole call (``run_spectrum_path``)
* ``propagate``  the mixed-precision propagation alone, complex-float amplitude rows
* ``spectrum``   the time -> energy step alone, in one of its modes
* ``hk``         the plain Herman-Kluk spectrum from recorded summands
* ``mlp_eval``   the learned residual's value, gradient and Hessian at many points
* ``mlp_train``  one training step of the learned residual (loss, gradient, AdamW)
* ``mlp_prop``   propagation on a surface with a learned residual

``exact`` restates each of them in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

from paper_1312_4698_gb300 import scivr as G
from paper_1312_4698_gb300 import workloads as wl

DEV = "cuda"
HIDDEN = G.SCIVR_MLP_HIDDEN
MIXED_TOL = 1e-6 * 2.0 ** 29     # the FP64 stability threshold scaled by eps32 / eps64
FT_MODES = {"fp64": G.SCIVR_FT_FP64, "bf16": G.SCIVR_FT_TC_BF16, "bf16x3": G.SCIVR_FT_TC_BF16X3,
            "bf16x6": G.SCIVR_FT_TC_BF16X6, "czt64": G.SCIVR_FT_CZT64}


def listed():
    return [
        # the smallest whole run: a water-sized quick look with the library's default arithmetic
        {"name": "path_f3_small", "kind": "path", "F": 3, "n": 96, "steps": 400, "n_E": 300, "ft": "fp64"},
        # a formaldehyde-sized spectrum in FP64 throughout, as run to check a mixed one
        {"name": "path_f6_fp64", "kind": "path", "F": 6, "n": 4096, "steps": 2000, "n_E": 4000, "ft": "czt64"},
        # the formaldehyde-sized production propagation (full length)
        {"name": "prop_f6", "kind": "propagate", "F": 6, "n": 16384, "steps": 4000},
        # the methane-sized production propagation: the benchmark's trajectories, a fifth of its steps
        {"name": "prop_f9", "kind": "propagate", "F": 9, "n": 65536, "steps": 1000},
        # the middle of the molecule batch, an odd number of trajectories and steps
        {"name": "prop_f15", "kind": "propagate", "F": 15, "n": 3001, "steps": 501},
        # the largest molecules of the batch
        {"name": "prop_f24", "kind": "propagate", "F": 24, "n": 2048, "steps": 200},
        # production spectrum of a methane-sized run on the tensor cores
        {"name": "ft_bf16x3_f9", "kind": "spectrum", "F": 9, "n": 16384, "steps": 5000, "n_E": 4000,
         "ft": "bf16x3", "amp_f32": True},
        # FP64 spectrum of the water-sized run
        {"name": "ft_czt64_f3", "kind": "spectrum", "F": 3, "n": 1024, "steps": 3000, "n_E": 2000,
         "ft": "czt64", "amp_f32": False},
        # plain Herman-Kluk spectrum of the formaldehyde-sized run
        {"name": "hk_f6", "kind": "hk", "F": 6, "n": 16384, "steps": 4000, "n_E": 4000},
        # learned residual at one force stage of the methane-sized run
        {"name": "mlp_eval_f9", "kind": "mlp_eval", "F": 9, "n": 65536, "hessian": True},
        # training step of the learned residual at the benchmark's batch
        {"name": "mlp_train_f9", "kind": "mlp_train", "F": 9, "n": 16384},
        # propagation on the learned surface
        {"name": "mlp_prop_f9", "kind": "mlp_prop", "F": 9, "n": 16384, "steps": 20},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["path", "propagate", "propagate", "propagate", "spectrum", "spectrum", "hk", "mlp_eval",
                       "mlp_train", "mlp_prop"])
    if kind == "path":      # FP64 whole calls from quick looks to a fraction of a second
        F = rng.randint(1, 9)
        n, steps = _log(rng, 64, 8192), _log(rng, 100, 2000)
        while n * steps * F ** 3 > 8e8:
            n, steps = max(64, n * 2 // 3), max(100, steps * 4 // 5)
        return {"kind": kind, "F": F, "n": n, "steps": steps, "n_E": rng.randint(200, 4000),
                "ft": rng.choice(["fp64", "czt64"]) if n * steps < 4e5 else "czt64"}
    if kind == "propagate":  # every F of the mixed path
        F = rng.randint(1, 24)
        n, steps = _log(rng, 64, 65536), _log(rng, 64, 4000)
        while n * steps * F ** 3 > (4e10 if F <= 9 else 6e9 if F <= 16 else 3e9):
            n, steps = max(64, n * 2 // 3), max(64, steps * 4 // 5)
        return {"kind": kind, "F": F, "n": n, "steps": steps}
    if kind == "spectrum":
        ft = rng.choice(["bf16", "bf16x3", "bf16x6", "czt64", "czt64", "fp64"])
        n, steps, n_E = _log(rng, 64, 16384), _log(rng, 200, 6000), _log(rng, 200, 8000)
        most = 3.3e11 if ft.startswith("bf16") else 8e10 if ft == "czt64" else 8e9
        while n * steps * n_E > most:
            n = max(64, n * 2 // 3)
            steps, n_E = max(200, steps * 5 // 6), max(200, n_E * 5 // 6)
        return {"kind": kind, "F": rng.randint(1, 9), "n": n, "steps": steps, "n_E": n_E, "ft": ft,
                "amp_f32": rng.random() < 0.5}
    if kind == "hk":
        return {"kind": kind, "F": rng.randint(1, 9), "n": _log(rng, 64, 16384), "steps": _log(rng, 200, 4000),
                "n_E": _log(rng, 200, 4000)}
    if kind == "mlp_eval":
        return {"kind": kind, "F": rng.randint(1, 9), "n": _log(rng, 64, 65536), "hessian": rng.random() < 0.7}
    if kind == "mlp_train":
        return {"kind": kind, "F": rng.randint(1, 9), "n": _log(rng, 256, 16384)}
    return {"kind": kind, "F": rng.randint(1, 9), "n": _log(rng, 128, 16384), "steps": rng.randint(5, 20)}


# ---------------------------------------------------------------- inputs

def _molecule(F):
    """The repository's own workload of F modes."""
    if F == 3:
        return wl.config_f3()
    if F == 6:
        return wl.config_f6()
    if F == 9:
        return wl.config_f9()
    return wl.config_generic(F, F, 1, 1)


def _normals(shape, seed):
    return torch.randn(shape, dtype=torch.float64, device=DEV, generator=torch.Generator(DEV).manual_seed(seed))


def _husimi(w8, n, seed):
    """Initial conditions and weights of n Husimi-sampled trajectories."""
    z = _normals((2, w8.F, n), seed)
    gam = torch.as_tensor(w8.gamma, device=DEV)[:, None]
    q0 = torch.as_tensor(w8.q_eq[0], device=DEV)[:, None] + z[0] / gam.sqrt()
    p0 = torch.as_tensor(w8.p_eq[0], device=DEV)[:, None] + z[1] * gam.sqrt()
    return p0.contiguous(), q0.contiguous(), torch.exp(0.5 * (z * z).sum((0, 1)))


def _series(w8, n, K, hk, seed):
    """Amplitude rows [n, K, 2] of harmonic modes with a slightly different frequency in every
    trajectory (anharmonic detuning), their weights and good flags (one trajectory in a hundred bad)."""
    p0, q0, w = _husimi(w8, n, seed)
    gam = torch.as_tensor(w8.gamma, device=DEV)
    om = torch.as_tensor(w8.pes.omega, device=DEV)[:, None] * (1.0 + 0.02 * _normals((w8.F, n), seed + 7919))
    beta = (gam.sqrt()[:, None] * q0 + 1j * p0 / gam.sqrt()[:, None]) / math.sqrt(2.0)
    alpha = (gam.sqrt() * torch.as_tensor(w8.q_eq[0], device=DEV)
             + 1j * torch.as_tensor(w8.p_eq[0], device=DEV) / gam.sqrt()) / math.sqrt(2.0)
    t = torch.arange(K, dtype=torch.float64, device=DEV) * w8.dt
    out = torch.empty((n, K, 2), dtype=torch.float64, device=DEV)
    for j0 in range(0, n, 2048):
        sl = slice(j0, min(n, j0 + 2048))
        ex = torch.zeros((out[sl].shape[0], K), dtype=torch.complex128, device=DEV)
        for a in range(w8.F):
            turn = om[a, sl, None] * t
            ex += alpha[a].conj() * beta[a, sl, None] * torch.polar(torch.ones_like(turn), -turn) - 0.5j * turn
        norm = -0.5 * (alpha.abs() ** 2).sum() - 0.5 * (beta[:, sl].abs() ** 2).sum(0)
        ex = ex - ex[:, :1] if hk else ex + norm[:, None]   # Herman-Kluk summand: divided by the initial overlap
        out[sl] = torch.view_as_real(torch.exp(ex))
    good = (torch.rand(n, device=DEV, generator=torch.Generator(DEV).manual_seed(seed + 104729)) > 0.01)
    return out, w, good.to(torch.uint8)


def _network(w8, seed, s_out):
    m = wl.init_mlp(w8.F, HIDDEN, seed, s_in=np.sqrt(w8.pes.omega), s_out=s_out)
    rng = np.random.default_rng(seed + 100)
    m.b1, m.b2, m.b3 = (rng.normal(0.0, 0.3, HIDDEN) for _ in range(3))
    return m


def _diagonal(pes):
    return wl.PesDesc(pes.F, pes.diag_kind, pes.omega, pes.D, pes.a, np.zeros((0, 3)), np.zeros(0),
                      np.zeros((0, 4)), np.zeros(0))


def _points(w8, n, seed):
    """Points spread like those of sampled trajectories, q_i ~ N(0, 2 / omega_i)."""
    return _normals((n, w8.F), seed) * torch.as_tensor(np.sqrt(2.0 / w8.pes.omega), device=DEV)


def prepare(case, seed):
    kind, F, n = case["kind"], case["F"], case["n"]
    w8 = _molecule(F).with_(n_traj=n, seed=seed)
    s = {"kind": kind, "case": case, "seed": seed}
    if kind in ("path", "propagate", "spectrum", "hk", "mlp_prop"):
        w8 = w8.with_(n_steps=case["steps"], n_E=case.get("n_E", w8.n_E))
    s["w8"] = w8
    if kind == "path":
        s["pes"] = G.scivr_create_pes(w8.pes)
        s["bufs"] = G.alloc_buffers(w8)
    elif kind in ("propagate", "mlp_prop"):
        if kind == "mlp_prop":
            desc = _diagonal(w8.pes)
            desc.mlp = _network(w8, seed, 3e-6)
            s["w8"] = w8.with_(pes=desc)
        s["pes"] = G.scivr_create_pes(s["w8"].pes)
        s["p0"], s["q0"], _ = _husimi(w8, n, seed)
        s["amp"] = torch.empty((1, n, w8.n_steps + 1, 2), dtype=torch.float32, device=DEV)
        s["good"] = torch.empty(n, dtype=torch.uint8, device=DEV)
    elif kind in ("spectrum", "hk"):
        amp, s["w"], s["good"] = _series(w8, n, w8.n_steps + 1, kind == "hk", seed)
        s["amp"] = amp.float() if case.get("amp_f32") else amp
        s["I"] = torch.empty(w8.n_E, dtype=torch.float64, device=DEV)
        s["n_good"] = torch.zeros(1, dtype=torch.int64, device=DEV)
        if kind == "hk":
            s["C"] = torch.empty((w8.n_steps + 1, 2), dtype=torch.float64, device=DEV)
    else:
        q = _points(w8, n, seed)
        if kind == "mlp_train":   # targets: the coupling polynomial; the network scaled to their spread
            V, g, _ = _Couplings(w8.pes)(q, hess=False)
            if not w8.pes.c3.size:   # one mode has no couplings: learn a cubic of the dimensionless coordinate
                x = q * torch.as_tensor(np.sqrt(w8.pes.omega), device=DEV)
                V, g = 1e-6 * (x ** 3).sum(1), 3e-6 * x ** 2 * torch.as_tensor(np.sqrt(w8.pes.omega), device=DEV)
            s["V"], s["g"] = V.float().contiguous(), g.float().contiguous()
            s["alpha"], s["beta"] = 1.0 / float(V.var()), 1.0 / (float(g.var()) * F)
            s["net"] = _network(w8, seed, float(V.std()))
            npar = G.scivr_mlp_param_count(F)
            s["grad"], s["m1"], s["m2"] = (torch.zeros(npar, device=DEV) for _ in range(3))
            s["loss"], s["t"] = torch.zeros(1, device=DEV), 0
        else:
            s["net"] = _network(w8, seed, 3e-4)
            s["V"], s["g"] = torch.empty(n, device=DEV), torch.empty((n, F), device=DEV)
            s["H"] = torch.empty((n, F, F), device=DEV) if case["hessian"] else None
        desc = _diagonal(w8.pes)
        desc.mlp = s["net"]
        s["pes"] = G.scivr_create_pes(desc)
        s["q"] = q.float().contiguous()
    return s


# ---------------------------------------------------------------- one pass

def run(s):
    kind, w8, case = s["kind"], s["w8"], s["case"]
    n = case["n"]
    if kind == "path":
        b = s["bufs"]
        G.run_spectrum_path(s["pes"], w8, b, ft_mode=FT_MODES[case["ft"]])
        return {"I": b.I, "n_good": b.n_good, "good": b.good, "p0": b.p0, "q0": b.q0, "w": b.w}
    if kind in ("propagate", "mlp_prop"):
        G.scivr_propagate(s["pes"], w8.dt, w8.n_steps, w8.gamma, w8.p_eq, w8.q_eq, n, s["p0"], s["q0"], s["amp"],
                          w8.n_steps + 1, s["good"], precision=G.SCIVR_MIXED, stab_tol=MIXED_TOL)
        return {"amp": s["amp"], "good": s["good"]}
    if kind == "spectrum":
        G.scivr_spectrum(s["amp"], w8.n_steps + 1, s["w"], s["good"], n, w8.n_steps, w8.dt, w8.E_min, w8.E_max,
                         w8.n_E, s["I"], s["n_good"], ft_mode=FT_MODES[case["ft"]])
        return {"I": s["I"], "n_good": s["n_good"]}
    if kind == "hk":
        G.scivr_spectrum_hk(s["amp"], w8.n_steps + 1, s["good"], n, w8.n_steps, w8.dt, w8.E_min, w8.E_max, w8.n_E,
                            s["I"], s["C"], s["n_good"])
        return {"I": s["I"], "C": s["C"], "n_good": s["n_good"]}
    if kind == "mlp_eval":
        G.scivr_mlp_eval(s["pes"], n, s["q"], s["V"], s["g"], s["H"])
        return {"V": s["V"], "g": s["g"]} if s["H"] is None else {"V": s["V"], "g": s["g"], "H": s["H"]}
    s["t"] += 1
    G.scivr_mlp_loss_grad(s["pes"], n, s["q"], s["V"], s["g"], s["alpha"], s["beta"], s["grad"], s["loss"])
    G.scivr_mlp_adamw(s["pes"], s["grad"], s["m1"], s["m2"], s["t"], 1e-3)
    return {"loss": s["loss"], "grad": s["grad"], "m1": s["m1"], "m2": s["m2"]}


# ---------------------------------------------------------------- what a pass cannot do without

def _step_flops(F, mixed):
    """One trajectory step: three potential evaluations with their Hessians and monodromy kicks, four
    drifts, the stability determinant (every 16th step in mixed precision), the prefactor determinant
    and one amplitude."""
    P = F * (F + 1) // 2
    pes = 2 * (P + P * F + P * P + 4 * P) + 6 * F
    return (3 * (pes + 4 * F ** 3) + 16 * F * F + (16.0 / 3.0) * F ** 3 / (16 if mixed else 1) + 6 * F * F
            + (8.0 / 3.0) * F ** 3 + 32 * F + 60)


def _point_flops(F):
    """Value, gradient and Hessian of the network at one point."""
    R, H = F + 1, HIDDEN
    return 4 * F * H + 4 * R * H * H + 2 * H + 4 * H * H + 2 * F * H + 3 * F * (F + 1) * H


def work(case):
    kind, F, n = case["kind"], case["F"], case["n"]
    K, n_E = case.get("steps", 0) + 1, case.get("n_E", 0)
    tensors = 8 * (F * (F + 1) // 2) * (F + F * (F + 1) // 2)
    fft = 10 * 2 ** math.ceil(math.log2(K + n_E)) * math.ceil(math.log2(K + n_E)) + 20 * K   # chirp-z, per trajectory
    if kind == "path":
        ft = min(8.0 * K * n_E, fft) if case["ft"] == "czt64" else 8.0 * K * n_E
        return {"bytes": 8 * n * (2 * F + 1) + n + 8 * n_E + tensors,
                "flops": n * (case["steps"] * _step_flops(F, False) + ft)}
    if kind == "propagate":
        return {"bytes": 16 * F * n + 8 * n * K + n + tensors / 2, "flops": n * case["steps"] * _step_flops(F, True)}
    if kind == "spectrum":
        per = 8 if case["amp_f32"] else 16
        return {"bytes": per * n * K + 9 * n + 8 * n_E,
                "flops": n * (min(8.0 * K * n_E, fft) if case["ft"] == "czt64" else 8.0 * K * n_E)}
    if kind == "hk":
        return {"bytes": 16 * n * K + n + 16 * K + 8 * n_E, "flops": 2.0 * n * K + 4.0 * K * n_E}
    params = 4 * G.scivr_mlp_param_count(F)
    if kind == "mlp_eval":
        out = 4 * n * (1 + F + (F * F if case["hessian"] else 0))
        flops = _point_flops(F) if case["hessian"] else 8 * F * HIDDEN + 8 * HIDDEN ** 2
        return {"bytes": 4 * n * F + out + params, "flops": n * flops}
    if kind == "mlp_train":   # value and gradient, then the reverse pass over a pass with one direction
        return {"bytes": 4 * n * (2 * F + 1) + 7 * params, "flops": n * (8 + 24) * (HIDDEN ** 2 + F * HIDDEN)}
    return {"bytes": 16 * F * n + 8 * n * K + n + params,
            "flops": n * case["steps"] * (3 * _point_flops(F) + _step_flops(F, False))}


# ---------------------------------------------------------------- the same in 64 bits, plain torch

class _Couplings:
    """The cubic and quartic coupling polynomial from dense symmetric tensors: V, gradient, Hessian."""

    def __init__(self, pes):
        F = pes.F
        T3, T4 = np.zeros((F,) * 3), np.zeros((F,) * 4)
        for idx, c, T in ((pes.idx3, pes.c3, T3), (pes.idx4, pes.c4, T4)):
            d = T.ndim
            for pos in _permutations(d):   # d^deg V / dq: every order of the indices adds c
                if c.size:
                    np.add.at(T, tuple(idx[:, k] for k in pos), c)
        self.T3, self.T4 = torch.as_tensor(T3, device=DEV), torch.as_tensor(T4, device=DEV)

    def __call__(self, q, hess=True):
        n, F = q.shape
        H3 = (q @ self.T3.reshape(F, F * F)).reshape(n, F, F)
        qq = (q[:, :, None] * q[:, None, :]).reshape(n, F * F)
        H4 = 0.5 * (qq @ self.T4.reshape(F * F, F * F)).reshape(n, F, F)
        g3 = 0.5 * (H3 @ q[:, :, None])[..., 0]
        g4 = (H4 @ q[:, :, None])[..., 0] / 3.0
        V = (g3 * q).sum(1) / 3.0 + (g4 * q).sum(1) / 4.0
        return V, g3 + g4, (H3 + H4 if hess else None)


def _permutations(d):
    if d == 1:
        return [(0,)]
    return [p[:k] + (d - 1,) + p[k:] for p in _permutations(d - 1) for k in range(d)]


def _silu(z):
    s = torch.sigmoid(z)
    d1 = s * (1 + z * (1 - s))
    return z * s, d1, s * (1 - s) * (2 + z * (1 - 2 * s))


class _Net:
    """The learned residual: V, gradient, Hessian."""

    def __init__(self, m):
        self.p = [torch.as_tensor(np.asarray(x), dtype=torch.float64, device=DEV)
                  for x in (m.s_in, m.W1, m.b1, m.W2, m.b2, m.W3, m.b3, m.w4)]
        self.b4, self.s_out = float(m.b4), float(m.s_out)

    def value(self, q, p):
        x = q * self.p[0]
        for W, b in ((p[0], p[1]), (p[2], p[3]), (p[4], p[5])):
            x = torch.nn.functional.silu(x @ W.T + b)
        return self.s_out * (x @ p[6] + p[7])

    def __call__(self, q, hess=True):
        parts = [self._chunk(c, hess) for c in q.split(4096)]
        return tuple(None if x[0] is None else torch.cat(x) for x in zip(*parts))

    def _chunk(self, q, hess):
        s, W1, b1, W2, b2, W3, b3, w4 = self.p
        n, F = q.shape
        z1 = (q * s) @ W1.T + b1
        a1, d1, e1 = _silu(z1)
        z2 = a1 @ W2.T + b2
        a2, d2, e2 = _silu(z2)
        z3 = a2 @ W3.T + b3
        a3, d3, e3 = _silu(z3)
        V = self.s_out * (a3 @ w4 + self.b4)
        r3 = w4.expand_as(z3)                # dV / da_l (without s_out)
        r2 = (r3 * d3) @ W3
        r1 = (r2 * d2) @ W2
        g = self.s_out * ((r1 * d1) @ W1) * s
        if not hess:
            return V, g, None
        J1 = (W1 * s).T.expand(n, F, -1)     # dz_l / dq
        J2 = (J1 * d1[:, None]) @ W2.T
        J3 = (J2 * d2[:, None]) @ W3.T
        H = sum((J * (r * e)[:, None]) @ J.transpose(1, 2)
                for J, r, e in ((J1, r1, e1), (J2, r2, e2), (J3, r3, e3)))
        return V, g, self.s_out * H


def _propagate64(w8, p0, q0, potential):
    """Amplitudes [n, K, 2] and good flags: Yoshida's fourth-order triple jump of (p, q), the action and
    the monodromy, the Herman-Kluk phase followed relative to its harmonic rotation."""
    F, n = p0.shape
    pes = w8.pes
    om, D, a = (torch.as_tensor(x, device=DEV) for x in (pes.omega, pes.D, pes.a))
    gam = torch.as_tensor(w8.gamma, device=DEV)
    pe, qe = torch.as_tensor(w8.p_eq[0], device=DEV), torch.as_tensor(w8.q_eq[0], device=DEV)
    w1 = 1.0 / (2.0 - 2.0 ** (1.0 / 3.0))
    w0 = 1.0 - 2.0 * w1
    drift = [0.5 * w1 * w8.dt, 0.5 * (w0 + w1) * w8.dt, 0.5 * (w0 + w1) * w8.dt, 0.5 * w1 * w8.dt]
    kick = [w1 * w8.dt, w0 * w8.dt, w1 * w8.dt]
    p, q = p0.T.contiguous(), q0.T.contiguous()
    eye = torch.eye(2 * F, dtype=torch.float64, device=DEV).expand(n, -1, -1)
    Mp, Mq = eye[:, :F].clone(), eye[:, F:].clone()
    S, theta, arg = (torch.zeros(n, dtype=torch.float64, device=DEV) for _ in range(3))
    good = torch.ones(n, dtype=torch.bool, device=DEV)
    rg = gam.sqrt()
    c_qq, c_qp = rg[:, None] / rg[None, :], rg[:, None] * rg[None, :]
    turn = float(gam.sum()) * w8.dt
    out = torch.empty((n, w8.n_steps + 1, 2), dtype=torch.float64, device=DEV)

    def record(c):
        dq, dp = qe - q, pe - p
        re = -(0.25 * gam * dq * dq + dp * dp / (4.0 * gam)).sum(1)
        ph = (0.5 * (pe + p) * dq).sum(1) + S + 0.5 * theta
        out[:, c] = torch.view_as_real(torch.polar(torch.exp(re), ph))

    def step():
        nonlocal p, q, Mp, Mq, S
        for k in range(4):
            q = q + drift[k] * p
            S = S + drift[k] * 0.5 * (p * p).sum(1)
            Mq = Mq + drift[k] * Mp
            if k == 3:
                break
            V, g, H = potential(q)
            if pes.diag_kind == wl.DIAG_MORSE:
                u = torch.exp(-a * q)
                V = V + (D * (1 - u) ** 2).sum(1)
                g = g + 2 * D * a * u * (1 - u)
                h = 2 * D * a * a * u * (2 * u - 1)
            else:
                V, g, h = V + 0.5 * (om * om * q * q).sum(1), g + om * om * q, (om * om).expand_as(q)
            p = p - kick[k] * g
            S = S - kick[k] * V
            Mp = Mp - kick[k] * ((H + torch.diag_embed(h)) @ Mq)

    record(0)
    for c in range(1, w8.n_steps + 1):
        step()
        A = 0.5 * torch.complex(c_qq * Mq[..., F:] + Mp[..., :F] / c_qq, -c_qp * Mq[..., :F] + Mp[..., F:] / c_qp)
        new = torch.angle(torch.linalg.det(A))
        d = new - arg + turn
        theta, arg = theta + d - 2 * math.pi * torch.round(d / (2 * math.pi)) - turn, new
        det = torch.linalg.det(torch.cat([Mp, Mq], 1))
        good &= ((det * det - 1).abs() <= w8.stab_tol) & torch.isfinite(theta + S)
        record(c)
    return out, good.to(torch.uint8)


def _energies(w8):
    return torch.as_tensor(w8.energies(), device=DEV)


def _spectrum64(w8, amp, w, good):
    K = w8.n_steps + 1
    t = torch.arange(K, dtype=torch.float64, device=DEV) * w8.dt
    ph = t[:, None] * _energies(w8)
    tw = torch.polar(torch.ones_like(ph), ph)
    I = torch.zeros(w8.n_E, dtype=torch.float64, device=DEV)
    rows = torch.nonzero(good)[:, 0]
    for r in rows.split(2048):
        X = torch.view_as_complex(amp[r].double().contiguous()) @ tw
        I += (w[r, None] * (X.real ** 2 + X.imag ** 2)).sum(0)
    n_good = rows.shape[0]
    return I * (w8.dt ** 2 / (2 * math.pi * w8.n_steps * w8.dt * max(n_good, 1)))


def exact(case, seed):
    kind, F, n = case["kind"], case["F"], case["n"]
    if kind in ("path", "propagate", "mlp_prop"):   # a trajectory step takes launches and F^3 work per trajectory
        net = 2e-7 * (1 + F) if kind == "mlp_prop" else 0.0
        if case["steps"] * (8e-3 + n * (F ** 3 * 4e-9 + F ** 4 * 6e-12 + 3 * net)) > 30.0:
            return None
    if kind == "spectrum" and 8.0 * n * case["steps"] * case["n_E"] > 8e12:
        return None
    s = prepare(case, seed)
    w8 = s["w8"]
    if kind == "path":   # the sampler's initial conditions are taken as they are
        b = s["bufs"]
        G.scivr_sample_initial(s["pes"], w8.gamma, w8.p_eq[0], w8.q_eq[0], n, w8.seed, b.p0, b.q0, b.w)
        amp, good = _propagate64(w8, b.p0, b.q0, _Couplings(w8.pes))
        return {"I": _spectrum64(w8, amp, b.w, good)[None], "n_good": good.sum(dtype=torch.int64)[None], "good": good,
                "p0": None, "q0": None, "w": None}
    if kind == "propagate":
        amp, _ = _propagate64(w8, s["p0"], s["q0"], _Couplings(w8.pes))
        return {"amp": amp[None], "good": None}
    if kind == "mlp_prop":
        amp, _ = _propagate64(w8, s["p0"], s["q0"], _Net(w8.pes.mlp))
        return {"amp": amp[None], "good": None}
    if kind == "spectrum":
        return {"I": _spectrum64(w8, s["amp"], s["w"], s["good"]), "n_good": s["good"].sum(dtype=torch.int64)[None]}
    if kind == "hk":
        C = torch.view_as_complex(s["amp"])[s["good"].bool()].mean(0)
        t = torch.arange(w8.n_steps + 1, dtype=torch.float64, device=DEV) * w8.dt
        ph = _energies(w8)[:, None] * t[1:]
        I = w8.dt / math.pi * (0.5 * C[0].real + (C[1:].real * ph.cos() - C[1:].imag * ph.sin()).sum(1))
        return {"I": I, "C": torch.view_as_real(C), "n_good": s["good"].sum(dtype=torch.int64)[None]}
    net = _Net(s["net"])
    q = s["q"].double()
    if kind == "mlp_eval":
        V, g, H = net(q, case["hessian"])
        return {"V": V, "g": g, "H": H} if case["hessian"] else {"V": V, "g": g}
    par = [x.clone().requires_grad_() for x in net.p[1:]] + [torch.tensor(net.b4, dtype=torch.float64, device=DEV,
                                                                          requires_grad=True)]
    q.requires_grad_()
    V = net.value(q, par)
    (g,) = torch.autograd.grad(V.sum(), q, create_graph=True)
    loss = (s["alpha"] * (V - s["V"].double()) ** 2 + s["beta"] * ((g - s["g"].double()) ** 2).sum(1)).mean()
    grad = torch.cat([x.reshape(-1) for x in torch.autograd.grad(loss, par)])
    return {"loss": loss.detach()[None], "grad": grad, "m1": 0.1 * grad, "m2": 1e-3 * grad * grad}
