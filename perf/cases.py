"""Performance cases: the work that a user of this package has it do.

Every case goes through the public entry points (`modal.Simulator`,
`modal.simulate_autograd`, `proposal.features`, `proposal.MLP`).  The kinds:

  block        one short block of a string with its state carried over: the
               call of a real-time audio callback (latency and launches count)
  string       one plucked, tension-modulated string, a whole sound
  strings_fit  a batch of strings, forward with checkpoints and the adjoint: one
               step of an inverse fit
  plate        one von Karman plate, a whole sound
  dataset      a batch of strings and plates of uneven sizes, forward only:
               training data of the learned proposal
  plates_fit   a batch of plates of several aspects, forward and adjoint with the
               aspect direction: one step of the benchmark's inverse fit
  groups       plates that share geometries, and membranes, forward: a bank of
               percussion voices stepped together
  coupling_fit small plates with unstructured coupling tensors, forward and
               adjoint with the full dL/dH: one step of a coupling fit
  linear       the linear response of strings, membranes and plates
  features     log-mel features of a batch of sounds
  mlp          one training pass of the proposal network (loss, gradients)

`listed()` holds one or two sizes of each kind, `draw(rng)` others of the same
ranges.  `exact` evaluates the same definitions step by step in 64 bits with
plain torch operations.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2505_05940_gb300 import coupling, modal, physics, proposal
from paper_2505_05940_gb300 import workloads as W

FS = 44100.0
STEEL_D = 18.315               # bending stiffness of a 1 mm steel plate (N m)


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # a plug-in's audio callback: 8 partials, 64 samples, state in and out
        dict(name="block_string8_64", kind="block", n=8, steps=64),
        # one second of the 40-mode string at 48 kHz
        dict(name="string40_48000", kind="string", n=40, steps=48000),
        # an inverse fit of 48 strings with 40 to 100 modes on 0.1 s of audio
        dict(name="strings_fit48_4410", kind="strings_fit", inst=48, n_min=40, n_max=100,
             steps=4410, K=1024),
        # a quarter of a second of the 100 x 30 plate
        dict(name="plate100x30_11025", kind="plate", n=100, m=30, steps=11025),
        # 96 sounds of the proposal's training data: half strings, half plates
        dict(name="dataset96_11025", kind="dataset", inst=96, n_min=50, n_max=200, steps=11025),
        # the fit of 64 plates (200 x 50) on 0.1 s of audio
        dict(name="plates_fit64_200x50_4410", kind="plates_fit", inst=64, n=200, m=50,
             steps=4410, K=1024),
        # a few smaller plates with an odd size, a short checkpoint interval
        dict(name="plates_fit6_117x29_3001", kind="plates_fit", inst=6, n=117, m=29,
             steps=3001, K=256),
        # 160 plates and membranes of 20 to 400 modes on 4 shared geometries, 50 ms
        dict(name="groups160_2205", kind="groups", inst=160, n_min=20, n_max=400, geoms=4,
             steps=2205),
        # eight candidate tensors of a 16 x 4 plate, 0.1 s
        dict(name="coupling_fit8_16x4_4410", kind="coupling_fit", inst=8, n=16, m=4, steps=4410,
             K=1024),
        # half a second of linear response of 64 objects
        dict(name="linear64_22050", kind="linear", inst=64, n_min=20, n_max=400, steps=22050),
        # features of one simulated batch of the training set
        dict(name="features1024_11025", kind="features", batch=1024, T=11025),
        # one training pass at the proposal's batch size
        dict(name="mlp_train256", kind="mlp", batch=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["block", "string", "strings_fit", "plate", "dataset", "plates_fit",
                       "plates_fit", "groups", "coupling_fit", "linear", "features", "mlp"])
    if kind == "block":
        return dict(kind=kind, n=_log_int(rng, 4, 100), steps=_log_int(rng, 32, 512))
    if kind == "string":
        return dict(kind=kind, n=_log_int(rng, 20, 100), steps=_log_int(rng, 4410, 48000))
    if kind == "strings_fit":
        return dict(kind=kind, inst=_log_int(rng, 1, 128), n_min=40, n_max=100,
                    steps=_log_int(rng, 2205, 4410), K=rng.choice([256, 500, 1024]))
    if kind == "plate":
        n = rng.randint(40, 128)
        return dict(kind=kind, n=n, m=rng.randint(max(4, n // 5), n // 3),
                    steps=_log_int(rng, 4410, 11025))
    if kind == "dataset":
        return dict(kind=kind, inst=_log_int(rng, 12, 96), n_min=50, n_max=200,
                    steps=_log_int(rng, 4410, 11025))
    if kind == "plates_fit":
        n = rng.randint(60, 200)
        return dict(kind=kind, inst=_log_int(rng, 1, 64), n=n, m=max(1, n // 4),
                    steps=_log_int(rng, 1500, 4410), K=rng.choice([256, 1000, 1024]))
    if kind == "groups":
        return dict(kind=kind, inst=_log_int(rng, 32, 160), n_min=20,
                    n_max=rng.randint(200, 400), geoms=rng.randint(2, 6),
                    steps=_log_int(rng, 1000, 2205))
    if kind == "coupling_fit":
        n = rng.randint(10, 24)
        return dict(kind=kind, inst=rng.randint(2, 12), n=n, m=max(2, n // 4),
                    steps=_log_int(rng, 2205, 4410), K=rng.choice([256, 1024]))
    if kind == "linear":
        return dict(kind=kind, inst=_log_int(rng, 4, 64), n_min=20, n_max=400,
                    steps=_log_int(rng, 4410, 22050))
    if kind == "features":
        return dict(kind=kind, batch=_log_int(rng, 64, 1024), T=rng.randint(4410, 11025))
    return dict(kind=kind, batch=_log_int(rng, 32, 256))


# ------------------------------------------------------------------ inputs

@functools.lru_cache(maxsize=None)
def _tensors(aspect, n, m, derivative):
    """Mode labels, coupling tensor, zeta^4, stress classes and (optionally) the
    aspect derivatives of one geometry: the offline input of a plan."""
    inst = W.Instance(kind="plate", n_phi=n, aspect=aspect)
    labels = physics.mode_labels(inst, n)
    if derivative:
        H, z, dH, dz, kc = coupling.coupling_with_aspect_derivative(inst.area, aspect, labels, m)
        return labels, H.astype(np.float32), z, kc, dH.astype(np.float32), dz
    lx, ly = coupling.sides(inst.area, aspect)
    airy = coupling.airy_modes(lx, ly, m)
    H, z = coupling.coupling_tensor(lx, ly, labels, m, airy=airy)
    return labels, H.astype(np.float32), z, coupling.airy_classes(airy[1]), None, None


def _from_bank(n, m, derivative=False):
    """Coupling of an instance as the leading block of its geometry's tensors."""
    def cp(inst, labels, M):
        _, H, z, kc, _, _ = _tensors(float(inst.aspect), n, m, derivative)
        N = len(labels)
        return H[:M, :N, :N], z[:M], kc[:M]
    return cp


def _string(rng, n, **kw):
    lu = lambda centre, dec: float(centre * 10.0 ** rng.uniform(-dec, dec))
    # up to 100 modes stay below the stability bound at 44.1 kHz
    return W.Instance(kind="string", n_phi=n, length=1.0, rho_lin=1e-3, T0=lu(30.0, 0.2),
                      D=lu(1e-4, 0.2), sigma0=lu(0.5, 0.3), sigma1=lu(1e-5, 0.3),
                      EA=lu(15853.0, 0.3), pickup=(float(rng.uniform(0.55, 0.9)),), **kw)


def _plate(rng, n, m, aspect, dec=0.3, T0=100.0):
    lu = lambda centre: float(centre * 10.0 ** rng.uniform(-dec, dec))
    return W.Instance(kind="plate", n_phi=n, n_psi=m, aspect=float(aspect), thickness=1e-3,
                      rho_lin=7.8, T0=lu(T0), D=lu(STEEL_D), sigma0=lu(1.0), sigma1=lu(3e-6),
                      strike=(float(rng.uniform(0.2, 0.4)), float(rng.uniform(0.3, 0.45))),
                      pickup=(float(rng.uniform(0.6, 0.8)), float(rng.uniform(0.55, 0.7))))


def _sizes(case):
    """Log-uniform mode counts of a batch: they belong to the case, not to the seed."""
    rng = np.random.default_rng([case["inst"], case["steps"], case["n_min"], case["n_max"]])
    return np.floor(np.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"] + 1),
                                       size=case["inst"]))).astype(int)


def _instances(case, seed):
    """The prepared instances of a simulation case (modal inputs on the host)."""
    kind = case["kind"]
    rng = np.random.default_rng([seed, len(kind), case["steps"]])
    steps = case["steps"]
    pick = np.random.default_rng([case["steps"], case.get("inst", 1)])   # geometries, too
    if kind in ("block", "string"):
        fs = 48000.0
        inst = _string(rng, case["n"], excitation="pluck", pluck_amp=5e-3,
                       pluck_x0=float(rng.uniform(0.2, 0.45)), pluck_width=0.1)
        return [physics.prepare(inst, fs, steps)]
    if kind == "strings_fit":
        return [physics.prepare(_string(rng, int(n), excitation="strike", F0=1.0,
                                        strike=(float(rng.uniform(0.1, 0.45)),)), FS, steps)
                for n in _sizes(case)]
    if kind == "plate":
        inst = _plate(rng, case["n"], case["m"], 1.5, T0=1.0)
        return [physics.prepare(inst, FS, steps, coupling=_from_bank(case["n"], case["m"]))]
    if kind == "dataset":
        n1 = case["n_max"]
        cp = _from_bank(n1, n1 // 4)
        out = []
        for i, n in enumerate(_sizes(case)):
            if i % 2:
                inst = _plate(rng, int(n), int(n) // 4, pick.choice([0.7, 1.0, 1.4, 1.8]), dec=0.5)
            else:
                inst = _string(rng, int(n) // 2 + 15, excitation="strike", F0=1.0,
                               strike=(float(rng.uniform(0.1, 0.45)),))
            out.append(physics.prepare(inst, FS, steps, coupling=cp))
        return out
    if kind == "plates_fit":
        n, m = case["n"], case["m"]
        out = []
        for i in range(case["inst"]):
            inst = _plate(rng, n, m, pick.choice([1.1, 1.3, 1.5, 1.7]))
            p = physics.prepare(inst, FS, steps, coupling=_from_bank(n, m, True))
            N, M = len(p["omega2"]), len(p["kappa"])
            _, _, _, _, dH, dz = _tensors(float(inst.aspect), n, m, True)
            p["dH"], p["dzeta4"] = dH[:M, :N, :N], dz[:M]
            out.append(p)
        return out
    if kind == "groups":
        n1 = case["n_max"]
        aspects = np.linspace(0.5, 2.0, case["geoms"])
        cp = _from_bank(n1, n1 // 4)
        out = []
        for i, n in enumerate(_sizes(case)):
            g = int(pick.integers(case["geoms"]))
            if i % 2:
                inst = _plate(rng, int(n), max(1, int(n) // 4), aspects[g], dec=0.5, T0=1.0)
            else:
                inst = W.Instance(kind="membrane", n_phi=int(n), aspect=float(aspects[g]),
                                  thickness=1e-3, rho_lin=7.8,
                                  T0=float(100.0 * 10.0 ** rng.uniform(-0.5, 1.0)), sigma0=1.0,
                                  sigma1=3e-6, F0=1.0, strike=(0.45, 0.45), pickup=(0.55, 0.52))
            p = physics.prepare(inst, FS, steps, coupling=cp)
            if i % 2:
                p["geom_group"] = 1 + g
            out.append(p)
        return out
    if kind == "coupling_fit":
        inst = W.Instance(kind="plate", n_phi=case["n"], n_psi=case["m"], aspect=1.3,
                          thickness=1e-3, rho_lin=7.8, T0=30.0, D=STEEL_D, sigma0=1.0,
                          sigma1=3e-6, F0=300.0)
        p = physics.prepare(inst, FS, steps)
        H = np.asarray(p["H"], np.float64)
        s = math.sqrt(np.mean(H ** 2))
        out = []
        for i in range(case["inst"]):
            R = rng.standard_normal(H.shape)
            d = {k: v for k, v in p.items() if k not in ("phi_class", "psi_class")}
            d["H"] = (s * 0.5 * (R + R.transpose(0, 2, 1))).astype(np.float32)
            out.append(d)
        return out
    # linear: strings, membranes and plates with the nonlinear terms off
    out = []
    for i, n in enumerate(_sizes(case)):
        if i % 3 == 0:
            inst = _string(rng, min(int(n), 100), excitation="strike", F0=1.0, strike=(0.3,))
        elif i % 3 == 1:
            inst = W.Instance(kind="membrane", n_phi=int(n), aspect=float(rng.uniform(0.5, 2.0)),
                              thickness=1e-3, rho_lin=7.8, T0=100.0, sigma0=1.0, sigma1=3e-6,
                              F0=1.0, strike=(0.45, 0.45), pickup=(0.55, 0.52))
        else:
            inst = _plate(rng, int(n), 0, rng.uniform(0.5, 2.0))
        out.append(physics.prepare(inst, FS, steps, coupling=None))
    return out


def _d_audio(case, seed, n_inst):
    """dL/dy of a spectral loss: noise-like, different for every instance."""
    rng = np.random.default_rng([seed, 7])
    return rng.standard_normal((n_inst, case["steps"])).astype(np.float32)


def _sounds(case, seed):
    """Decaying partials over a low noise floor [batch, T]."""
    rng = np.random.default_rng([seed, 11])
    B, T = case["batch"], case["T"]
    t = np.arange(T, dtype=np.float32) / np.float32(FS)
    y = 1e-4 * rng.standard_normal((B, T), dtype=np.float32)
    for p in range(3):
        f = rng.uniform(60.0, 9000.0, (B, 1)).astype(np.float32)
        d = rng.uniform(2.0, 30.0, (B, 1)).astype(np.float32)
        y += np.float32(1e-2 / (p + 1)) * np.exp(-d * t) * np.sin(np.float32(2 * np.pi) * f * t)
    return y


DIMS = (1024, 512, 512, 512, 6)


def _mlp_data(case, seed):
    rng = np.random.default_rng([seed, 13])
    x = rng.standard_normal((case["batch"], DIMS[0]), dtype=np.float32)
    y = rng.standard_normal((case["batch"], DIMS[-1]), dtype=np.float32)
    return x, y


def _dev(a):
    return torch.tensor(a, device="cuda:0")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "features":
        return dict(kind=kind, audio=_dev(_sounds(case, seed)))
    if kind == "mlp":
        x, y = _mlp_data(case, seed)
        net = proposal.MLP(DIMS, seed=seed)
        return dict(kind=kind, net=net, x=_dev(x).to(torch.bfloat16), target=_dev(y))
    preps = _instances(case, seed)
    st = dict(kind=kind, sim=modal.Simulator(preps), steps=case["steps"], K=case.get("K", 0))
    if kind in ("strings_fit", "plates_fit", "coupling_fit"):
        st["d_audio"] = _dev(_d_audio(case, seed, len(preps)))
    return st


# ------------------------------------------------------------------ one pass

GRADS = ("d_omega2", "d_gamma", "d_b", "d_c", "d_tau", "d_kappa", "d_q0", "d_qm1", "d_dir")


def run(state):
    kind = state["kind"]
    if kind == "features":
        return proposal.features(state["audio"])
    if kind == "mlp":
        net = state["net"]
        y = net.forward(state["x"])
        diff = y - state["target"]
        net.backward((2.0 / diff.numel()) * diff)
        return [y] + net.dw + net.db
    sim, steps, K = state["sim"], state["steps"], state["K"]
    if kind in ("block", "string"):
        r = sim.simulate(steps, want_state=True)
        return [r["audio"], r["q_end"], r["qm1_end"]]
    if kind == "linear":
        r = sim.simulate_linear(steps, want_state=True)
        return [r["audio"], r["q_end"], r["qm1_end"]]
    if kind == "plates_fit":
        audio = modal.simulate_autograd(sim, steps, K=K)
        leaves = (sim.omega2, sim.gamma, sim.b, sim.c, sim.tau, sim.kappa, sim.q0, sim.qm1,
                  sim.direction)
        return [audio.detach()] + list(torch.autograd.grad(audio, leaves, state["d_audio"]))
    if kind in ("strings_fit", "coupling_fit"):
        r = sim.simulate(steps, K=K)
        g = sim.grad(steps, state["d_audio"], K, r["ckpt"], want_dH=kind == "coupling_fit")
        out = [r["audio"]] + [g[k] for k in GRADS]
        return out + [g["d_H"]] if kind == "coupling_fit" else out
    return [sim.simulate(steps)["audio"]]


# ------------------------------------------------------------------ necessary work

def work(case):
    kind = case["kind"]
    if kind == "features":
        frames = 1 + case["T"] // 256
        return {"bytes": 4 * case["batch"] * (case["T"] + 1024),
                "flops": case["batch"] * frames * (2.5 * 1024 * 10 + 2 * 1024 + 4 * 513)}
    if kind == "mlp":
        mac = sum(a * b for a, b in zip(DIMS[:-1], DIMS[1:]))
        first = DIMS[0] * DIMS[1]
        B = case["batch"]
        return {"bytes": 2 * mac + 4 * mac + 2 * B * DIMS[0] + 12 * B * DIMS[-1],
                "flops": 2 * B * (3 * mac - first)}
    steps, inst = case["steps"], case.get("inst", 1)
    io = inst * steps * 8                        # excitation in, audio out
    if kind in ("block", "string"):
        return {"bytes": io + 80 * case["n"], "flops": 16 * case["n"] * steps}
    # expected sizes: log-uniform counts
    if "n_min" in case:
        lo, hi = case["n_min"], case["n_max"]
        span = math.log(hi / lo)
        n = (hi - lo) / span
        n3 = (hi ** 3 - lo ** 3) / (3 * span)
    if kind == "linear":
        return {"bytes": io + inst * n * 80, "flops": inst * n * steps * 6}
    if kind == "strings_fit":
        return {"bytes": io + inst * steps * 4 + inst * n * 200, "flops": inst * n * steps * 60}
    if kind in ("dataset", "groups"):
        plates = inst // 2
        entries = plates * n3 / 16               # nonzero class blocks of H: M N^2 / 4
        held = entries if kind == "dataset" else case["geoms"] * case["n_max"] ** 3 / 16
        return {"bytes": io + 4 * held + inst * n * 80,
                "flops": steps * (2 * entries + inst * n * 20)}
    N, M = case["n"], case["m"]
    dense = kind == "coupling_fit"
    entries = inst * M * N * N / (1 if dense else 4)
    if kind == "plate":
        return {"bytes": io + 4 * entries + N * 80, "flops": steps * (2 * entries + 4 * M * N)}
    # forward once, recomputed once, two more products in reverse, one for the direction / dH
    byts = io + 4 * inst * steps + (8 * entries if not dense else 12 * entries) + inst * N * 200
    return {"bytes": byts, "flops": steps * (2 * entries * 5 + inst * (12 * M * N + 60 * N))}


# ------------------------------------------------------------------ 64-bit values

def _pad(rows, width, dtype=np.float64):
    out = np.zeros((len(rows), width), dtype)
    for i, r in enumerate(rows):
        out[i, :len(r)] = r
    return torch.tensor(out, device="cuda:0", dtype=torch.float64)


class _Model:
    """The instances of a case in 64 bits, padded to one size."""

    def __init__(self, preps, steps, linear=False):
        self.preps, self.steps = preps, steps
        I = len(preps)
        self.N = [len(p["omega2"]) for p in preps]
        Nx = max(self.N)
        col = lambda k: _pad([np.asarray(p[k], np.float64) for p in preps], Nx)
        self.w2, self.gm, self.b, self.c = (col(k) for k in ("omega2", "gamma", "b", "c"))
        self.q0, self.qm1 = col("q0"), col("qm1")
        T = _pad([[p["dt"]] for p in preps], 1)
        self.T = T
        den = 1.0 + self.gm * T
        self.eps, self.r = 2.0 * self.gm * T / den, T * T / den
        self.rho = self.r * self.w2
        self.lam = _pad([np.asarray(p["lam"], np.float64) if p["kind"] == "tension" else []
                         for p in preps], Nx)
        self.tau = _pad([[float(p.get("tau", 0.0)) if p["kind"] == "tension" else 0.0]
                         for p in preps], 1)
        if linear:
            self.tau = torch.zeros_like(self.tau)
        exc = np.zeros((I, steps), np.float32)
        for i, p in enumerate(preps):
            exc[i, :min(steps, len(p["e"]))] = p["e"][:steps]
        self.exc = torch.tensor(exc, device="cuda:0", dtype=torch.float64).T.contiguous()
        self.plates = [i for i, p in enumerate(preps)
                       if not linear and p["kind"] == "plate" and p.get("H") is not None]
        self.strings = any(p["kind"] == "tension" for p in preps)
        self.H = self.dH = None
        if self.plates:
            self.M = [len(preps[i]["kappa"]) for i in self.plates]
            Mx = max(self.M)
            self.H = self._tensor("H", Mx, Nx)
            if all(preps[i].get("dH") is not None for i in self.plates):
                self.dH = self._tensor("dH", Mx, Nx)
            self.kap = _pad([np.asarray(preps[i]["kappa"], np.float64) for i in self.plates], Mx)
            self.pidx = torch.tensor(self.plates, device="cuda:0")
            self.all_plates = len(self.plates) == I

    def _tensor(self, key, Mx, Nx):
        H = torch.zeros(len(self.plates), Mx, Nx, Nx, device="cuda:0", dtype=torch.float64)
        for j, i in enumerate(self.plates):
            h = torch.tensor(self.preps[i][key], device="cuda:0")
            H[j, :h.shape[0], :h.shape[1], :h.shape[1]] = h.double()
        return H

    def rows(self, q):
        return q if self.all_plates else q[self.pidx]

    def mul(self, H, q):
        """H^k q of every plate and stress mode."""
        P, M, N, _ = H.shape
        return torch.bmm(H.view(P, M * N, N), q.unsqueeze(-1)).view(P, M, N)

    def force(self, q):
        """fnl(q) and the pieces that the adjoint reuses."""
        f, S, u, eta = None, None, None, None
        if self.strings:
            lq = self.lam * q
            S = (lq * q).sum(1, keepdim=True)
            f = self.tau * lq * S
        if self.H is not None:
            qp = self.rows(q)
            u = self.mul(self.H, qp)
            eta = torch.bmm(u, qp.unsqueeze(-1)).squeeze(-1)
            fp = torch.bmm((self.kap * eta).unsqueeze(1), u).squeeze(1)
            if self.all_plates:
                f = fp if f is None else f + fp
            else:
                f = torch.zeros_like(q) if f is None else f
                f = f.index_add(0, self.pidx, fp)
        return (torch.zeros_like(q) if f is None else f), S, u, eta

    def cat(self, x, sizes=None):
        sizes = self.N if sizes is None else sizes
        return torch.cat([x[i, :n] for i, n in enumerate(sizes)])

    def forward(self, keep=False):
        q, v = self.q0.clone(), self.q0 - self.qm1
        y = torch.empty(self.steps, len(self.preps), device="cuda:0", dtype=torch.float64)
        traj = []
        for n in range(self.steps):
            if keep:
                traj.append((q, v))
            f = self.force(q)[0]
            v = v - self.eps * v - self.rho * q + self.r * (self.b * self.exc[n].unsqueeze(1) - f)
            q = q + v
            y[n] = (self.c * q).sum(1)
        traj.append((q, v))
        return y.T.contiguous(), traj

    def adjoint(self, traj, ybar, want_dH=False):
        yb = torch.tensor(ybar, device="cuda:0", dtype=torch.float64).T.contiguous()
        z = torch.zeros_like(self.q0)
        A, V, F, E, C = (z.clone() for _ in range(5))
        dtau = torch.zeros(len(self.preps), device="cuda:0", dtype=torch.float64)
        dkap = torch.zeros_like(self.kap) if self.H is not None else None
        ddir = torch.zeros_like(dtau)
        G = torch.zeros_like(self.H) if want_dH else None
        a = self.c * yb[self.steps - 1].unsqueeze(1)
        mu = a.clone()
        for n in range(self.steps - 1, -1, -1):
            q, v = traj[n]
            w = self.r * a
            f, S, u, eta = self.force(q)
            e = self.exc[n].unsqueeze(1)
            Jw = torch.zeros_like(q)
            if self.strings:
                Pq = (self.lam * q * w).sum(1, keepdim=True)
                Jw = Jw + self.tau * self.lam * (S * w + 2.0 * q * Pq)
                dtau -= (S * Pq).squeeze(1)
            if self.H is not None:
                wp, qp = self.rows(w), self.rows(q)
                xi = torch.bmm(u, wp.unsqueeze(-1)).squeeze(-1)
                zz = self.mul(self.H, wp)
                Jp = (2.0 * torch.bmm((self.kap * xi).unsqueeze(1), u)
                      + torch.bmm((self.kap * eta).unsqueeze(1), zz)).squeeze(1)
                Jw = Jw + Jp if self.all_plates else Jw.index_add(0, self.pidx, Jp)
                dkap -= eta * xi
                if self.dH is not None:
                    d = self.mul(self.dH, qp)
                    qd = torch.bmm(d, qp.unsqueeze(-1)).squeeze(-1)
                    wd = torch.bmm(d, wp.unsqueeze(-1)).squeeze(-1)
                    ddir -= (self.kap * (xi * qd + eta * wd)).sum(1)
                if want_dH:
                    t = xi.unsqueeze(-1) * qp.unsqueeze(1) + eta.unsqueeze(-1) * wp.unsqueeze(1)
                    G += t.unsqueeze(-1) * qp.unsqueeze(1).unsqueeze(1)
            A += a * q
            V += a * v
            F += a * (self.b * e - f)
            E += a * e
            C += yb[n].unsqueeze(1) * traj[n + 1][0]
            pick = self.c * yb[n - 1].unsqueeze(1) if n >= 1 else 0.0
            mu = mu - self.eps * mu - self.rho * a - Jw + pick
            a = a + mu
        den = 1.0 + self.gm * self.T
        dw2 = -A * self.r
        dgm = (A * self.T ** 3 * self.w2 - V * 2.0 * self.T - F * self.T ** 3) / den ** 2
        dk = (self.cat(dkap, self.M) if dkap is not None
              else torch.zeros(0, device="cuda:0", dtype=torch.float64))
        out = [self.cat(dw2), self.cat(dgm), self.cat(self.r * E), self.cat(C), dtau, dk,
               self.cat(a), self.cat(-(1.0 - self.eps) * (a - mu)), ddir]
        if want_dH:
            G = -self.kap.unsqueeze(-1).unsqueeze(-1) * 0.5 * (G + G.transpose(-1, -2))
            out.append(torch.cat([G[j, :self.M[j], :self.N[i], :self.N[i]].reshape(-1)
                                  for j, i in enumerate(self.plates)]))
        return out


def _exact_features(x):
    """Log-mel features of [B, T] sounds: centred reflected frames of 1024
    samples every 256, periodic Hann window, 128 HTK triangles from 20 Hz."""
    n, hop, nm, S = 1024, 256, 128, 8
    mel = lambda f: 2595.0 * np.log10(1.0 + f / 700.0)
    pts = 700.0 * (10.0 ** (np.linspace(mel(20.0), mel(FS / 2), nm + 2) / 2595.0) - 1.0)
    f = np.linspace(0.0, FS / 2, n // 2 + 1)
    up = (f[None] - pts[:-2, None]) / (pts[1:-1] - pts[:-2])[:, None]
    dn = (pts[2:, None] - f[None]) / (pts[2:] - pts[1:-1])[:, None]
    Wm = torch.tensor(np.maximum(0.0, np.minimum(up, dn)), device="cuda:0")
    win = torch.hann_window(n, periodic=True, dtype=torch.float64, device="cuda:0")
    out = []
    for xb in torch.tensor(x, device="cuda:0").double().split(64):
        X = torch.stft(xb, n, hop, n, win, center=True, pad_mode="reflect", return_complex=True)
        L = torch.log(Wm @ (X.real ** 2 + X.imag ** 2) + 1e-6)
        F = L.shape[-1]
        seg = [L[..., s * F // S:(s + 1) * F // S].mean(-1) for s in range(S)]
        out.append(torch.stack(seg, -1).reshape(len(xb), -1))
    return torch.cat(out)


def _exact_mlp(case, seed):
    x, t = _mlp_data(case, seed)
    rng = np.random.default_rng(seed)
    ws = []
    for l in range(len(DIMS) - 1):
        bound = math.sqrt(6.0 / DIMS[l])
        w = rng.uniform(-bound, bound, size=(DIMS[l + 1], DIMS[l])).astype(np.float32)
        if l == len(DIMS) - 2:
            w *= 0.1
        ws.append(_dev(w).to(torch.bfloat16).double())
    acts = [_dev(x).to(torch.bfloat16).double()]
    for l, w in enumerate(ws):
        z = acts[-1] @ w.T
        acts.append(torch.relu(z) if l < len(ws) - 1 else z)
    dz = (2.0 / acts[-1].numel()) * (acts[-1] - _dev(t).double())
    dw, db = [], []
    for l in range(len(ws) - 1, -1, -1):
        dw.insert(0, dz.T @ acts[l])
        db.insert(0, dz.sum(0))
        if l:
            dz = (dz @ ws[l]) * (acts[l] > 0)
    return [acts[-1]] + dw + db


def exact(case, seed):
    kind = case["kind"]
    if kind == "features":
        return _exact_features(_sounds(case, seed))
    if kind == "mlp":
        return _exact_mlp(case, seed)
    preps = _instances(case, seed)
    m = _Model(preps, case["steps"], linear=kind == "linear")
    fit = kind in ("strings_fit", "plates_fit", "coupling_fit")
    y, traj = m.forward(keep=fit)
    if fit:
        return [y] + m.adjoint(traj, _d_audio(case, seed, len(preps)), kind == "coupling_fit")
    if kind in ("block", "string", "linear"):
        q, v = traj[-1]
        return [y, m.cat(q), m.cat(q - v)]
    return [y]
