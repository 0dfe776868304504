"""The work that users of the library have it do, as measurable cases.

A case advances simulations of decaying isotropic turbulence (or an ensemble
of them) through the public entry points and reads out what such a program
keeps: E and eps at its logging cadence, the spectrum, and the field at the
end.  Every pass goes on from the state the last one left, as a run does.

Read-outs arrive as FP64 host arrays whatever the storage; a program keeps
them at the precision the simulation computes with, so an FP32 simulation's
fields, logs and spectra are kept in FP32, a 2-byte simulation's field in its
2-byte type (its logs in FP32), an FP64 simulation's in FP64.

The initial field is the solenoidal Gaussian field with
E(k) ~ k^4 exp(-2 k^2 / k0^2), at Ma = 0.1 and Re_lambda = 25, handed over as
a velocity field (kin_set_velocity), which serves odd boxes too; the
viscosity follows from the field.  What is read at the end is the velocity at
every cell, or, for the smallest boxes, every population (kin_get_f is the
checkpoint call: 19 doubles a cell).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1601_03815_gb300 as kin

MA, RE_LAMBDA = 0.1, 25.0
STORAGE = {"f32": kin.F32, "f16": kin.F16, "bf16": kin.BF16, "f64": kin.F64}
SCHEME = {"lbe": kin.LBE_MRT, "dugks": kin.DUGKS}
BYTES = {"f32": 4, "f16": 2, "bf16": 2, "f64": 8}
KEPT = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16, "f64": torch.float64}
LOGGED = {"f32": torch.float32, "f16": torch.float32, "bf16": torch.float32, "f64": torch.float64}
# arithmetic of one cell update: moments, relaxation and back-transform (LBE);
# pre-step, three face reconstructions, face equilibria and update (DUGKS)
FLOPS = {"lbe": 420.0, "dugks": 700.0}

# The reference ensemble's sizes (24 realisations) and a seeded scheme each.
ENSEMBLE = "32:8,64:8,96:6,128:2"


def listed():
    return [
        # a short served request on the smallest box: 500 steps in ticks of 50
        # (the server's chunk), E and eps at the end, the state handed back
        {"name": "lbe_f32_32_request", "kind": "request", "scheme": "lbe", "storage": "f32", "N": 32, "steps": 500,
         "every": 50, "read": "f"},
        # the same with DUGKS on the next box size the server takes
        {"name": "dugks_f32_48_request", "kind": "request", "scheme": "dugks", "storage": "f32", "N": 48,
         "steps": 500, "every": 50, "read": "u"},
        # E and eps of every step, logged without waiting (page-locked rows)
        {"name": "dugks_f32_64_log", "kind": "log", "scheme": "dugks", "storage": "f32", "N": 64, "steps": 200,
         "every": 1, "read": "u"},
        # an odd, ragged box (no spectrum: the FP32 transforms take even boxes)
        {"name": "dugks_f32_97_ragged", "kind": "history", "scheme": "dugks", "storage": "f32", "N": 97,
         "steps": 100, "every": 10, "read": "u"},
        # the 128^3 history: E, eps every 10 steps, E(k) every 200
        {"name": "dugks_f32_128_history", "kind": "history", "scheme": "dugks", "storage": "f32", "N": 128,
         "steps": 200, "every": 10, "read": "u"},
        # the headline boxes, 256^3 FP32, E and eps every 10 steps
        {"name": "lbe_f32_256", "kind": "history", "scheme": "lbe", "storage": "f32", "N": 256, "steps": 200,
         "every": 10, "read": "u"},
        {"name": "dugks_f32_256", "kind": "history", "scheme": "dugks", "storage": "f32", "N": 256, "steps": 100,
         "every": 10, "read": "u"},
        # the reduced-precision runs
        {"name": "lbe_f16_256", "kind": "history", "scheme": "lbe", "storage": "f16", "N": 256, "steps": 200,
         "every": 10, "read": "u"},
        {"name": "dugks_f16_256", "kind": "history", "scheme": "dugks", "storage": "f16", "N": 256, "steps": 100,
         "every": 10, "read": "u"},
        # the 32^3 FP64 run, E and eps logged each step
        {"name": "dugks_f64_32", "kind": "history", "scheme": "dugks", "storage": "f64", "N": 32, "steps": 100,
         "every": 1, "read": "f"},
        # the reference ensemble of 24 realisations, mixed sizes and schemes
        {"name": "ensemble_24", "kind": "ensemble", "sizes": ENSEMBLE, "storage": "f32", "steps": 100},
        # an analysis stop: a step with its spectrum, then the derived
        # statistics (Taylor scale, dissipation spectrum, skewness, flatness)
        {"name": "analysis_f32_256", "kind": "analysis", "scheme": "dugks", "storage": "f32", "N": 256, "steps": 1},
    ]


def draw(rng):
    kind = rng.choice(["request", "log", "history", "history", "history", "ensemble", "analysis"])
    if kind == "ensemble":
        sizes = ",".join("%d:%d" % (n, rng.randint(1, 3)) for n in sorted(rng.sample([24, 32, 48, 50, 64, 80, 96], 3)))
        return {"kind": kind, "sizes": sizes, "storage": "f32", "steps": rng.randint(40, 100)}
    scheme = rng.choice(["lbe", "dugks"])
    storage = "f32" if kind == "analysis" else rng.choice(["f32", "f32", "f32", "f16", "f64", "bf16"])
    top = {"request": 128, "log": 128, "history": 250, "analysis": 224}[kind]
    if storage == "f64":
        top = 64
    N = int(round(math.exp(rng.uniform(math.log(16), math.log(top)))))
    case = {"kind": kind, "scheme": scheme, "storage": storage, "N": N}
    if kind == "analysis":
        case.update(N=N - N % 2, steps=rng.randint(1, 3))
        return case
    every = {"request": 50, "log": 1, "history": rng.choice([5, 10])}[kind]
    if storage == "bf16":
        case.update(steps=20 if kind != "request" else 50, every=every)
    else:
        case.update(steps=every * max(1, rng.randint(40, 100) // every), every=every)
    case["read"] = "f" if N <= 40 else "u"
    return case


# --------------------------------------------------------------------- inputs
def _k0(N):
    return 2.0 if N < 32 else 4.0 if N <= 64 else 8.0


def _field(N, seed):
    """The initial velocity (3, N, N, N), FP64 on the GPU, and its viscosity."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(seed)
    kx = torch.fft.rfftfreq(N, 1.0 / N, device=dev, dtype=torch.float64)[None, None, :]
    ka = torch.fft.fftfreq(N, 1.0 / N, device=dev, dtype=torch.float64)
    ky, kz = ka[None, :, None], ka[:, None, None]
    k2 = kx * kx + ky * ky + kz * kz
    amp = torch.sqrt(k2) * torch.exp(-k2 / _k0(N) ** 2) * ((k2 >= 1.0) & (k2 < (N / 2) ** 2))
    uh = [torch.fft.rfftn(torch.randn((N, N, N), generator=gen, device=dev, dtype=torch.float64)) * amp
          for _ in range(3)]
    along = (kx * uh[0] + ky * uh[1] + kz * uh[2]) / k2.clamp(min=1.0)
    for c, k in enumerate((kx, ky, kz)):
        uh[c] = uh[c] - k * along
    u = torch.stack([torch.fft.irfftn(h, s=(N, N, N)) for h in uh])
    scale = MA / math.sqrt(float((u * u).sum(0).mean()))
    both = torch.where((kx > 0) & (2 * kx < N), 2.0, 1.0)  # a half-space mode and its conjugate
    omega = 0.5 * sum(float((both * k2 * h.abs().square()).sum()) for h in uh)
    omega *= (2.0 * math.pi / N) ** 2 * (scale / N ** 3) ** 2
    nu = MA * MA / 3.0 * math.sqrt(15.0 / (2.0 * omega)) / RE_LAMBDA
    return u * scale, nu


def _dt(scheme):
    return 1.0 if scheme == "lbe" else 0.5


def _sim(N, scheme, storage, seed):
    u, nu = _field(N, seed)
    sim = kin.Sim(N, SCHEME[scheme], nu, MA, _dt(scheme), STORAGE[storage])
    sim.set_velocity(u.cpu().numpy())
    return sim


def _members(case):
    """(N, scheme) of every ensemble member: sizes as given, schemes alternating
    within a size, so that both are there at every size with two members."""
    out = []
    for part in case["sizes"].split(","):
        n, count = (int(v) for v in part.split(":"))
        out += [(n, "lbe" if (k + len(out)) % 2 == 0 else "dugks") for k in range(count)]
    return out


def prepare(case, seed):
    if case["kind"] == "ensemble":
        sims = [_sim(n, scheme, case["storage"], 1000 * seed + m) for m, (n, scheme) in enumerate(_members(case))]
        return {"case": case, "sims": sims, "ens": kin.Ensemble(sims)}
    state = {"case": case, "sim": _sim(case["N"], case["scheme"], case["storage"], seed)}
    if case["kind"] == "log":
        state["rows"] = torch.zeros((case["steps"], 2), dtype=torch.float64, pin_memory=True).numpy()
    return state


# ----------------------------------------------------------------------- runs
def _read(sim, case):
    a = sim.get_f() if case.get("read") == "f" else sim.get_velocity()
    return torch.from_numpy(a).to(KEPT[case["storage"]])


def _log(rows, case):
    return torch.tensor(rows, dtype=torch.float64).to(LOGGED[case["storage"]])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "ensemble":
        state["ens"].step(case["steps"])
        return {"log": _log([s.stats() for s in state["sims"]], case), "field": [_read(s, case) for s in state["sims"]]}
    sim = state["sim"]
    if kind == "request":
        for _ in range(case["steps"] // case["every"]):
            sim.step(case["every"])
            sim.sync()
        return {"log": _log(sim.stats(), case), "field": _read(sim, case)}
    if kind == "log":
        rows = state["rows"]
        for k in range(case["steps"]):
            sim.step_stats_async(1, rows[k])
        sim.sync()
        return {"log": _log(rows, case), "field": _read(sim, case)}
    if kind == "history":
        rows = [sim.step_stats(case["every"]) for _ in range(case["steps"] // case["every"] - 1)]
        if case["N"] % 2:
            rows.append(sim.step_stats(case["every"]))
            return {"log": _log(rows, case), "field": _read(sim, case)}
        E, eps, Ek = sim.step_stats(case["every"], spectrum=True)
        return {"log": _log(rows + [(E, eps)], case), "spectrum": _log(Ek, case), "field": _read(sim, case)}
    # analysis
    E, eps, Ek = sim.step_stats(case["steps"], spectrum=True)
    d = sim.derived_stats()
    D = d.pop("D")
    return {"log": _log((E, eps), case), "spectrum": _log(Ek, case), "dissipation": _log(D, case),
            "scales": _log([d[k] for k in ("E", "uprime", "eps", "lambda", "Re_lambda", "eta", "F")], case),
            "field": _read(sim, case)}


def _cells(case):
    """(cells, scheme) of every simulation of the case."""
    return [(n ** 3, s) for n, s in _members(case)] if case["kind"] == "ensemble" else [(case["N"] ** 3, case["scheme"])]


def work(case):
    """Each step reads and writes every population once; the field and the
    statistics' velocity are read once per read-out."""
    b = BYTES[case["storage"]]
    byt = flo = 0.0
    for cells, scheme in _cells(case):
        byt += cells * (case["steps"] * 2 * 19 * b + (19 if case.get("read") == "f" else 3) * 8)
        flo += cells * case["steps"] * FLOPS[scheme]
    return {"bytes": byt, "flops": flo}


# ---------------------------------------------------- the same in 64 bits
_XI = np.array([(0, 0, 0)] + [v for p in ((1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1),
                                          (1, 0, -1), (0, 1, 1), (0, 1, -1)) for v in (p, tuple(-c for c in p))])
_W = np.array([1 / 3 if not any(v) else 1 / 18 if np.abs(v).sum() == 1 else 1 / 36 for v in _XI])


def _contract(m, f):
    return (m @ f.reshape(f.shape[0], -1)).reshape((m.shape[0],) + f.shape[1:])


class _Exact:
    """Both schemes on FP64 tensors f[19, z, y, x], written out from the paper's
    equations."""

    def __init__(self, scheme, nu, N):
        t = lambda a: torch.tensor(np.asarray(a, dtype=np.float64), device="cuda")  # noqa: E731
        self.scheme, self.nu, self.N = scheme, nu, N
        self.xi, self.w = t(_XI), t(_W)
        x, y, z = _XI.T.astype(np.float64)
        r = x * x + y * y + z * z
        M = np.stack([np.ones(19), 19 * r - 30, (21 * r * r - 53 * r + 24) / 2, x, (5 * r - 9) * x, y, (5 * r - 9) * y,
                      z, (5 * r - 9) * z, 3 * x * x - r, (3 * r - 5) * (3 * x * x - r), y * y - z * z,
                      (3 * r - 5) * (y * y - z * z), x * y, y * z, x * z, (y * y - z * z) * x, (z * z - x * x) * y,
                      (x * x - y * y) * z])
        s9 = 1.0 / (3.0 * nu + 0.5)
        S = [0, 1.19, 1.4, 0, 1.2, 0, 1.2, 0, 1.2, s9, 1.4, s9, 1.4, s9, s9, s9, 1.98, 1.98, 1.98]
        back = np.linalg.inv(M) @ np.diag(S)
        # equilibrium moments as a linear map of (rho, j) and of the six products j_a j_b
        lin, quad = np.zeros((19, 4)), np.zeros((19, 6))  # products: xx yy zz xy yz xz
        lin[1, 0], quad[1, :3] = -11, 19
        quad[2, :3] = -475 / 63
        for k in range(3):
            lin[4 + 2 * k, 1 + k] = -2 / 3
        quad[9, :3] = (2, -1, -1)
        quad[11, 1:3] = (1, -1)
        quad[13, 3] = quad[14, 4] = quad[15, 5] = 1
        cons = np.concatenate([np.ones((1, 19)), _XI.T])
        self.cons = t(cons)
        self.relax = t(np.eye(19) - back @ M + back @ lin @ cons)
        self.relax2 = t(back @ quad)
        self.roll = [tuple(int(c) for c in v[::-1]) for v in _XI]
        # equilibrium (Eq. 7) the same way: 3 W xi.u + W rho + W (9/2 (xi.u)^2 - 3/2 u^2)
        w = _W[:, None]
        self.eq1 = t(np.concatenate([w, 3 * w * _XI], axis=1))
        prod = np.stack([x * x, y * y, z * z, 2 * x * y, 2 * y * z, 2 * x * z], axis=1)
        self.eq2 = t(w * (4.5 * prod - 1.5 * np.array([1, 1, 1, 0, 0, 0])))

    @staticmethod
    def _products(m):
        j = m[1:]
        return torch.stack([j[0] * j[0], j[1] * j[1], j[2] * j[2], j[0] * j[1], j[1] * j[2], j[0] * j[2]])

    def equilibrium(self, m):
        return _contract(self.eq1, m).add_(_contract(self.eq2, self._products(m)))

    def start(self, u):
        return self.equilibrium(torch.cat([torch.zeros_like(u[:1]), u]))

    def step(self, f):
        if self.scheme == "lbe":
            g = _contract(self.relax, f).add_(_contract(self.relax2, self._products(_contract(self.cons, f))))
            return torch.stack([torch.roll(g[i], self.roll[i], (0, 1, 2)) for i in range(19)])
        tau, dt = 3.0 * self.nu, 0.5
        h = dt / 2
        b = 3 * h / (2 * tau + dt)
        X = torch.lerp(f, self.equilibrium(_contract(self.cons, f)), b)
        new = (4.0 / 3.0) * X - f / 3.0
        c2 = h / (2 * tau + h)
        # dims of f[1:]: z, y, x = 1, 2, 3 for axes z, y, x
        slope = [torch.roll(X, -1, 3 - a).sub_(torch.roll(X, 1, 3 - a)).mul_(0.5) for a in range(3)]
        for a in range(3):
            d = 3 - a
            face = torch.roll(X, -1, d).sub_(X).mul_(self._col(-h, a)).add_(X)
            face.add_(torch.roll(X, -1, d).sub_(X).mul_(0.5))
            for c in range(3):
                if c != a:
                    both = (slope[c] + torch.roll(slope[c], -1, d)).mul_(0.5)
                    face.addcmul_(both, self._col(-h, c).expand_as(both))
                    del both
            face = torch.lerp(face, self.equilibrium(_contract(self.cons, face)), c2)
            new.addcmul_(face - torch.roll(face, 1, d), self._col(-dt, a).expand_as(face))
        return new

    def _col(self, s, a):
        return (s * self.xi[:, a]).reshape(19, 1, 1, 1)

    def velocity(self, f):
        return _contract(self.cons, f)[1:]

    def stats(self, f):
        u = self.velocity(f)
        g = [(torch.roll(u, -1, 3 - a) - torch.roll(u, 1, 3 - a)) * 0.5 for a in range(3)]
        ss = sum(((g[a][b] + g[b][a]) * 0.5).square().mean() for a in range(3) for b in range(3))
        return float(0.5 * u.square().sum(0).mean()), float(2.0 * self.nu * ss)

    def _modes(self, f):
        N = self.N
        ka = torch.fft.fftfreq(N, 1.0 / N, device="cuda", dtype=torch.float64)
        kx = torch.arange(N // 2 + 1, device="cuda", dtype=torch.float64)[None, None, :]
        ks = (kx, ka[None, :, None], ka[:, None, None])
        n2 = kx * kx + ka[None, :, None] ** 2 + ka[:, None, None] ** 2
        uh = torch.fft.rfftn(self.velocity(f), dim=(1, 2, 3)) / N ** 3
        both = torch.where((kx > 0) & (2 * kx < N), 2.0, 1.0)
        return ks, n2, uh, 0.5 * both * uh.abs().square().sum(0)

    def _shells(self, n2, e):
        top = 1 + int(math.floor(math.sqrt(3.0 * (self.N // 2) ** 2) + 0.5))
        sh = torch.floor(torch.sqrt(n2) + 0.5).long().reshape(-1)
        return torch.bincount(sh, weights=e.reshape(-1), minlength=top)[:top]

    def spectrum(self, f):
        _, n2, _, e = self._modes(f)
        return self._shells(n2, e)

    def derived(self, f):
        N, nu = self.N, self.nu
        ks, n2, uh, e = self._modes(f)
        k1 = 2.0 * math.pi / N
        D = 2.0 * nu * k1 * k1 * self._shells(n2, e * n2)
        E, eps = 0.5 * float(self.velocity(f).square().sum(0).mean()), float(D.sum())
        m2 = m4 = 0.0
        for a in range(3):
            k = torch.where(ks[a].abs() * 2 == N, 0.0, ks[a]) * k1
            g = torch.fft.irfftn(1j * k * uh[a], s=(N, N, N)) * float(N) ** 3
            m2 += float(g.square().mean()) ** 2
            m4 += float(g.square().square().mean())
        up = math.sqrt(2.0 * E / 3.0)
        lam = math.sqrt(15.0 * nu / eps) * up
        return [E, up, eps, lam, up * lam / nu, (nu ** 3 / eps) ** 0.25, m4 / m2], D


def _exact_one(case, N, scheme, seed):
    u, nu = _field(N, seed)
    x = _Exact(scheme, nu, N)
    f = x.start(u)
    steps, every, kind = case["steps"], case.get("every", 0), case["kind"]
    rows = []
    for k in range(1, steps + 1):
        f = x.step(f)
        if kind in ("log", "history") and k % every == 0 or k == steps:
            rows.append(x.stats(f))
    field = f if case.get("read") == "f" else x.velocity(f)
    return x, f, torch.tensor(rows, dtype=torch.float64), field


def exact(case, seed):
    if case["kind"] == "ensemble":
        got = [_exact_one(case, n, s, 1000 * seed + m) for m, (n, s) in enumerate(_members(case))]
        return {"log": torch.cat([g[2] for g in got]), "field": [g[3] for g in got]}
    x, f, rows, field = _exact_one(case, case["N"], case["scheme"], seed)
    if case["kind"] == "request":
        return {"log": rows[0], "field": field}
    if case["kind"] == "log" or (case["kind"] == "history" and case["N"] % 2):
        return {"log": rows, "field": field}
    if case["kind"] == "history":
        return {"log": rows, "spectrum": x.spectrum(f), "field": field}
    scales, D = x.derived(f)
    return {"log": rows[0], "spectrum": x.spectrum(f), "dissipation": D,
            "scales": torch.tensor(scales, dtype=torch.float64), "field": field}
