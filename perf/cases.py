"""The work that users of this library have it do, as cases for timing and comparison.

Every case goes through the public entry points of ``paper_1810_12707_gb300.mhd``: runs of the
solver from given fields to given fields (the paper's flows and the ensembles and served batches
built on them), single right-hand sides, and the diagnostics of a state.  ``exact`` restates the
method with torch's FP64 FFTs, without this package.
"""
import math

import numpy as np
import torch

from paper_1810_12707_gb300 import mhd

PRECISIONS = {"fp64": mhd.MHD_FP64, "df": mhd.MHD_FP64_DF, "mixed": mhd.MHD_FP32_MIXED}
INTEGRATORS = {"ab2": mhd.MHD_AB2, "rk4": mhd.MHD_RK4, "pc": mhd.MHD_PC}
EVALS = {"ab2": 1, "rk4": 4, "pc": 2}  # right-hand sides per step
FORCE = (0.25, 1.0, 1.0, 1.0, 1)       # amplitude, A, B, C, k_f of the forced runs


def listed():
    return [
        # the call of a host framework that owns the device memory: one small right-hand side
        # without allocation, the smallest unit of work the library offers
        {"name": "noalloc32", "kind": "rhs_noalloc", "n": 32},
        # the paper's Orszag-Tang type run on the smallest usual grid: 100 fixed steps, bound by
        # launches and by latency
        {"name": "ot32_fp64", "kind": "run", "n": 32, "precision": "fp64", "integrator": "ab2", "ic": "ot",
         "batch": 1, "steps": 100, "dt": 1e-3, "tracers": 0, "forced": False},
        # a served batch: runs admitted to a pool, advanced together, polled, and retired to the host
        {"name": "pool32_mixed", "kind": "pool", "n": 32, "precision": "mixed", "runs": 13, "steps": 60, "k": 20},
        # one right-hand side of a broadband state, for analysis or an outer integrator
        {"name": "rhs64_fp64", "kind": "rhs", "n": 64, "precision": "fp64"},
        # the 64 x 64^3 parameter ensemble in mixed precision, one launch per kernel for all
        {"name": "ens64_mixed", "kind": "run", "n": 64, "precision": "mixed", "integrator": "ab2", "ic": "ot",
         "batch": 64, "steps": 40, "dt": 0.0, "tracers": 0, "forced": False},
        # a forced run with the fourth-order solver and tracer particles (energy exchange runs)
        {"name": "rk4_128_df", "kind": "run", "n": 128, "precision": "df", "integrator": "rk4", "ic": "abc",
         "batch": 1, "steps": 5, "dt": 0.0, "tracers": 100003, "forced": True},
        # the ABC dynamo at 256^3 in IEEE FP64, the default precision
        {"name": "abc256_fp64", "kind": "run", "n": 256, "precision": "fp64", "integrator": "ab2", "ic": "abc",
         "batch": 1, "steps": 30, "dt": 0.0, "tracers": 0, "forced": False},
        # the diagnostics and spectra that a run takes every few hundred steps
        {"name": "diag256_fp64", "kind": "diag", "n": 256, "precision": "fp64"},
        # fields from and to pinned host memory around every step (coupled codes, out-of-core use)
        {"name": "host256_df", "kind": "host", "n": 256, "precision": "df"},
        # the Taylor-Green runs at 512^3, the largest usual grid, in both reduced forms
        {"name": "tg512_mixed", "kind": "run", "n": 512, "precision": "mixed", "integrator": "ab2", "ic": "tg",
         "batch": 1, "steps": 20, "dt": 0.0, "tracers": 0, "forced": False},
        {"name": "tg512_df", "kind": "run", "n": 512, "precision": "df", "integrator": "ab2", "ic": "tg",
         "batch": 1, "steps": 20, "dt": 0.0, "tracers": 0, "forced": False},
    ]


def draw(rng):
    kind = rng.choices(["run", "rhs", "rhs_noalloc", "pool", "diag", "host"], [10, 2, 1, 2, 2, 1])[0]
    if kind == "rhs_noalloc":
        return {"kind": kind, "n": rng.choice([16, 32]), "cs": round(rng.uniform(2.0, 20.0), 3)}
    precision = rng.choice(["fp64", "df", "mixed"])
    if kind == "pool":
        n = rng.choice([32, 64])
        runs = rng.randint(1, 29 if n == 32 else 9)
        k = rng.choice([5, 10, 20])
        return {"kind": kind, "n": n, "precision": precision, "runs": runs, "steps": k * rng.randint(1, 4), "k": k}
    if kind in ("rhs", "diag", "host"):
        return {"kind": kind, "n": rng.choice([16, 32, 64, 128, 256]), "precision": precision,
                "cs": round(rng.uniform(2.0, 20.0), 3)}
    n = rng.choice([16, 32, 64, 128, 256, 512])
    integrator = "ab2" if n == 512 and precision == "fp64" else rng.choices(["ab2", "rk4", "pc"], [6, 2, 2])[0]
    most = {16: 200, 32: 32, 64: 16, 128: 5, 256: 2, 512: 1}[n]
    batch = max(1, min(most, int(round(math.exp(rng.uniform(0.0, math.log(most + 0.5)))))))
    most = {16: 100, 32: 100, 64: 60, 128: 40, 256: 24, 512: 4 if precision == "fp64" else 12}[n]
    steps = rng.randint(1, max(1, min(most if batch <= 8 else 25, most // EVALS[integrator])))
    tracers = rng.choice([0, 0, 0, int(10 ** rng.uniform(1.0, 5.5)) // batch])
    return {"kind": "run", "n": n, "precision": precision, "integrator": integrator,
            "ic": rng.choice(["ot", "abc", "tg"]), "batch": batch, "steps": steps,
            "dt": rng.choice([0.0, 0.0, 5e-4]), "tracers": tracers, "forced": rng.random() < 0.25}


# ---- inputs ----

def _grid(n):
    x = (2.0 * math.pi / n) * torch.arange(n, dtype=torch.float64, device="cuda")
    return x[None, None, :], x[None, :, None], x[:, None, None]


def _low_k(n, gen):
    """Seeded real solenoidal field of the modes 0 < |k|^2 <= 16, unit RMS (3, n, n, n)."""
    k = torch.arange(-4, 5, dtype=torch.float64)
    kz, ky, kx = torch.meshgrid(k, k, k, indexing="ij")
    kk = torch.stack([kx, ky, kz])
    k2 = (kk * kk).sum(0)
    a = torch.complex(torch.randn(3, 9, 9, 9, dtype=torch.float64, generator=gen),
                      torch.randn(3, 9, 9, 9, dtype=torch.float64, generator=gen))
    a = (a - kk * ((kk * a).sum(0) / k2.clamp(min=1.0))) * ((k2 > 0) & (k2 <= 16))
    x = (2.0 * math.pi / n) * torch.arange(n, dtype=torch.float64)
    e = torch.exp(1j * k[:, None] * x[None, :]).cuda()
    f = torch.empty(3, n, n, n, dtype=torch.float64, device="cuda")
    for c in range(3):
        t = torch.einsum("zyk,kx->zyx", a[c].cuda(), e)
        t = torch.einsum("zkx,ky->zyx", t, e)
        for z0 in range(0, n, 64):
            f[c, z0:z0 + 64] = torch.einsum("kyx,kz->zyx", t, e[:, z0:z0 + 64]).real
    return f / f.square().sum(0).mean().sqrt()


def _waves(n):
    k1 = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda")
    kr = torch.fft.rfftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda")
    return kr[None, None, :], k1[None, :, None], k1[:, None, None]


def _mask(n):
    kx, ky, kz = _waves(n)
    return (3 * kx.abs() < n) & (3 * ky.abs() < n) & (3 * kz.abs() < n)


def _broad(n, gen, comps):
    """Seeded real fields with a k^-11/6 amplitude on every mode of the 2/3 box, unit RMS, no mean."""
    kx, ky, kz = _waves(n)
    k2 = kx * kx + ky * ky + kz * kz
    amp = torch.where((k2 > 0) & _mask(n), k2.clamp(min=1.0) ** (-11.0 / 12.0), torch.zeros_like(k2))
    f = torch.randn(comps, n, n, n, dtype=torch.float64, generator=gen).cuda() if n <= 64 else torch.randn(
        comps, n, n, n, dtype=torch.float64, device="cuda",
        generator=torch.Generator("cuda").manual_seed(int(torch.randint(1 << 40, (1,), generator=gen))))
    for c in range(comps):
        f[c] = torch.fft.irfftn(torch.fft.rfftn(f[c]) * amp, s=(n, n, n))
    return f / f.square().sum(0).mean().sqrt()


def _flow(case, seed, inst=0):
    """(rho, u, B) of one instance and its (nu, eta, cs)."""
    n, ic = case["n"], case.get("ic", "broad")
    gen = torch.Generator().manual_seed(seed * 1000003 + inst * 7919 + 17)
    X, Y, Z = _grid(n)
    rho = torch.ones(n, n, n, dtype=torch.float64, device="cuda")
    zero = torch.zeros_like(rho)
    if ic == "ot":      # Orszag-Tang type, 1e-3 solenoidal perturbation
        u = torch.stack([zero - torch.sin(Y), zero + torch.sin(X), zero]) + 1e-3 * _low_k(n, gen)
        b = torch.stack([zero - torch.sin(Y), zero + torch.sin(2 * X), zero])
        phys = (1e-2, 1e-2, 10.0)
        if case.get("batch", 1) > 1:  # the ensemble's parameters: log-uniform nu, eta, uniform Mach
            r = torch.rand(3, dtype=torch.float64, generator=gen)
            phys = (10.0 ** (-3.0 + float(r[0])), 10.0 ** (-3.0 + float(r[1])), 1.0 / (0.05 + 0.45 * float(r[2])))
    elif ic == "abc":   # ABC dynamo with a weak random seed field
        u = torch.stack([zero + torch.sin(Z) + torch.cos(Y), zero + torch.sin(X) + torch.cos(Z),
                         zero + torch.sin(Y) + torch.cos(X)])
        b = math.sqrt(2e-5) * _low_k(n, gen)
        phys = (2e-3, 2e-3, 10.0)
    elif ic == "tg":    # Taylor-Green with a random seed field
        u = torch.stack([torch.sin(X) * torch.cos(Y) * torch.cos(Z), -torch.cos(X) * torch.sin(Y) * torch.cos(Z),
                         zero])
        b = math.sqrt(2e-3) * _low_k(n, gen)
        phys = (1e-3, 1e-3, 1.0 / 0.3)
    else:               # a developed state: broadband fields, density variations, a guide field; as a
        # snapshot of another code has it, B is solenoidal to a part in a thousand only
        rho = 1.0 + 0.1 * _broad(n, gen, 1)[0].clamp(-4.0, 4.0)
        u = _broad(n, gen, 3)
        b = 0.5 * _broad(n, gen, 3)
        kx, ky, kz = _waves(n)
        s = [torch.fft.rfftn(b[c]) for c in range(3)]
        k = (kx, ky, kz)
        div = sum(k[c] * s[c] for c in range(3)) / (kx * kx + ky * ky + kz * kz).clamp(min=1.0)
        for c in range(3):
            b[c] = torch.fft.irfftn(s[c] - (1.0 - 1e-3) * k[c] * div, s=(n, n, n)) + 0.1 * (c + 1)
        u += torch.tensor([0.05, -0.03, 0.02], dtype=torch.float64, device="cuda")[:, None, None, None]
        phys = (5e-3, 4e-3, 4.0)
    if "cs" in case:
        phys = (phys[0], phys[1], case["cs"])
    return (rho.contiguous(), u.contiguous(), b.contiguous()), phys


def _instances(case):
    return case["runs"] if case["kind"] == "pool" else case.get("batch", 1)


def _ic_case(case):
    """The case as the input recipe reads it: a pool's runs are Orszag-Tang or ABC flows."""
    return dict(case, ic="ot", batch=max(2, case["runs"])) if case["kind"] == "pool" else case


def _tracers(case, seed, inst):
    rng = np.random.default_rng([seed, inst, 3])
    return rng.uniform(0.0, 2.0 * math.pi, (case["tracers"], 3))


def prepare(case, seed):
    flows = [_flow(_ic_case(case), seed, i) for i in range(_instances(case))]
    fields, phys = [f for f, _ in flows], [p for _, p in flows]
    st = {"case": case, "fields": fields, "phys": phys}
    kind, n = case["kind"], case["n"]
    if kind == "rhs_noalloc":
        return st
    precision = PRECISIONS[case["precision"]]
    if kind == "pool":
        st["pool"] = mhd.mhd_pool_create(n, case["runs"], precision=precision)
        return st
    st["ctx"] = mhd.mhd_init(n, phys, dt=case.get("dt", 0.0), precision=precision,
                             integrator=INTEGRATORS[case.get("integrator", "ab2")])
    if kind == "run":
        if case["forced"]:
            for i in range(len(fields)):
                mhd.mhd_set_forcing(st["ctx"], i, *FORCE)
        st["pos"] = [_tracers(case, seed, i) for i in range(len(fields))] if case["tracers"] else []
    elif kind == "host":
        pin = [torch.empty(a.shape, dtype=torch.float64, pin_memory=True) for a in fields[0]]
        for p, a in zip(pin, fields[0]):
            p.copy_(a)
        out = [torch.empty(a.shape, dtype=torch.float64, pin_memory=True) for a in fields[0]]
        st["keep"], st["in"], st["out"] = (pin, out), [p.numpy() for p in pin], [o.numpy() for o in out]
        st["fields"] = fields = []
    else:
        mhd.mhd_set_state(st["ctx"], 0, *fields[0])
    return st


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "rhs_noalloc":
        return mhd.mhd_rhs_noalloc(case["n"], state["phys"][0], *state["fields"][0])
    if kind == "pool":
        pool = state["pool"]
        slots = [mhd.mhd_pool_admit(pool, ph, *f, nsteps=case["steps"]) for ph, f in zip(state["phys"], state["fields"])]
        done = None
        for _ in range(case["steps"] // case["k"]):
            mhd.mhd_pool_step(pool, case["k"])
            done = mhd.mhd_pool_progress(pool)
        out = [mhd.mhd_pool_retire(pool, s) for s in slots]
        return {"steps": done[0], "status": done[1], "fields": [np.stack([o[f] for o in out]) for f in range(3)]}
    ctx = state["ctx"]
    if kind == "rhs":
        return mhd.mhd_rhs(ctx, 0, device=True)
    if kind == "diag":
        return {"diag": mhd.mhd_diagnostics(ctx, 0), "spectra": mhd.mhd_spectra(ctx, 0)}
    if kind == "host":
        mhd.mhd_set_state(ctx, 0, *state["in"])
        mhd.mhd_step(ctx, 1)
        mhd.mhd_get_state_async(ctx, 0, *state["out"])
        mhd.mhd_synchronize(ctx)
        return list(state["out"])
    for i, f in enumerate(state["fields"]):
        mhd.mhd_set_state(ctx, i, *f)
    for i, p in enumerate(state["pos"]):
        mhd.mhd_tracers_set(ctx, i, p)
    mhd.mhd_step(ctx, case["steps"])
    got = [mhd.mhd_get_state(ctx, i, device=True) for i in range(len(state["fields"]))]
    out = {"fields": list(got[0]) if len(got) == 1 else [torch.stack([g[f] for g in got]) for f in range(3)]}
    if state["pos"]:
        tr = [mhd.mhd_tracers_get(ctx, i) for i in range(len(state["pos"]))]
        out["pos"], out["vel"] = np.concatenate([t[0] for t in tr]), np.concatenate([t[1] for t in tr])
    return out


def work(case):
    n, kind, inst = case["n"], case["kind"], _instances(case)
    n3 = float(n) ** 3
    fft = 2.5 * n3 * 3.0 * math.log2(n)  # one real 3D transform
    rhs = 19 * fft + 60 * n3             # 7 inverse, 12 forward, products and assembly
    io = 7 * 8 * n3
    if kind in ("run", "pool"):
        evals = case["steps"] * EVALS[case.get("integrator", "ab2")]
        tr = case.get("tracers", 0)
        return {"bytes": inst * (2 * io + tr * 9 * 8), "flops": inst * (evals * rhs + 14 * fft + tr * case["steps"] * 120)}
    if kind == "host":
        return {"bytes": 2 * io, "flops": rhs + 14 * fft}
    if kind == "rhs_noalloc":
        return {"bytes": 2 * io, "flops": rhs + 14 * fft}
    if kind == "rhs":  # the state's kept modes in, the fields out
        return {"bytes": io * 8.0 / 27.0 + io, "flops": rhs + 7 * fft}
    return {"bytes": io * 8.0 / 27.0, "flops": 7 * fft + 3 * fft + 2 * fft + 100 * n3}


# ---- the method in FP64 with torch's FFTs ----

class _Exact:
    """Pseudo-spectral RHS and solvers on the half-complex spectra of one instance."""

    def __init__(self, n, phys, force=None):
        self.n, (self.nu, self.eta, self.cs), self.force = n, phys, force
        self.k = _waves(n)
        self.k2 = self.k[0] ** 2 + self.k[1] ** 2 + self.k[2] ** 2
        self.keep = _mask(n)
        self.kmax = (n - 1) // 3

    def fwd(self, f):
        return torch.fft.rfftn(f, norm="forward") * self.keep

    def inv(self, s):
        return torch.fft.irfftn(s, s=(self.n,) * 3, norm="forward")

    def spectra(self, rho, u, b):
        return torch.stack([self.fwd(rho)] + [self.fwd(rho * u[c]) for c in range(3)] + [self.fwd(b[c]) for c in range(3)])

    def real(self, y):
        f = torch.stack([self.inv(y[q]) for q in range(7)])
        return [f[0], f[1:4], f[4:7]]

    def rhs(self, y):
        """RHS spectra, max |u| + c_f, and B on the grid."""
        k, i = self.k, 1j
        f = [self.inv(y[q]) for q in range(7)]
        u = [f[1 + c] / f[0] for c in range(3)]
        m, b = f[1:4], f[4:7]
        b2 = b[0] ** 2 + b[1] ** 2 + b[2] ** 2
        smax = float((torch.sqrt(u[0] ** 2 + u[1] ** 2 + u[2] ** 2) + torch.sqrt(self.cs ** 2 + b2 / f[0])).max())
        r = torch.empty_like(y)
        r[0] = -i * (k[0] * y[1] + k[1] * y[2] + k[2] * y[3])
        for a in range(3):
            r[1 + a] = -i * k[a] * self.cs ** 2 * y[0] - self.nu * self.k2 * self.fwd(u[a])
        for a in range(3):
            for c in range(a, 3):
                t = self.fwd(m[a] * u[c] - b[a] * b[c] + (0.5 * b2 if a == c else 0.0))
                r[1 + a] -= i * k[c] * t
                if c != a:
                    r[1 + c] -= i * k[a] * t
        if self.force:
            amp, A, B, C, q = self.force
            X, Y, Z = _grid(self.n)
            g = (A * torch.sin(q * Z) + C * torch.cos(q * Y), B * torch.sin(q * X) + A * torch.cos(q * Z),
                 C * torch.sin(q * Y) + B * torch.cos(q * X))
            for a in range(3):
                r[1 + a] += amp * self.fwd(f[0] * g[a])
        e = [self.fwd(u[(a + 1) % 3] * b[(a + 2) % 3] - u[(a + 2) % 3] * b[(a + 1) % 3]) for a in range(3)]
        for a in range(3):
            p, q = (a + 1) % 3, (a + 2) % 3
            r[4 + a] = i * (k[p] * e[q] - k[q] * e[p]) - self.eta * self.k2 * y[4 + a]
        return r, smax, b

    def dt(self, smax):
        d = 0.2 * (2.0 * math.pi / self.n) / smax
        diff = max(self.nu, self.eta)
        return min(d, 0.5 / (diff * self.kmax ** 2)) if diff > 0 else d

    def advance(self, y, steps, integrator, dt_fixed, tracers=None):
        old, dt_old = None, 0.0
        for _ in range(steps):
            f, smax, b = self.rhs(y)
            dt = dt_fixed if dt_fixed > 0 else self.dt(smax)
            w = 0.5 * dt / dt_old if old is not None else 0.0
            if integrator == "rk4":
                k2 = self.rhs(y + 0.5 * dt * f)[0]
                k3 = self.rhs(y + 0.5 * dt * k2)[0]
                k4 = self.rhs(y + dt * k3)[0]
                y = y + dt / 6.0 * (f + 2.0 * k2 + 2.0 * k3 + k4)
            else:
                p = y + dt * ((1.0 + w) * f - (w * old if old is not None else 0.0))
                y = p if integrator == "ab2" else y + 0.5 * dt * (f + self.rhs(p)[0])
            old, dt_old = f, dt
            if tracers is not None:
                self.push(tracers, b, dt)
        return y

    def corners(self, pos):
        n, h = self.n, 2.0 * math.pi / self.n
        g = pos / h
        i = torch.floor(g)
        l = g - i
        i = i.long() % n
        for c in range(8):
            s = [(c >> a) & 1 for a in range(3)]
            w = 1.0
            for a in range(3):
                w = w * (l[:, a] if s[a] else 1.0 - l[:, a])
            yield w, ((i[:, 2] + s[2]) % n * n + (i[:, 1] + s[1]) % n) * n + (i[:, 0] + s[0]) % n

    def gather(self, pos, fields):
        out = torch.zeros(len(pos), 3, dtype=torch.float64, device=pos.device)
        for w, at in self.corners(pos):
            for a in range(3):
                out[:, a] += w * fields[a].reshape(-1)[at]
        return out

    def push(self, tr, b, dt):
        t = self.gather(tr["pos"], b) * (0.5 * dt)
        s = 2.0 * t / (1.0 + t.square().sum(1, keepdim=True))
        v = tr["vel"]
        v = v + torch.linalg.cross(v + torch.linalg.cross(v, t), s)
        tr["vel"] = v
        tr["pos"] = torch.remainder(tr["pos"] + v * dt, 2.0 * math.pi)


def _exact_diag(x, rho, u, b):
    y = x.spectra(rho, u, b)
    f = x.real(y)
    r, m, bb = f[0], f[1], f[2]
    v = m / r
    u2, b2 = v.square().sum(0), bb.square().sum(0)
    w = torch.where(x.k[0] > 0, 2.0, 1.0) * torch.ones_like(x.k2)
    div = x.k[0] * y[4] + x.k[1] * y[5] + x.k[2] * y[6]
    d = {"ke": 0.5 * (r * u2).mean(), "me": 0.5 * b2.mean(), "eint": x.cs ** 2 * (r * torch.log(r)).mean(),
         "cross_hel": (v * bb).sum(0).mean(), "mean_speed": u2.sqrt().mean(), "mean_bmag": b2.sqrt().mean(),
         "smax": (u2.sqrt() + torch.sqrt(x.cs ** 2 + b2 / r)).max(), "mean_rho": r.mean(),
         "divb_rms": (w * div.abs().square()).sum().sqrt()}
    d = {q: float(t) for q, t in d.items()}
    d["mach_s"] = d["mean_speed"] / x.cs
    d["v_a"] = d["mean_bmag"] / math.sqrt(d["mean_rho"])
    d["mach_a"] = d["mean_speed"] / d["v_a"]
    d["etot"] = d["ke"] + d["me"] + d["eint"]
    d["mean_m"], d["mean_b"] = [float(t) for t in m.mean((1, 2, 3))], [float(t) for t in bb.mean((1, 2, 3))]
    uh, bh = torch.stack([x.fwd(v[c]) for c in range(3)]), y[4:7]
    shell = torch.floor(x.k2.sqrt() + 0.5).long()
    ns = int(math.floor(math.sqrt(3.0) * x.kmax + 0.5)) + 1

    def shells(s):
        e = (0.5 * w * s.abs().square().sum(0))[x.keep]
        return torch.zeros(ns, dtype=torch.float64, device=e.device).index_add_(0, shell[x.keep], e).cpu().numpy()

    def hel(s, over):
        k = x.k
        c = [1j * (k[1] * s[2] - k[2] * s[1]), 1j * (k[2] * s[0] - k[0] * s[2]), 1j * (k[0] * s[1] - k[1] * s[0])]
        return float((w * over * sum((s[a].conj() * c[a]).real for a in range(3))).sum())

    dx = x.inv(1j * x.k[0] * uh[0])
    d2, d3 = float(dx.square().mean()), float((dx ** 3).mean())
    theta = (w * (x.k[0] * uh[0] + x.k[1] * uh[1] + x.k[2] * uh[2]).abs().square()).sum().sqrt()
    one = torch.ones_like(x.k2)
    spec = {"ek": shells(uh), "em": shells(bh), "theta": float(theta), "s3": d3 / d2 ** 1.5, "d2": d2, "d3": d3,
            "kin_hel": hel(uh, one), "mag_hel": hel(bh, torch.where(x.k2 > 0, 1.0 / x.k2.clamp(min=1.0), 0.0 * one)),
            "divb_max": float(x.inv(1j * div).abs().max())}
    return {"diag": dict({"t": None, "dt": None, "step": None, "status": None}, **d), "spectra": spec}


def exact(case, seed):
    n, kind = case["n"], case["kind"]
    got, tracers = [], []
    for i in range(_instances(case)):
        (rho, u, b), phys = _flow(_ic_case(case), seed, i)
        x = _Exact(n, phys, FORCE if case.get("forced") else None)
        if kind == "diag":
            return _exact_diag(x, rho, u, b)
        y = x.spectra(rho, u, b)
        del rho, u, b
        if kind in ("rhs", "rhs_noalloc"):
            return tuple(x.real(x.rhs(y)[0]))
        tr = None
        if case.get("tracers"):
            tr = {"pos": torch.from_numpy(_tracers(case, seed, i)).cuda()}
            f = x.real(y)
            tr["vel"] = x.gather(tr["pos"], f[1] / f[0])
            tracers.append(tr)
        y = x.advance(y, case.get("steps", 1), case.get("integrator", "ab2"), case.get("dt", 0.0), tr)
        got.append([t if n > 128 else t.cpu() for t in x.real(y)])
    if kind == "host":
        return got[0]
    if kind == "pool":
        return {"steps": None, "status": None, "fields": [np.stack([g[f].numpy() for g in got]) for f in range(3)]}
    out = {"fields": got[0] if len(got) == 1 else [torch.stack([g[f] for g in got]) for f in range(3)]}
    if tracers:
        out["pos"] = torch.cat([t["pos"] for t in tracers]).cpu().numpy()
        out["vel"] = torch.cat([t["vel"] for t in tracers]).cpu().numpy()
    return out
