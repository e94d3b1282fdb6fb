"""The solver's workloads that its speed is judged by, through the public Python API.

Every case starts from a state a user's program would hold: a developed,
solenoidal velocity field with a scalar that is partly correlated with u2 (as a
mean gradient makes it), drawn on the GPU from the seed alone.  ``exact`` is the
same work in 64 bits with torch's FFTs, written from the method's equations.
"""
import math

import numpy as np
import torch

import paper_2012_04838_gb300 as psc
from paper_2012_04838_gb300.serve import nu_for_resolution

DEV = "cuda:0"
SIZES = (8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 512, 520, 1024)
ENSEMBLE_SIZES = (32, 48, 64, 96, 128)


def _box(name, N, precision="fp32", steps=1, record=False, **kw):
    """Time steps of one box (CFL 0.5, a dt reset every 10 steps), and a
    statistics record after them where `record`."""
    case = dict(name=name, kind="step", N=N, precision=precision, steps=steps, record=record, dealias="two_thirds",
                form="rotational", integrator="ifrk4", forcing="const_power", cfl=0.5)
    case.update(kw)
    return case


def listed():
    return [
        # one record interval of the small Taylor-Green-sized FP64 run (32^3, dt = 0.005, records every 10 steps):
        # the smallest calls a user makes, where launches and latency are everything
        _box("record_interval_32_fp64", 32, "fp64", steps=10, record=True, cfl=0.0),
        # one record interval of a 64^3 box on its own, the commonest request of the served stream
        _box("record_interval_64", 64, steps=10, record=True),
        # the largest box of the ensemble on its own; kx rows of odd length (43)
        _box("record_interval_128", 128, steps=10, record=True),
        # one record interval of the 256^3 forced run in FP32-mixed ...
        _box("record_interval_256", 256, steps=10, record=True),
        # ... and a step of the same run in FP64, run side by side with it
        _box("step_256_fp64", 256, "fp64"),
        # the nonlinear term as the paper writes it, at the same grid
        _box("steps_256_convective", 256, steps=2, form="convective"),
        # a step of the 512^3 companion run (kx rows of odd length, 171)
        _box("step_512", 512),
        # a step of the full-size 1024^3 run, the headline
        _box("step_1024", 1024),
        # a step of the paper's own example: 520^3, phase-shift dealiasing on the sphere, plain RK4, band energy held
        _box("paper_step_520", 520, dealias="phase_shift", integrator="rk4", forcing="hold", cfl=0.0),
        # what a long run takes between steps: a full record with spectra, and the pressure field for output
        dict(name="diagnostics_512", kind="diagnostics", N=512, precision="fp32", pressure=True),
        # three quarters of the 84-box ensemble (64 x 64^3 + 16 x 96^3 + 4 x 128^3), ten steps of every box by graph
        dict(name="ensemble_graph", kind="ensemble", mode="graph", steps=10, n32=0, n48=0, n64=48, n96=12, n128=3),
        # the same boxes by one persistent launch per RK stage
        dict(name="ensemble_persistent", kind="ensemble", mode="persistent", steps=10, n32=0, n48=0, n64=48, n96=12,
             n128=3),
    ]


def draw(rng):
    """One more case of the same ranges: every grid size, both precisions, both
    dealiasings and forms, every forcing and integrator; no more work than the
    1024^3 step."""
    what = rng.choice(["step"] * 6 + ["diagnostics", "ensemble"])
    if what == "ensemble":
        n = {N: rng.randint(0, m) for N, m in ((32, 16), (48, 12), (64, 24), (96, 8), (128, 3))}
        n[64] = max(n[64], 1)
        return dict(kind="ensemble", mode=rng.choice(["graph", "persistent"]), steps=rng.randint(1, 10),
                    **{"n%d" % N: n[N] for N in ENSEMBLE_SIZES})
    N = rng.choice(SIZES)
    precision = rng.choice(["fp32", "fp32", "fp64"]) if N <= 256 else "fp32"
    if what == "diagnostics":
        return dict(kind="diagnostics", N=N, precision=precision, pressure=rng.random() < 0.7)
    dealias = "phase_shift" if N <= 520 and rng.random() < 0.25 else "two_thirds"
    form = "convective" if N <= 512 and rng.random() < 0.2 else "rotational"
    steps = rng.randint(1, 10) if N <= 128 else rng.randint(1, 2) if N <= 256 and precision == "fp32" else 1
    forcing = rng.choice(["const_power", "const_power", "hold", "none"])
    case = _box("", N, precision, steps=steps, record=N <= 256 and rng.random() < 0.5, dealias=dealias, form=form,
                integrator=rng.choice(["ifrk4", "ifrk4", "rk4"]), forcing=forcing,
                cfl=0.0 if forcing == "none" else rng.choice([0.5, 0.5, 0.0]))  # a decaying flow has no CFL limit
    del case["name"]
    return case


# ---------------------------------------------------------------- inputs


def _params(case, member=0):
    N = case["N"]
    paper = N == 520  # the paper's Table 2
    nu = 8e-4 if paper else 0.02 if N <= 32 else nu_for_resolution(N, 1.5)
    opt = dict(dealias=case.get("dealias", "two_thirds"), form=case.get("form", "rotational"),
               integrator=case.get("integrator", "ifrk4"), forcing=case.get("forcing", "const_power"))
    return psc.Params(
        N=N, precision=psc.FP64 if case["precision"] == "fp64" else psc.FP32_MIXED, nu=nu,
        Sc=(1.0, 0.7, 2.0)[member % 3], beta=1.0, kF=2.0, eps_inj=0.1, dt=5e-4 if paper else 0.16 / max(N, 32),
        cfl=case.get("cfl", 0.5), record_every=10,
        dealias=dict(two_thirds=psc.DEALIAS_TWO_THIRDS, phase_shift=psc.DEALIAS_PHASE_SHIFT)[opt["dealias"]],
        nonlinear_form=dict(rotational=psc.NL_ROTATIONAL, convective=psc.NL_CONVECTIVE)[opt["form"]],
        integrator=dict(ifrk4=psc.INTEG_IFRK4, rk4=psc.INTEG_RK4)[opt["integrator"]],
        forcing=dict(none=psc.FORCE_NONE, const_power=psc.FORCE_CONST_POWER, hold=psc.FORCE_HOLD_ENERGY)[opt["forcing"]])


def _wavenumbers(K, dtype):
    k = torch.arange(-K, K + 1, device=DEV, dtype=dtype)
    return k[:, None, None], k[None, :, None], torch.arange(0, K + 1, device=DEV, dtype=dtype)[None, None, :]


def _state(p, seed):
    """The compact state [4][2K+1][2K+1][K+1] of a developed flow: random phases,
    E(k) rising as k^4, falling as k^(-5/3) and rolling off at the dissipative
    end, u solenoidal with u_rms = 1, phi half carried by u2; conjugate-symmetric
    on kx = 0, zero at k = 0 and outside the retained set."""
    N, K = p.N, psc.compact_shape(p.N, p.dealias)[3] - 1
    sphere = p.dealias == psc.DEALIAS_PHASE_SHIFT
    real = torch.float64 if p.precision == psc.FP64 else torch.float32
    g = torch.Generator(device=DEV).manual_seed(seed)
    kz, ky, kx = _wavenumbers(K, real)
    k2 = kx * kx + ky * ky + kz * kz
    k2s = k2.clamp(min=1)
    k = k2s.sqrt()
    env = (k / 2.5) ** 2 / (1 + (k / 2.5) ** 2) ** (17 / 12) * torch.exp(-6.75 / N * k) / k
    env[K, K, 0] = 0
    if sphere:
        env *= 9 * k2 < 2 * N * N
    a = torch.empty((4, *env.shape), dtype=torch.complex128 if real == torch.float64 else torch.complex64, device=DEV)
    for f in range(4):
        v = torch.view_as_complex(torch.randn((*env.shape, 2), generator=g, device=DEV, dtype=real))
        plane = v[:, :, 0].clone()
        v[:, :, 0] = (plane + plane.flip(0, 1).conj()) * math.sqrt(0.5)
        torch.mul(v, env, out=a[f])
    dot = (a[0] * kx + a[1] * ky + a[2] * kz) / k2s
    a[0] -= dot * kx
    a[1] -= dot * ky
    a[2] -= dot * kz
    del dot, k2, k2s, k
    norm = 0.0
    for f in range(3):
        m = torch.view_as_real(a[f]).square().sum(-1)
        norm += 2 * float(m[:, :, 1:].sum(dtype=torch.float64)) + float(m[:, :, 0].sum(dtype=torch.float64))
    a *= math.sqrt(3.0 / norm) * float(N) ** 3
    a[3] = 0.6 * a[3] - 0.5 * a[1]
    return a


def _members(case):
    i = 0
    for N in ENSEMBLE_SIZES:
        for _ in range(case["n%d" % N]):
            yield i, _params(dict(N=N, precision="fp32"), member=i)
            i += 1


def prepare(case, seed):
    """The simulation (or batch) a user's program keeps, holding its state."""
    if case["kind"] == "ensemble":
        sims = []
        for i, p in _members(case):
            sim = psc.Simulation(p, device=DEV, stream=torch.cuda.Stream(DEV))
            sim.set_state(_state(p, 1000 * seed + i))
            sims.append(sim)
        if case["mode"] == "graph":
            batch = psc.Batch(sims)
        else:
            batch = psc.PersistentBatch(sims, max_boxes=128, max_N=128, device=DEV)
        return dict(case=case, sims=sims, batch=batch)
    p = _params(case)
    sim = psc.Simulation(p, device=DEV)
    sim.set_state(_state(p, seed))
    return dict(case=case, sim=sim)


def _record(sim, precision):
    """A statistics record with its spectra.  The numbers of an FP32-mixed run
    are kept as FP32, the accuracy they are computed and documented with; the
    skewnesses (near zero for some fields) stand beside the flatnesses."""
    rec, E, Ephi = sim.stats()
    return _layout(rec, E, Ephi, precision)


def _layout(rec, E, Ephi, precision):
    real = np.float64 if precision == "fp64" else np.float32
    shape = np.array(rec["skew"] + rec["flat"] + rec["skew_phi"] + rec["flat_phi"], dtype=real)
    out = {k: real(v) for k, v in rec.items() if k not in ("skew", "flat", "skew_phi", "flat_phi", "step")}
    return dict(scalars=out, step=rec["step"], moments=shape, E=np.asarray(E, dtype=real),
                Ephi=np.asarray(Ephi, dtype=real))


def run(state):
    case = state["case"]
    if case["kind"] == "ensemble":
        state["batch"].step(case["steps"])
        state["batch"].synchronize()
        return [sim.get_state() for sim in state["sims"]]
    sim = state["sim"]
    if case["kind"] == "diagnostics":
        out = dict(record=_record(sim, case["precision"]))
        if case["pressure"]:
            out["pressure"] = sim.pressure()
        return out
    sim.step(case["steps"])
    out = dict(state=sim.get_state())
    if case["record"]:
        out["record"] = _record(sim, case["precision"])
    return out


def work(case):
    """Each state read once and written once (a record reads it, the pressure is
    one field); flops: the transforms of the right-hand sides at 2.5 N^3 log2 N^3
    per real 3D transform."""

    def of(p, steps, transforms):
        shape = psc.compact_shape(p.N, p.dealias)
        state = math.prod(shape) * (16 if p.precision == psc.FP64 else 8)
        return state, steps * transforms * 2.5 * p.N ** 3 * 3 * math.log2(p.N)

    b = f = 0.0
    if case["kind"] == "ensemble":
        for _, p in _members(case):
            s, fl = of(p, case["steps"], 4 * 13)
            b, f = b + 2 * s, f + fl
    elif case["kind"] == "diagnostics":
        b, f = of(_params(case), 1, 13 + (10 if case["pressure"] else 0))
        b *= 1.25 if case["pressure"] else 1.0
    else:
        p = _params(case)
        per_rhs = (16 if case["form"] == "convective" else 13) * (2 if case["dealias"] == "phase_shift" else 1)
        s, f = of(p, case["steps"], 4 * per_rhs)
        b = (3 if case["record"] else 2) * s
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------- the same in 64 bits


class _Exact:
    """The method in complex128 with torch.fft, one field at a time."""

    def __init__(self, p):
        self.p, self.N = p, p.N
        self.K = psc.compact_shape(p.N, p.dealias)[3] - 1
        self.sphere = p.dealias == psc.DEALIAS_PHASE_SHIFT
        K = self.K
        self.k = _wavenumbers(K, torch.float64)[::-1]  # kx, ky, kz
        self.k2 = sum(q * q for q in self.k)
        self.inside = 9 * self.k2 < 2 * p.N ** 2 if self.sphere else None
        self.band = (self.k2 > 0) & (self.k2 <= p.kF ** 2)
        self.weight = torch.full((K + 1,), 2.0, device=DEV, dtype=torch.float64)
        self.weight[0] = 1.0
        self.at = torch.arange(-K, K + 1, device=DEV) % p.N
        self.D = p.nu / p.Sc
        self.dx = 2 * math.pi / p.N

    def phase(self, sign):
        return torch.exp(1j * sign * math.pi / self.N * (self.k[0] + self.k[1] + self.k[2]))

    def grid(self, c, shift=None):
        full = torch.zeros((self.N, self.N, self.N // 2 + 1), dtype=torch.complex128, device=DEV)
        full[self.at[:, None], self.at[None, :], : self.K + 1] = c if shift is None else c * shift
        return torch.fft.irfftn(full, s=(self.N,) * 3)

    def modes(self, x, shift=None):
        c = torch.fft.rfftn(x)[self.at[:, None], self.at[None, :], : self.K + 1]
        return c if shift is None else c * shift

    def curl(self, a, i):
        j, l = (i + 1) % 3, (i + 2) % 3
        return 1j * (self.k[j] * a[l] - self.k[l] * a[j])

    def products(self, a, shifted):
        """(nonlinear term, u . grad phi) in spectral space on one grid."""
        up, down = (self.phase(1), self.phase(-1)) if shifted else (None, None)
        u = [self.grid(a[i], up) for i in range(3)]
        umax = float((u[0].abs() + u[1].abs() + u[2].abs()).max())
        out = []
        if self.p.nonlinear_form == psc.NL_CONVECTIVE:
            for i in range(3):
                out.append(-self.modes(sum(u[j] * self.grid(1j * self.k[j] * a[i], up) for j in range(3)), down))
        else:
            w = [self.grid(self.curl(a, i), up) for i in range(3)]
            for i in range(3):
                j, l = (i + 1) % 3, (i + 2) % 3
                out.append(self.modes(u[j] * w[l] - u[l] * w[j], down))
            del w
        out.append(self.modes(sum(u[j] * self.grid(1j * self.k[j] * a[3], up) for j in range(3)), down))
        return out, umax

    def band_energy(self, a):
        e = sum((torch.where(self.band, a[i].abs() ** 2, 0.0) * self.weight).sum() for i in range(3))
        return float(e) / (2 * float(self.N) ** 6)

    def rhs(self, a, force=True):
        q, umax = self.products(a, False)
        if self.sphere:
            q = [0.5 * (x + y) for x, y in zip(q, self.products(a, True)[0])]
        r = torch.empty_like(a)
        dot = (self.k[0] * q[0] + self.k[1] * q[1] + self.k[2] * q[2]) / self.k2.clamp(min=1)
        for i in range(3):
            r[i] = q[i] - self.k[i] * dot
            r[i][self.K, self.K, 0] = 0
        if self.p.forcing == psc.FORCE_CONST_POWER:
            e = self.band_energy(a)
            A = self.p.eps_inj / (2 * e) if e > 1e-300 else 0.0
            for i in range(3):
                r[i] += torch.where(self.band, A * a[i], 0.0)
        r[3] = -q[3] - self.p.beta * a[1]
        if self.sphere:
            r *= self.inside
        if self.p.integrator == psc.INTEG_RK4:
            for i in range(4):
                r[i] -= (self.D if i == 3 else self.p.nu) * self.k2 * a[i]
        return r, umax

    def steps(self, u, n):
        p, dt = self.p, self.p.dt
        t, held, A = 0.0, None, 0.0
        for step in range(n):
            e0 = self.band_energy(u)
            r, umax = self.rhs(u)
            if p.cfl > 0 and step % p.record_every == 0 and umax > 0:
                dt = p.cfl * self.dx / umax
            ex = torch.ones((4, *self.k2.shape), dtype=torch.float64, device=DEV)
            if p.integrator == psc.INTEG_IFRK4:
                for i in range(4):
                    ex[i] = torch.exp(-(self.D if i == 3 else p.nu) * self.k2 * dt / 2)
            v = ex * (u + 0.5 * dt * r)
            acc = ex * ex * (u + dt / 6 * r)
            r, _ = self.rhs(v)
            v = ex * u + 0.5 * dt * r
            acc += dt / 3 * ex * r
            r, _ = self.rhs(v)
            v = ex * ex * u + dt * ex * r
            acc += dt / 3 * ex * r
            r, _ = self.rhs(v)
            self.last_stage = v
            u = acc + dt / 6 * r
            t += dt
            if p.forcing == psc.FORCE_HOLD_ENERGY:
                held = e0 if held is None else held
                e = self.band_energy(u)
                f = math.sqrt(held / e) if e > 1e-300 else 1.0
                u[:3] = torch.where(self.band, f * u[:3], u[:3])
                A = math.log(f) / dt
        return u, t, dt, n, A

    def record(self, u, t, dt, step, A):
        p, N = self.p, self.N
        n3 = float(N) ** 3
        k = self.k
        x = [self.grid(u[i]) for i in range(4)]
        umax = float((x[0].abs() + x[1].abs() + x[2].abs()).max())
        mean = lambda v: float(v.mean())  # noqa: E731
        r = dict(K_phys=0.5 * sum(mean(x[i] ** 2) for i in range(3)), phi_var=mean(x[3] ** 2),
                 phi_prod_phys=-2 * p.beta * mean(x[3] * x[1]))
        del x
        r["eps_phys"] = p.nu * sum(mean(self.grid(self.curl(u, i)) ** 2) for i in range(3))
        chi = 0.0
        for f, s, fl in ((None, "skew", "flat"), (3, "skew_phi", "flat_phi")):
            r[s], r[fl] = [], []
            for i in range(3):
                d = self.grid(1j * k[i] * u[i if f is None else f])
                m2, m3, m4 = mean(d ** 2), mean(d ** 3), mean(d ** 4)
                r[s].append(m3 / m2 ** 1.5 if m2 > 0 else 0.0)
                r[fl].append(m4 / m2 ** 2 if m2 > 0 else 0.0)
                chi += m2 if f == 3 else 0.0
        r["chi_phys"] = 2 * self.D * chi
        e = sum(u[i].abs() ** 2 for i in range(3)) * self.weight / (2 * n3 * n3)
        ep = u[3].abs() ** 2 * self.weight / (2 * n3 * n3)
        shell = torch.floor(self.k2.sqrt() + 0.5).long()
        hw = next(q for q in range(N, 0, -1) if 9 * q * q < 2 * N * N)
        ns = hw + 2 if self.sphere else int(math.floor(math.sqrt(3 * self.K ** 2) + 0.5)) + 1
        sums = lambda v: torch.bincount(shell.reshape(-1), weights=v.reshape(-1), minlength=ns)[:ns].cpu().numpy()  # noqa: E731
        E, Ephi = sums(e), sums(ep)
        r["K"] = float(e.sum())
        r["eps"] = 2 * p.nu * float((self.k2 * e).sum())
        r["chi"] = 4 * self.D * float((self.k2 * ep).sum())
        r["phi_prod"] = -2 * p.beta * float(((u[3].conj() * u[1]).real * self.weight).sum()) / (n3 * n3)
        if p.cfl > 0 and step % p.record_every == 0 and umax > 0:
            dt = p.cfl * self.dx / umax
        r.update(t=t, dt=dt, step=step, umax=umax, cfl=dt / self.dx * umax)
        r["urms"] = math.sqrt(2 * r["K"] / 3)
        r["eta"] = (p.nu ** 3 / r["eps"]) ** 0.25
        r["lam"] = r["urms"] * math.sqrt(15 * p.nu / r["eps"])
        r["Re_lambda"] = r["lam"] * r["urms"] / p.nu
        r["l0"] = r["urms"] ** 3 / r["eps"]
        r["Te"] = r["l0"] / r["urms"]
        r["kmax_eta"] = N / 3 * r["eta"]
        r["kmax_eta_sqrt2"] = math.sqrt(2) * N / 3 * r["eta"]
        ef = self.band_energy(u)
        if p.forcing != psc.FORCE_HOLD_ENERGY:
            A = p.eps_inj / (2 * ef) if p.forcing == psc.FORCE_CONST_POWER and ef > 1e-300 else 0.0
        r.update(A=A, E_forced=ef, P_inj=2 * A * ef)
        return _layout(r, E, Ephi, "fp64")

    def pressure(self, u):
        w = [self.grid(self.curl(u, i)) for i in range(3)]
        x = [self.grid(u[i]) for i in range(3)]
        q = self.modes(0.5 * (x[0] ** 2 + x[1] ** 2 + x[2] ** 2))
        dot = 0
        for i in range(3):
            j, l = (i + 1) % 3, (i + 2) % 3
            dot = dot + self.k[i] * self.modes(x[j] * w[l] - x[l] * w[j])
        out = -1j * dot / self.k2.clamp(min=1) - q
        out[self.K, self.K, 0] = 0
        return out


def exact(case, seed):
    if case["kind"] == "ensemble":
        return [_Exact(p).steps(_state(p, 1000 * seed + i).to(torch.complex128), case["steps"])[0]
                for i, p in _members(case)]
    if case["N"] > 520:  # 64-bit transforms of 1024^3 fields take too long
        return None
    p = _params(case)
    e, u = _Exact(p), _state(p, seed).to(torch.complex128)
    if case["kind"] == "diagnostics":
        out = dict(record=e.record(u, 0.0, p.dt, 0, 0.0))
        if case["pressure"]:
            out["pressure"] = e.pressure(u)
        return out
    u, *time = e.steps(u, case["steps"])
    out = dict(state=u)
    if case["record"]:
        out["record"] = e.record(u, *time)
    return out
