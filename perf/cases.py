"""Performance cases: the work a user has this library do, through its public calls.

A case is a dict of plain values; ``kind`` names the call:

  pipeline   ``pipeline.run``: handles, births, dipole and both spectra of a small run
  dipole     ``sfhk_dipole`` on births in hand (mixed, FP64 or double-float)
  sweep      a ``Batch`` of uneven laser configurations, run on its plan
  propagate  ``sfhk_propagate``: endpoints with stability matrix, action and prefactor
  births     ``sfhk_sample_births`` (standard or modified SPA, ADK)
  resample   ``sfhk_resample_births``: |I0| importance sampling of a pool
  spectrum   ``sfhk_spectrum`` of the length and the velocity bins
  gabor      ``sfhk_gabor`` and ``sfhk_emission_time`` of one burst

Targets, pulses and proposal widths are those of ``workloads.py``; the seed sets
the carrier-envelope phase and the birth draws, so every seed is another run.
"""
import math

import numpy as np
import torch

from paper_2601_17164_gb300 import pipeline as PL
from paper_2601_17164_gb300 import sfhk as S
from paper_2601_17164_gb300 import workloads as W

DEV = "cuda"
TARGETS = {"h": W.HYDROGEN, "ar": W.ARGON}
PRECISIONS = {"fp64": S.FP64, "mixed": S.MIXED, "df": S.DF}


# --- the cases ------------------------------------------------------------------
def listed():
    return [
        # a first look at a pulse: everything of one run, from handles to spectra, on few births
        dict(name="pipeline_h2_256", kind="pipeline", target="h", intensity=1e14, lam=800.0, cycles=2, dt=0.02,
             n_t=16, n_k=16),
        # the FP64 reference run on the 32 x 32 birth grid
        dict(name="fp64_h2_grid1024", kind="dipole", precision="fp64", target="h", intensity=1e14, lam=800.0, cycles=2,
             dt=0.02, n_t=32, n_k=32),
        # FP64 at a converged shape of the paper's first figure (H, 1600 nm, 3 cycles)
        dict(name="fp64_h3_20k", kind="dipole", precision="fp64", target="h", intensity=1e14, lam=1600.0, cycles=3,
             dt=0.02, n=20011),
        # a small mixed run: one point of a parameter scan, the size of the parity sample
        dict(name="mixed_h8_4096", kind="dipole", precision="mixed", target="h", intensity=1.5e14, lam=800.0, cycles=8,
             dt=0.01, n=4096),
        # the headline run: H, 800 nm, 8 cycles, one million births
        dict(name="mixed_h8_1m", kind="dipole", precision="mixed", target="h", intensity=1.5e14, lam=800.0, cycles=8,
             dt=0.01, n=1_000_000),
        # argon at 1600 nm (Tong-Lin potential), one shard of a large sample
        dict(name="mixed_ar6_50k", kind="dipole", precision="mixed", target="ar", intensity=1e14, lam=1600.0, cycles=6,
             dt=0.01, n=50_000),
        # a scan over intensity, wavelength, phase and duration, H and Ar, in one plan
        dict(name="sweep_8cfg", kind="sweep", n_cfg=8, pick=4, n_lo=3e3, n_hi=3e4, dt=0.02),
        # endpoints of a classical analysis (returns, angular momenta, stability), full 3D state
        dict(name="propagate_h2_4096", kind="propagate", precision="fp64", target="h", intensity=1e14, lam=800.0,
             cycles=2, dt=0.02, n=4096, frac=1.0),
        # the births of the headline run
        dict(name="births_h8_1m", kind="births", target="h", amp=0, intensity=1.5e14, lam=800.0, cycles=8, dt=0.01,
             n=1_000_000),
        # importance sampling: a pool four times the sample
        dict(name="resample_h8_4m", kind="resample", target="h", intensity=1.5e14, lam=800.0, cycles=8, dt=0.01,
             m=4_000_000, n=1_000_000),
        # both spectra of the headline run: 20 points per harmonic up to 60
        dict(name="spectrum_h8", kind="spectrum", target="h", intensity=1.5e14, lam=800.0, cycles=8, dt=0.01,
             n_omega=1200),
        # time-frequency map of the paper's three-cycle run and the emission times of its main burst
        dict(name="gabor_h3", kind="gabor", target="h", intensity=1e14, lam=1600.0, cycles=3, dt=0.02, n_times=400,
             n_omega=800),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["pipeline", "dipole", "dipole", "dipole", "sweep", "propagate", "births", "births", "resample",
                       "spectrum", "gabor"])
    target = rng.choice(["h", "h", "ar"])
    c = dict(kind=kind, target=target, intensity=round(rng.uniform(0.5e14, 2e14) / 1e11) * 1e11,
             lam=float(rng.randint(800, 1700)), cycles=rng.randint(2, 8), dt=rng.choice([0.01, 0.02]))
    if kind == "pipeline":
        c.update(target="h", lam=float(rng.randint(780, 900)), cycles=rng.randint(1, 2), dt=0.02,
                 n_t=rng.randint(3, 32), n_k=rng.randint(3, 32))
    elif kind == "dipole":
        c["precision"] = rng.choice(["mixed", "mixed", "mixed", "fp64", "fp64", "df"])
        if c["precision"] == "mixed":
            c.update(cycles=rng.randint(2, 6) if target == "ar" else rng.randint(2, 8), n=int(_log(rng, 100, 1e5)),
                     deterministic=rng.choice([0, 0, 0, 1]), pw_mask=rng.choice([0, 0, 0, 1, 6]))
            if c["deterministic"]:
                c["n"] = min(c["n"], 30_000)
        else:
            c.update(target="h" if c["precision"] == "df" else target, lam=float(rng.randint(800, 1100)),
                     cycles=rng.randint(2, 3), dt=0.02, n=int(_log(rng, 64, 2e4)))
    elif kind == "sweep":
        c = dict(kind="sweep", n_cfg=rng.randint(2, 12), pick=rng.randint(1, 10_000), n_lo=1e3, n_hi=2e4, dt=0.02)
    elif kind == "propagate":
        c.update(target="h", lam=float(rng.randint(800, 1000)), cycles=2, dt=0.02, n=int(_log(rng, 64, 8192)),
                 precision=rng.choice(["fp64", "fp64", "mixed"]), frac=round(rng.uniform(0.4, 1.0), 3))
    elif kind == "births":
        c.update(amp=rng.choice([0, 0, 1, 2]), n=int(_log(rng, 200, 2e6)))
    elif kind == "resample":
        m = int(_log(rng, 1000, 8e6))
        c.update(m=m, n=max(1, int(m * rng.uniform(0.05, 1.0))))
    elif kind == "spectrum":
        c.update(n_omega=int(_log(rng, 20, 6000)))
    else:
        c.update(n_times=int(_log(rng, 10, 800)), n_omega=int(_log(rng, 20, 1500)), cycles=rng.randint(2, 6))
    return c


# --- inputs ---------------------------------------------------------------------
def _cep(seed):
    return float(np.random.default_rng([int(seed), 1]).uniform(0.0, 2.0 * math.pi))


def _workload(case, seed):
    t = TARGETS[case["target"]]
    pulse = W.Pulse(case["intensity"], case["lam"], float(case["cycles"]), _cep(seed))
    sigma = W.adk_sigma(pulse.intensity_wcm2, t.ip)
    kw = dict(dt=case["dt"], sigma=sigma, seed=int(seed) + 1, h_max=40)
    if "n_t" in case:
        return W.Workload("grid", t, pulse, birth_mode=W.BIRTH_GRID, n=case["n_t"] * case["n_k"], n_t=case["n_t"],
                          n_k=case["n_k"], kmax=4.0 * sigma, **kw)
    return W.Workload("uniform", t, pulse, n=int(case.get("m", case.get("n", 1))), **kw)


def _bins(n):
    return torch.zeros(n, dtype=torch.float64, device=DEV)


def _cutoff(target, info):
    """Classical cutoff Ip + 3.17 Up as a harmonic order."""
    return (target.ip + 3.17 * info["E0"] ** 2 / (4.0 * info["omega"] ** 2)) / info["omega"]


def _signal(field, target, seed):
    """Dipole bins of a driven atom's shape: odd harmonics with a plateau up to the cutoff, each
    chirped and enveloped by the pulse, over the noise of a finite trajectory sample."""
    i = field.info
    n_h = int(_cutoff(target, i)) + 1
    rng = np.random.default_rng([int(seed), 2])
    t = i["t_start"] + i["t_out"] * torch.arange(i["n_bins"], dtype=torch.float64, device=DEV)
    env = torch.cos(math.pi * t / i["Tp"]) ** 2
    x = torch.zeros_like(t)
    for h in range(1, n_h, 2):
        a = (1.0 if h == 1 else 3e-3 * math.exp(-0.02 * h)) * rng.uniform(0.5, 1.5)
        chirp = rng.uniform(-1e-3, 1e-3) * i["omega"]
        x += a * env ** min(6, 1 + h // 8) * torch.cos(h * i["omega"] * t + chirp * t * t / i["Tp"] + rng.uniform(0, 6.28))
    noise = torch.from_numpy(rng.standard_normal(i["n_bins"])).to(DEV)
    return x + 1e-5 * env * noise


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        return _prepare_sweep(case, seed)
    w = _workload(case, seed)
    if kind == "pipeline":
        return {"kind": kind, "w": w}
    field, target = PL.make_handles(w, case.get("amp"))
    st = {"kind": kind, "w": w, "field": field, "target": target}
    nb = field.info["n_bins"]
    if kind == "dipole":
        st["births"] = PL.sample(w, field, target)
        st["pp"] = S.prop_params(PRECISIONS[case["precision"]], w.gamma, w.d_t,
                                 deterministic=case.get("deterministic", 0), pw_mask=case.get("pw_mask", 0))
        st.update(dl=_bins(nb), dv=_bins(nb), stats=S.new_stats())
    elif kind == "propagate":
        st["births"] = PL.sample(w, field, target)
        st["pp"] = S.prop_params(PRECISIONS[case["precision"]], w.gamma, w.d_t)
        st["n_end"] = int(case["frac"] * field.info["n_steps"])
        # births after the end point are not asked for
        st["n"] = int((st["births"].n0 <= st["n_end"]).sum().item())
        st["stats"] = S.new_stats()
    elif kind == "births":
        st["births"] = S.Births.empty(w.n)
    elif kind == "resample":
        st["pool"] = PL.sample(w, field, target)
        st.update(n=case["n"], out=S.Births.empty(case["n"]), nd=torch.zeros(1, dtype=torch.int64, device=DEV),
                  seed=int(seed) + 7)
    elif kind == "spectrum":
        st["omega"] = (torch.arange(case["n_omega"], dtype=torch.float64, device=DEV) + 1.0) * (field.info["omega"] / 20)
        st.update(x=_signal(field, w.target, seed), v=_signal(field, w.target, int(seed) + 100_003))
    else:
        i = field.info
        st["x"] = _signal(field, w.target, seed)
        top = _cutoff(w.target, i) * i["omega"] / case["n_omega"]
        st["omega"] = (torch.arange(case["n_omega"], dtype=torch.float64, device=DEV) + 1.0) * top
        st["times"] = torch.linspace(-0.45 * i["Tp"], 0.45 * i["Tp"], case["n_times"], dtype=torch.float64, device=DEV)
        st["window"] = (-0.2 * i["Tp"], 0.25 * i["Tp"])
    return st


def _prepare_sweep(case, seed):
    ws = W.batched_sweep(n_cfg=case["n_cfg"], seed=case["pick"], n_lo=case["n_lo"], n_hi=case["n_hi"], dt=case["dt"])
    fields, targets, births, dls, dvs = [], [], [], [], []
    for k, w in enumerate(ws):
        p = w.pulse
        # durations of a scan: 2 to 5 cycles
        w = W.Workload(w.name, w.target, W.Pulse(p.intensity_wcm2, p.lambda_nm, 2.0 + p.cycles % 4, _cep(int(seed) + k)),
                       dt=w.dt, n=w.n, sigma=w.sigma, seed=w.seed + int(seed))
        f, t = PL.make_handles(w)
        fields.append(f)
        targets.append(t)
        births.append(PL.sample(w, f, t))
        dls.append(_bins(f.info["n_bins"]))
        dvs.append(_bins(f.info["n_bins"]))
    stats = S.new_stats()
    pp = S.prop_params(S.MIXED)
    batch = S.Batch(fields, targets, births, [len(b) for b in births], pp, dls, dvs, stats)
    return {"kind": "sweep", "batch": batch, "dls": dls, "dvs": dvs, "stats": stats}


# --- one pass -------------------------------------------------------------------
def run(st):
    kind = st["kind"]
    if kind == "pipeline":
        r = PL.run(st["w"])
        return {"d_len": r.d_len, "d_vel": r.d_vel, "D_re": r.D_re, "D_im": r.D_im, "V_re": r.V_re, "V_im": r.V_im,
                "stats": r.stats}
    if kind == "dipole":
        st["dl"].zero_()
        st["dv"].zero_()
        st["stats"].zero_()
        S.sfhk_dipole(st["field"], st["target"], st["births"], len(st["births"]), st["pp"], st["dl"], st["dv"], st["stats"])
        return {"d_len": st["dl"], "d_vel": st["dv"], "stats": st["stats"]}
    if kind == "sweep":
        for x in st["dls"] + st["dvs"]:
            x.zero_()
        st["stats"].zero_()
        st["batch"].run()
        return {"d_len": st["dls"], "d_vel": st["dvs"], "stats": st["stats"]}
    if kind == "propagate":
        st["stats"].zero_()
        y, c, flags = S.sfhk_propagate(st["field"], st["target"], st["births"], st["n"], st["pp"], st["n_end"], st["stats"])
        return {"state": y, "C": c, "flags": flags, "stats": st["stats"]}
    if kind == "births":
        PL.sample(st["w"], st["field"], st["target"], births=st["births"])
        return _births_out(st["births"])
    if kind == "resample":
        S.sfhk_resample_births(st["pool"], len(st["pool"]), st["n"], st["seed"], st["out"], st["nd"])
        return dict(_births_out(st["out"]), n_distinct=st["nd"])
    if kind == "spectrum":
        D = PL.spectrum_of(st["x"], st["field"], st["omega"])
        V = PL.spectrum_of(st["v"], st["field"], st["omega"])
        return {"D_re": D[0], "D_im": D[1], "V_re": V[0], "V_im": V[1]}
    re, im = PL.gabor_of(st["x"], st["field"], st["times"], st["omega"])
    cen, peak = PL.emission_times(re, im, st["times"], *st["window"])
    return {"re": re, "im": im, "centroid": cen, "peak": peak}


def _births_out(b):
    return {k: getattr(b, k) for k in ("n0", "t0", "p0x", "p0y", "p0z", "q0z", "amp_re", "amp_im")}


# --- what a pass cannot do without ----------------------------------------------
# flops of one RK4 step of the 25-component planar state with the branch of the
# prefactor (soft-core), of the 43-component state, and what the Tong-Lin potential adds
PLANAR, FULL, TONGLIN = 471, 1253, 4 * 120


def _grid(lam, cycles, dt):
    n_steps = math.ceil(cycles * 2.0 * math.pi * lam / 45.5633525 / dt - 1e-9)
    return n_steps, n_steps // round(0.1 / dt) + 1


def work(case):
    kind = case["kind"]
    if kind == "sweep":
        total = {"bytes": 0.0, "flops": 0.0}
        for w in W.batched_sweep(n_cfg=case["n_cfg"], seed=case["pick"], n_lo=case["n_lo"], n_hi=case["n_hi"], dt=case["dt"]):
            c = dict(kind="dipole", target="h" if w.target is W.HYDROGEN else "ar", lam=w.pulse.lambda_nm,
                     cycles=2.0 + w.pulse.cycles % 4, dt=w.dt, n=w.n)
            for k, v in work(c).items():
                total[k] += v
        return total
    n_steps, nb = _grid(case["lam"], case["cycles"], case["dt"])
    n = case["n_t"] * case["n_k"] if "n_t" in case else case.get("n", 0)
    per = PLANAR + (TONGLIN if case["target"] == "ar" else 0)
    if kind in ("dipole", "pipeline"):
        # births in, bins out; births live half the pulse on average
        extra = 2 * 8.0 * nb * 800 if kind == "pipeline" else 0.0
        return {"bytes": 60.0 * n + 8.0 * (2 * n_steps + 1) + 16.0 * nb, "flops": 0.5 * n * n_steps * per + extra}
    if kind == "propagate":
        f = case["frac"]
        return {"bytes": n * f * (60.0 + 43 * 8 + 17), "flops": 0.5 * n * f * f * n_steps * (FULL if case["target"] == "h" else FULL + TONGLIN)}
    if kind == "births":
        return {"bytes": 60.0 * n, "flops": 2000.0 * n}
    if kind == "resample":
        # the pool's amplitudes once, the drawn births read and written
        return {"bytes": 16.0 * case["m"] + 2 * 60.0 * n, "flops": 4.0 * case["m"]}
    if kind == "spectrum":
        return {"bytes": 2 * (8.0 * nb + 24.0 * case["n_omega"]), "flops": 2 * 4.0 * nb * case["n_omega"]}
    sigma_bins = case["lam"] / 45.5633525 / 3.0 / 0.1
    pairs = case["n_times"] * case["n_omega"] * min(nb, 18.0 * sigma_bins)
    return {"bytes": 8.0 * nb + 2 * 16.0 * case["n_times"] * case["n_omega"], "flops": 4.0 * pairs}


# --- the same in 64 bits, from the formulas alone --------------------------------
class _Pulse:
    def __init__(self, w):
        p = w.pulse
        self.E0 = math.sqrt(p.intensity_wcm2 / 3.50944758e16)
        self.om = 45.5633525 / p.lambda_nm
        self.Tp = p.cycles * 2.0 * math.pi / self.om
        self.cep, self.dt = p.cep, w.dt
        self.t0 = -0.5 * self.Tp
        self.n_steps = int(math.ceil(self.Tp / w.dt - 1e-9))
        self.n_out = int(math.floor(0.1 / w.dt + 0.5))
        self.n_bins = self.n_steps // self.n_out + 1
        Om = 2.0 * math.pi / self.Tp
        self.a = [-self.E0 / (2 * self.om), -self.E0 / (4 * self.om), -self.E0 / (4 * self.om)]
        self.w = [self.om, self.om + Om, self.om - Om]

    def A(self, t):
        return sum(a * torch.sin(w * t + self.cep) for a, w in zip(self.a, self.w))

    def E(self, t):
        return sum(-a * w * torch.cos(w * t + self.cep) for a, w in zip(self.a, self.w))

    def F(self, t):
        out = 0
        for a, w in zip(self.a, self.w):
            out = out + (a / w * (math.cos(self.cep) - torch.cos(w * t + self.cep)) if abs(w) > 1e-14
                         else a * math.sin(self.cep) * t)
        return out

    def G(self, t):
        def ic(w, th):
            return math.cos(th) * t if abs(w) < 1e-14 else (torch.sin(w * t + th) - math.sin(th)) / w
        return sum(0.5 * a * b * (ic(v - u, 0.0) - ic(v + u, 2 * self.cep))
                   for a, v in zip(self.a, self.w) for b, u in zip(self.a, self.w))

    def table(self):
        t = self.t0 + 0.5 * self.dt * torch.arange(2 * self.n_steps + 1, dtype=torch.float64, device=DEV)
        return torch.where(t.abs() <= 0.5 * self.Tp, self.E(t), torch.zeros_like(t))


def _saddle(P, ip, t0, kx, ky):
    """Smallest t_t > 0 with Im A(t0 + i t_t) = s kappa; nan where there is none."""
    c = [a * torch.cos(w * t0 + P.cep) for a, w in zip(P.a, P.w)]
    s = torch.where(P.E(t0) > 0, -1.0, 1.0)
    goal = s * torch.sqrt(2 * ip + kx * kx + ky * ky)
    f = lambda x: sum(cj * torch.sinh(w * x) for cj, w in zip(c, P.w)) - goal  # noqa: E731
    wmax = max(abs(w) for w in P.w)
    h = 0.02 / wmax
    lo = torch.full_like(t0, math.nan)
    up0 = -goal > 0
    live = torch.ones_like(up0)
    for k in range(1, int((25.0 / wmax) / h) + 1):
        hit = live & ((f(torch.full_like(t0, k * h)) > 0) != up0)
        lo = torch.where(hit, torch.full_like(t0, (k - 1) * h), lo)
        live = live & ~hit
        if k % 50 == 0 and not bool(live.any()):
            break
    hi = lo + h
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        same = (f(mid) > 0) == up0
        lo, hi = torch.where(same, mid, lo), torch.where(same, hi, mid)
    return 0.5 * (lo + hi)


def _tunnel(T, kx, ky, kz):
    k2 = kx * kx + ky * ky + kz * kz
    s = torch.zeros_like(kz)
    for c, a in zip(T.c, T.alpha):
        g = torch.exp(-0.25 / a * k2)
        s = s + (c * 0.5 * math.pi ** 1.5 * a ** -2.5 * kz * g if T.gto_l == 0
                 else c * 0.25 * math.pi ** 1.5 * a ** -3.5 * (2 * a - kz * kz) * g)
    return (2 * math.pi) ** -1.5 * (-1j * s if T.gto_l == 0 else s)


def _adk_rate(T, F):
    k = math.sqrt(2 * T.ip)
    return 0.5 * (2 * T.gto_l + 1) * k ** (1 - 2 / k) * (2 * k ** 3 / F) ** (2 / k - 1) * torch.exp(-2 * k ** 3 / (3 * F))


def _amplitude(P, T, t0, kx, ky, kind, n2=0.0):
    E0 = P.E(t0)
    tt = _saddle(P, T.ip, t0, kx, ky)
    none = torch.isnan(tt)
    tt = torch.where(none, torch.ones_like(tt), tt)
    ts = torch.complex(t0, tt)
    A0, As, kp2 = P.A(t0), P.A(ts), kx * kx + ky * ky
    kz = A0 - As.real
    dF, dG = P.F(t0) - P.F(ts), P.G(t0) - P.G(ts)
    qz = dF.real
    cc = kz - A0
    integ = 0.5 * ((kp2 + cc * cc) * torch.complex(torch.zeros_like(tt), -tt) + 2 * cc * dF + dG)
    act = T.ip * ts - integ
    if kind == 2:
        k = math.sqrt(2 * T.ip)
        F = E0.abs()
        rho = _adk_rate(T, F) * k / (math.pi * F) * torch.exp(-k * kp2 / F)
        kz, qz = torch.zeros_like(kz), -T.ip / E0
        amp = torch.sqrt(n2 * rho) * torch.exp(1j * act.real)
    else:
        v, Es = kz - A0 + As, P.E(ts)
        ph = torch.exp(1j * (act + kz * qz))
        amp = Es * _tunnel(T, kx, ky, v) / torch.sqrt(Es * v) * ph if kind == 0 else ph / (Es * v)
    amp = torch.where(none | ~torch.isfinite(amp.real) | ~torch.isfinite(amp.imag), torch.zeros_like(amp), amp)
    zero = torch.zeros_like(kz)
    return torch.where(none, zero, kz), torch.where(none, zero, qz), amp


def _adk_norm2(P, T):
    num = den = 0.0
    ks = math.floor(P.cep / math.pi + 0.5)
    for j in (-1, 1):
        tj = torch.tensor(((ks + j) * math.pi - P.cep) / P.om, dtype=torch.float64, device=DEV)
        F = P.E(tj).abs()
        h = 6 * torch.sqrt(F / math.sqrt(2 * T.ip)) / 128
        i = torch.arange(1, 129, dtype=torch.float64, device=DEV)
        c = torch.where(i == 128, 1.0, torch.where(i % 2 == 1, 4.0, 2.0))
        a = _amplitude(P, T, tj.expand(128), i * h, torch.zeros_like(i), 0)[2]
        num += float(2 * math.pi * h / 3 * (c * i * h * a.abs() ** 2).sum())
        den += float(_adk_rate(T, F))
    return num / den


def _exact_births(w, kind):
    P, T, n = _Pulse(w), w.target, w.n
    M = P.n_steps - 1
    if w.birth_mode == W.BIRTH_GRID:
        i = np.arange(n)
        nb = np.clip(np.floor((i // w.n_k + 0.5) * P.n_steps / w.n_t), 1, M).astype(np.int64)
        dk = w.kmax / w.n_k
        kx = (i % w.n_k + 0.5) * dk
        ky = np.zeros(n)
        wt = 2 * math.pi * kx * dk * (P.n_steps * P.dt / w.n_t)
    else:
        raw = np.random.Philox(key=[w.seed, 0], counter=[2 ** 64 - 1] * 4).random_raw(4 * n).reshape(n, 4)
        num = np.arange(n, dtype=object) * (1 << 32) + (raw[:, 0] >> np.uint64(32)).astype(object)
        nb = 1 + np.array(num * M // (n << 32), dtype=np.int64)
        u1 = ((raw[:, 1] >> np.uint64(11)) + np.uint64(1)).astype(np.float64) * 2.0 ** -53
        u2 = (raw[:, 2] >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
        rad = w.sigma * np.sqrt(-2 * np.log(u1))
        kx, ky = rad * np.cos(2 * math.pi * u2), rad * np.sin(2 * math.pi * u2)
        s2 = w.sigma ** 2
        wt = 2 * math.pi * s2 * np.exp((kx * kx + ky * ky) / (2 * s2)) * (M * P.dt) / n
    kx, ky, wt = (torch.from_numpy(np.ascontiguousarray(v)).to(DEV) for v in (kx, ky, wt))
    t0 = P.t0 + torch.from_numpy(nb).to(DEV).double() * P.dt
    kz, qz, amp = _amplitude(P, T, t0, kx, ky, kind, _adk_norm2(P, T) if kind == 2 else 0.0)
    return {"n0": torch.from_numpy(nb.astype(np.int32)), "t0": t0, "p0x": kx, "p0y": ky, "p0z": kz, "q0z": qz,
            "amp_re": wt * amp.real, "amp_im": wt * amp.imag}


def _exact_spectrum(x, info, omega):
    k = torch.arange(x.numel(), dtype=torch.float64, device=DEV)
    t = info["t_start"] + k * info["t_out"]
    tau = 0.5 * info["Tp"]
    y = torch.where(t.abs() <= tau, 0.5 * (1 + torch.cos(math.pi * t / tau)), torch.zeros_like(t)) * x * info["t_out"]
    re, im = torch.empty_like(omega), torch.empty_like(omega)
    for a in range(0, omega.numel(), 256):
        ph = omega[a:a + 256, None] * t
        re[a:a + 256], im[a:a + 256] = torch.cos(ph) @ y, torch.sin(ph) @ y
    return re, im


def _exact_gabor(st):
    i, x, om = st["field"].info, st["x"], st["omega"]
    sig = 1.0 / (3.0 * i["omega"])
    t = i["t_start"] + i["t_out"] * torch.arange(x.numel(), dtype=torch.float64, device=DEV)
    d = t - st["times"][:, None]
    y = torch.where(d.abs() <= 9 * sig, torch.exp(-d * d / (2 * sig * sig)), torch.zeros_like(d)) * x * i["t_out"]
    re, im = [], []
    for a in range(0, om.numel(), 256):
        ph = t[:, None] * om[a:a + 256]
        re.append(y @ torch.cos(ph))
        im.append(y @ torch.sin(ph))
    re, im = torch.cat(re, 1), torch.cat(im, 1)
    T = st["times"]
    sel = torch.nonzero((T >= st["window"][0]) & (T <= st["window"][1]))[:, 0]
    nan = torch.full((om.numel(),), math.nan, dtype=torch.float64, device=DEV)
    if sel.numel() == 0:
        return {"re": re, "im": im, "centroid": nan, "peak": nan}
    p, tt = (re * re + im * im)[sel], T[sel]
    cen = (tt[:, None] * p).sum(0) / p.sum(0)
    j = p.argmax(0)
    inner = (j > 0) & (j < sel.numel() - 1)
    jm = j.clamp(1, max(1, sel.numel() - 2))
    y0, ym, yp = (torch.log(p.gather(0, (jm + s).clamp(0, sel.numel() - 1)[None])[0]) for s in (0, -1, 1))
    curv = ym - 2 * y0 + yp
    h = float(tt[1] - tt[0]) if sel.numel() > 1 else 0.0
    return {"re": re, "im": im, "centroid": cen,
            "peak": torch.where(inner & (curv < 0), tt[j] + 0.5 * h * (ym - yp) / curv, tt[j])}


def _exact_resample(st):
    pool, m, n = _births_out(st["pool"]), len(st["pool"]), st["n"]
    re, im = pool["amp_re"].cpu().numpy(), pool["amp_im"].cpu().numpy()
    wgt = np.sqrt(re * re + im * im)
    B = 62 - max(1, math.ceil(math.log2(max(2, m))))
    q = np.floor(wgt * (2.0 ** B / wgt.max())).astype(np.uint64)
    C = np.cumsum(q)
    Q = int(C[-1])
    U = int(np.random.Philox(key=[st["seed"], 1], counter=[2 ** 64 - 1] * 4).random_raw(1)[0]) >> 32
    t = np.array([((j << 32) + U) * Q // (n << 32) for j in range(n)], dtype=np.uint64)
    mult = np.bincount(np.searchsorted(C, t, side="right"), minlength=m)
    idx = np.nonzero(mult)[0]
    f = (mult[idx].astype(np.float64) * float(Q)) / (float(n) * q[idx].astype(np.float64))
    pad = np.concatenate([idx, np.full(n - len(idx), idx[-1] if len(idx) else 0)])
    out = {k: v.cpu().numpy()[pad] for k, v in pool.items()}
    f = np.concatenate([f, np.zeros(n - len(idx))])
    out["amp_re"], out["amp_im"] = out["amp_re"] * f, out["amp_im"] * f
    return dict(out, n_distinct=np.array([len(idx)], dtype=np.int64))


def _det3(z):
    return (z[0][0] * (z[1][1] * z[2][2] - z[1][2] * z[2][1]) - z[0][1] * (z[1][0] * z[2][2] - z[1][2] * z[2][0])
            + z[0][2] * (z[1][0] * z[2][1] - z[1][1] * z[2][0]))


def _exact_trajectories(w, births, n_end, dipole):
    """RK4 of the full 43-component state of the soft-core atom in 64 bits, all births at
    once; the dipole bins, or the endpoints."""
    P, T, gam = _Pulse(w), w.target, w.gamma
    a2 = T.pot_param[0] ** 2
    n0 = births["n0"].to(DEV).long()
    n = n0.numel()
    amp = torch.complex(births["amp_re"], births["amp_im"])
    on = torch.ones_like(n0, dtype=torch.bool) if not dipole else amp != 0
    q = torch.stack([torch.zeros_like(births["q0z"]), torch.zeros_like(births["q0z"]), births["q0z"]])
    p = torch.stack([births["p0x"], births["p0y"], births["p0z"]])
    X = torch.zeros(3, 6, n, dtype=torch.float64, device=DEV)
    Y = torch.zeros_like(X)
    for c in range(3):
        X[c, c], Y[c, c + 3] = 1.0, 1.0
    act = torch.zeros(n, dtype=torch.float64, device=DEV)
    D = torch.ones(n, dtype=torch.complex128, device=DEV)
    sgn = torch.ones(n, dtype=torch.float64, device=DEV)
    E = P.table()
    h = P.dt
    al = torch.tensor(T.alpha, dtype=torch.float64, device=DEV)[:, None]
    be, cf = gam + al, torch.tensor(T.c, dtype=torch.float64, device=DEV)[:, None]
    nl = (2 * gam / math.pi) ** 0.75 * math.pi ** 1.5
    d_len = torch.zeros(P.n_bins, dtype=torch.float64, device=DEV)
    d_vel = torch.zeros_like(d_len)

    def rates(q, p, X, Y, e):
        s2 = 1.0 / ((q * q).sum(0) + a2)
        s = torch.sqrt(s2)
        g = s2 * s
        pd = -g * q
        pd[2] -= e
        Yd = -(g * X + (-3 * g * s2 * (q[:, None] * X).sum(0)) * q[:, None])
        return p, pd, Y, Yd, 0.5 * (p * p).sum(0) + s - q[2] * e

    for k in range(n_end + 1):
        if dipole and k % P.n_out == 0:
            live = on & (n0 <= k)
            p2, q2, pq = (p * p).sum(0), (q * q).sum(0), (p * q).sum(0)
            g = cf * be ** -2.5 * torch.exp(torch.complex(-0.25 / be * p2 - al * gam / be * q2, -al / be * pq))
            C = sgn * torch.sqrt(D)
            ph = torch.exp(1j * (act - T.ip * (P.t0 + k * h))) * C * amp
            dl = torch.complex(2 * gam * q[2], p[2]) * g.sum(0) * ph
            dv = torch.complex(p[2], -2 * gam * q[2]) * (al * g).sum(0) * ph
            d_len[k // P.n_out] = (-2 * 0.5 * nl * torch.where(live, dl.real, torch.zeros_like(act))).sum()
            d_vel[k // P.n_out] = (-2 * nl * torch.where(live, dv.real, torch.zeros_like(act))).sum()
        if k == n_end:
            break
        ea, eb, ec = E[2 * k], E[2 * k + 1], E[2 * k + 2]
        y0 = (q, p, X, Y)
        r1 = rates(*y0, ea)
        r2 = rates(*(u + 0.5 * h * r for u, r in zip(y0, r1)), eb)
        r3 = rates(*(u + 0.5 * h * r for u, r in zip(y0, r2)), eb)
        r4 = rates(*(u + h * r for u, r in zip(y0, r3)), ec)
        inc = [h / 6 * (a + 2 * (b + c) + d) for a, b, c, d in zip(r1, r2, r3, r4)]
        live = (n0 <= k).double()
        q, p, X, Y = (u + live * i for u, i in zip(y0, inc))
        act = act + live * inc[4]
        Z = 0.5 * torch.complex(Y[:, 3:] + X[:, :3], -2 * gam * X[:, 3:] + Y[:, :3] / (2 * gam))
        new = _det3(Z)
        flip = (D.imag * new.imag < 0) & ((D.real * new.imag - D.imag * new.real > 0) == (D.imag > 0))
        sgn = torch.where(flip, -sgn, sgn)
        D = new
    if dipole:
        return {"d_len": d_len, "d_vel": d_vel}
    y = torch.cat([q, p, X[:, :3].reshape(9, n), X[:, 3:].reshape(9, n), Y[:, :3].reshape(9, n), Y[:, 3:].reshape(9, n),
                   act[None]])
    return {"state": y, "C": sgn * torch.sqrt(D)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        return None
    w = _workload(case, seed)
    if kind == "births":
        return _exact_births(w, case["amp"]) if w.n <= 1_000_000 else None
    if kind in ("dipole", "pipeline", "propagate"):
        # some 160 torch operations a step: up to 12000 steps, H only
        if _Pulse(w).n_steps > 12_000 or case["target"] != "h" or w.n > 8192 or case.get("pw_mask"):
            return None
        b = _exact_births(w, 0)
        if kind == "propagate":
            n_end = int(case["frac"] * _Pulse(w).n_steps)
            keep = int((b["n0"] <= n_end).sum())
            return _exact_trajectories(w, {k: v[:keep] for k, v in b.items()}, n_end, False)
        out = _exact_trajectories(w, b, _Pulse(w).n_steps, True)
        if kind == "pipeline":
            P = _Pulse(w)
            info = {"t_start": P.t0, "t_out": 0.1, "Tp": P.Tp}
            om = torch.tensor(W.omega_grid(w), dtype=torch.float64, device=DEV)
            for k, x in (("D", "d_len"), ("V", "d_vel")):
                out[k + "_re"], out[k + "_im"] = _exact_spectrum(out[x], info, om)
        return out
    st = prepare(case, seed)
    if kind == "resample":
        return _exact_resample(st)
    if kind == "spectrum":
        D, V = (_exact_spectrum(st[k], st["field"].info, st["omega"]) for k in ("x", "v"))
        return {"D_re": D[0], "D_im": D[1], "V_re": V[0], "V_im": V[1]}
    return _exact_gabor(st)
