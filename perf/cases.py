"""The work a user has this library do, as measurable cases.

A case is one pass of a program that fits a galaxy: advance the fit (or the batch of fits)
by a segment of steps, then read what such a program reads back between segments: the
smoothed and raw observables, chi^2 and the particle weights. Every segment is a multiple
of the prior period (25 steps), so that every pass holds the same mix of steps. Particles
and targets are drawn on the GPU from the seed; the targets are the observables of a second
realisation, as measured data would be. A mixed-precision fit holds its particles and
computes their kernels in FP32, so its results are handed on in that type.

`exact` computes the same results in FP64 with plain torch operations and none of the
library's code, in the order of the paper: push, observables, smoothing, residuals, priors,
force of change, renormalisation.
"""
from __future__ import annotations

import ctypes as C
import math

import numpy as np
import torch

from paper_1202_2355_gb300 import binding as B
from paper_1202_2355_gb300.workloads import Group

EVERY = 25  # prior updates every 25 steps, as in all workloads of this repository


# ------------------------------------------------------------------ cases

def listed():
    return [
        # the smallest calls: a 3,001-particle FP64 fit watched step by step, chi^2 read after
        # each one and the particles followed (a first look at a potential, a notebook)
        dict(name="watch_fp64_3k", kind="fit", precision="fp64", pot="hernquist", obs="c1", prior="cell", n=3001,
             steps=1, reads=25),
        # the 20,000-particle FP64 Hernquist fit (the paper-scale run of workload c1)
        dict(name="fit_fp64_20k", kind="fit", precision="fp64", pot="hernquist", obs="c1", prior="cell", n=20000,
             steps=100, reads=1),
        # the million-particle FP64 fit of 150 observables (workload c2)
        dict(name="fit_fp64_1m", kind="fit", precision="fp64", pot="hernquist", obs="c2", prior="cell", n=1000000,
             steps=100, reads=1),
        # stars in a Hernquist + NFW halo, mixed precision (workload c3), an odd count
        dict(name="fit_nfw_mixed_2m", kind="fit", precision="mixed", pot="nfw", obs="c3", prior="cell", n=2000003,
             steps=200, reads=1),
        # the grid-less priors of the GWR/MPR experiment: a window of cells on a 90 x 30 lattice
        dict(name="window_mixed_1m", kind="fit", precision="mixed", pot="hernquist", obs="c2", prior="window",
             n=1000000, steps=200, reads=1),
        # 64 x 64 maps of five moments in the flattened log potential, 8,000,000 particles (c4)
        dict(name="maps64_mixed_8m", kind="fit", precision="mixed", pot="log", obs="maps", side=64, prior="cell",
             n=8000000, steps=50, reads=1),
        # smaller FP64 maps with the global entropy and the explicit-Euler update, ragged count
        dict(name="maps16_gwr_fp64_100k", kind="fit", precision="fp64", pot="log", obs="maps", side=16, prior="gwr",
             n=100003, steps=100, reads=1),
        # 3-D density coefficients a_lm fitted beside the annuli (the data of the paper's fits)
        dict(name="alm_fp64_50k", kind="fit", precision="fp64", pot="hernquist", obs="alm", prior="cell", n=50000,
             steps=50, reads=1),
        # the self-consistent potential with the mass-to-light ratio fitted during the run
        dict(name="scf_fp64_20k", kind="fit", precision="fp64", pot="scf", obs="c1", prior="cell", n=20001, steps=50,
             reads=1),
        # a grid of trial haloes x initial models: 96 uneven mixed fits at once (c5, 5e7 particles)
        dict(name="batch_mixed_96", kind="batch", precision="mixed", fits=96, nlo=50000, nhi=2000000, steps=100),
        # a quick FP64 scan: 24 small fits of uneven size
        dict(name="batch_fp64_24", kind="batch", precision="fp64", fits=24, nlo=2000, nhi=50000, steps=100),
        # the recovery diagnostics of a finished model and of its target (kinematics and (E, x) grid)
        dict(name="diagnose_mixed_2m", kind="diag", precision="mixed", pot="nfw", obs="c3", prior="cell", n=2000003),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) | 1


def draw(rng):
    what = rng.choice(["fit", "fit", "fit", "fit", "maps", "maps", "alm", "scf", "batch", "batch", "diag"])
    prec = rng.choice(["fp64", "mixed"])
    if what == "batch":
        fits = rng.randint(2, 96) if prec == "mixed" else rng.randint(2, 32)
        nlo = _log_int(rng, 1000, 20000)
        nhi = _log_int(rng, 2 * nlo, 500000 if prec == "mixed" else 100000)
        return dict(kind="batch", precision=prec, fits=fits, nlo=nlo, nhi=nhi, steps=rng.choice([25, 50, 100]))
    if what == "diag":
        return dict(kind="diag", precision=prec, pot=rng.choice(["hernquist", "nfw", "log"]), obs="c1", prior="cell",
                    n=_log_int(rng, 10000, 2000000))
    if what in ("alm", "scf"):
        return dict(kind="fit", precision="fp64", pot="scf" if what == "scf" else rng.choice(["hernquist", "nfw"]),
                    obs="c1" if what == "scf" else "alm", prior="cell", n=_log_int(rng, 2000, 50000), steps=25, reads=1)
    n = _log_int(rng, 1000, 1000000 if prec == "fp64" else 4000000)
    steps, reads = (1, 25) if n < 20000 and rng.random() < 0.5 else (rng.choice([50, 100]), 1)
    if what == "maps":
        return dict(kind="fit", precision=prec, pot="log", obs="maps", side=rng.randint(8, 64),
                    prior=rng.choice(["cell", "gwr", "window"]), n=max(n, 20001), steps=steps, reads=reads)
    return dict(kind="fit", precision=prec, pot=rng.choice(["hernquist", "nfw", "log"]),
                obs=rng.choice(["c1", "c2", "c3"]), prior=rng.choice(["cell", "cell", "window", "gwr"]), n=n,
                steps=steps, reads=reads)


def _batch_counts(case):
    g = np.random.default_rng(1)  # the sizes belong to the case, not to the seed
    u = g.random(case["fits"])
    return [int(v) for v in np.exp(math.log(case["nlo"]) + u * math.log(case["nhi"] / case["nlo"]))]


def work(case):
    """Per particle and step: the six coordinates and the weight read and written and the 2-byte
    prior cell read; 88 operations for the push, the observables, the force of change and the
    binning. A diagnosis reads every particle (coordinates and weight) for each of its two grids."""
    size = 8 if case["precision"] == "fp64" else 4
    if case["kind"] == "diag":
        n = case["n"] + DIAG_TARGET
        return {"bytes": 2 * 7 * size * n, "flops": 2 * 60 * n}
    n = sum(_batch_counts(case)) if case["kind"] == "batch" else case["n"]
    steps = case["steps"] * case.get("reads", 1)
    return {"bytes": (14 * size + 2) * n * steps + 8 * n, "flops": 88 * n * steps}


# ------------------------------------------------------------------ galaxies

DEV = "cuda"
DIAG_TARGET = 200001
SPH = dict(n_r=21, n_phi=8, n_ct=4, r_min=0.05, r_max=20.0)  # the spherical grid of the intrinsic kinematics


def _edges(lo, hi, n):
    return np.exp(np.linspace(math.log(lo), math.log(hi), n + 1))


def _rng(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1009 + stream) % (1 << 62))
    return g


def _rand(g, n):
    return torch.rand(n, generator=g, device=DEV, dtype=torch.float64)


def _randn(g, n):
    return torch.randn(n, generator=g, device=DEV, dtype=torch.float64)


def _nfw_mu(q):
    return np.log1p(q) - q / (1 + q)


def _halo(m200, rs):
    return dict(kind="hernquist_nfw", G=1.0, M=1.0, a=1.0, Ms=m200 / float(_nfw_mu(10.0)), rs=rs)


def _enclosed(pot, r):
    if pot["kind"] in ("log", "scf"):
        v0, r0 = pot["v0"], pot["r0"]
        star = 1.2 * r * r / (1 + r) ** 2 if pot["kind"] == "scf" else 0.0
        return v0 * v0 * r ** 3 / (r0 * r0 + r * r) + star
    m = r * r / (1 + r) ** 2
    return m + pot["Ms"] * _nfw_mu(r / pot["rs"]) if pot["kind"] == "hernquist_nfw" else m


def _realise(g, n, pot, aniso=1.0, flat=1.0, spin=0.0):
    """A Hernquist tracer (r < 50) with Gaussian velocities of the Jeans dispersion in `pot`."""
    lr = np.linspace(math.log(1e-4), math.log(1e4), 1600)
    r = np.exp(lr)
    rho = 1.0 / (r * (1 + r) ** 3)
    f = rho * _enclosed(pot, r) / r
    seg = 0.5 * (f[1:] + f[:-1]) * np.diff(lr)
    s2 = torch.tensor(np.concatenate([np.cumsum(seg[::-1])[::-1], [seg[-1]]]) / rho, device=DEV)
    u = torch.sqrt(_rand(g, n)) * (50.0 / 51.0)
    rad = (u / (1 - u)).clamp_min(1e-6)
    t = ((torch.log(rad) - lr[0]) / (lr[1] - lr[0])).clamp(0, len(lr) - 1.001)
    k = t.long()
    sig2 = s2[k] + (t - k) * (s2[k + 1] - s2[k])
    del t, k
    ct = 2 * _rand(g, n) - 1
    ph = 2 * math.pi * _rand(g, n)
    st, cp, sp = torch.sqrt(1 - ct * ct), torch.cos(ph), torch.sin(ph)
    a2 = aniso * aniso
    st_v = torch.sqrt(3 * sig2 / (a2 + 2))
    vr, vt, vp = aniso * st_v * _randn(g, n), st_v * _randn(g, n), st_v * _randn(g, n)
    pos = torch.stack([rad * st * cp, rad * st * sp, rad * ct * flat])
    vel = torch.stack([vr * st * cp + vt * ct * cp - vp * sp, vr * st * sp + vt * ct * sp + vp * cp, vr * ct - vt * st])
    if spin:
        R = rad * st
        v = spin * R / torch.sqrt(1 + R * R) * torch.tanh(R)
        vel[0] -= v * sp
        vel[1] += v * cp
    return pos, vel, torch.full((n,), 1.0 / n, device=DEV, dtype=torch.float64)


ALM = [f"alm_{l}_{m}" for l in range(3) for m in range(-l, l + 1)] + ["alm_4_0", "alm_4_4"]


def _groups(case):
    if case["obs"] == "c1":
        return [Group("annuli", ["mass"], [0.01], edges=_edges(0.05, 20, 30)),
                Group("annuli", ["v2", "gh4"], [0.01, 0.01], edges=_edges(0.1, 5, 15))]
    if case["obs"] == "c2":
        return [Group("annuli", ["mass"], [0.01], edges=_edges(0.05, 20, 60)),
                Group("annuli", ["v2", "gh3", "gh4"], [0.01] * 3, edges=_edges(0.1, 8, 30))]
    if case["obs"] == "c3":
        return [Group("annuli", ["mass"], [0.01], edges=_edges(0.05, 10, 40)),
                Group("annuli", ["v2", "gh4"], [0.05, 0.03], edges=_edges(0.1, 2, 10))]
    if case["obs"] == "alm":
        return _groups(dict(obs="c1")) + [Group("shells", ALM, [3.0] * len(ALM), edges=_edges(0.05, 20, 15))]
    side = case["side"]
    return [Group("pixels", ["mass", "gh1", "gh2", "gh3", "gh4"], [0.02] * 5, nx=side, ny=side,
                  box=(-4.0, 4.0, -4.0, 4.0))]


def _potential(case):
    if case["pot"] == "hernquist":
        return dict(kind="hernquist", G=1.0, M=1.0, a=1.0)
    if case["pot"] == "nfw":
        return _halo(20.0, 8.0)
    if case["pot"] == "log":
        return dict(kind="log", G=1.0, M=0.0, a=1.0, v0=1.0, r0=1.0, q=0.8)
    return dict(kind="scf", G=1.0, v0=0.45, r0=1.0, q=0.9, scf_r=_edges(0.05, 30, 11), scf_lmax=2, ups=1.2,
                eps_ups=2e-4)


def _prior(case, pot, pos, vel):
    """The (E, x) grid over the energies of the model; the log potential takes signed L_z in exp(E)."""
    if case["prior"] == "gwr":
        return dict(mode="gwr", nE=1, nx=1, e_spacing="linear", signed_lz=0, update_every=EVERY, Emin=0.0, Emax=1.0)
    nE, nx = {"c1": (30, 10), "c2": (50, 20), "c3": (30, 10), "alm": (30, 10), "maps": (40, 20)}[case["obs"]]
    grid = dict(mode="mpr", nE=nE, nx=nx, e_spacing="logneg", signed_lz=0, update_every=EVERY)
    if pot["kind"] == "scf":
        grid.update(nE=12, nx=6, e_spacing="linear", Emin=-3.0, Emax=2.0)
    elif pot["kind"] == "log":
        E = 0.5 * (vel * vel).sum(0) + _phi(pot, pos)
        grid.update(e_spacing="exp", signed_lz=1, Emin=float(E.min()), Emax=float(E.max()))
    else:
        ms, rs = pot.get("Ms", 0.0), pot.get("rs", 1.0)
        grid.update(Emin=-1.0 - ms / rs, Emax=-1.0 / 51.0 - ms * math.log1p(50.0 / rs) / 50.0)
    if case["prior"] == "window":
        grid.update(nE=90, nx=30, window=(1, 1))
    return grid


def _params(case):
    p = dict(dt=0.01, eps=1e-3, mu=1e-2, alpha=0.02, renormalize=1, update_rule="exp", n_relax=0)
    if case["obs"] == "c2":
        p.update(dt=0.005)
    # the explicit update is stable for a rate that falls with the particles per datum
    p["eps"] *= min(1.0, case["n"] / {"c1": 40000, "c2": 200000, "c3": 200000}.get(case["obs"], 20000))
    if case["obs"] == "alm" or case["pot"] != "hernquist":
        p["eps"] *= 0.3
    if case["prior"] == "window":
        p.update(mu=1e4)
    if case["obs"] == "maps":
        p.update(eps=1e-6 * min(1.0, case["n"] / (1000 * case["side"] ** 2)))
    if case["prior"] == "gwr":
        p.update(eps=0.1 * p["eps"], mu=1.0, update_rule="euler" if case["obs"] == "maps" else "exp")
    return p


def _targets(groups, incl, particles, gen):
    """Y, sigma(Y) and the Gaussian parameters V_p, sigma_p per aperture of a target realisation."""
    pos, vel, w = particles
    V, S = [], []
    for g in groups:
        if g.geometry == "shells":
            V.append(torch.zeros(g.n_ap, device=DEV, dtype=torch.float64))
            S.append(torch.ones(g.n_ap, device=DEV, dtype=torch.float64))
            continue
        p, vlos = _aperture(g, incl, pos, vel)
        l, m1, m2 = (_bins(p, x, g.n_ap) for x in (w, w * vlos, w * vlos * vlos))
        ok = l > 0
        safe = torch.where(ok, l, torch.ones_like(l))
        V.append(m1 / safe)
        var = (m2 / safe - (m1 / safe) ** 2).clamp_min(1e-4)
        S.append(torch.where(ok, torch.sqrt(var), torch.ones_like(var)))
    Vp, sp = torch.cat(V), torch.cat(S)
    y = _observe(groups, incl, Vp, sp, pos, vel, w)
    sig, off = [], 0
    for g in groups:
        yg = y[off:off + len(g.kinds) * g.n_ap].reshape(len(g.kinds), g.n_ap)
        off += yg.numel()
        if g.geometry == "shells":
            l2 = _shell_w2(g, pos, w)
            for e in g.errs:
                sig.append(e * torch.sqrt(l2.clamp_min(1e-12) / (4 * math.pi)))
            continue
        p, _ = _aperture(g, incl, pos, vel)
        l = _bins(p, w, g.n_ap).clamp_min(2.0 / w.numel())
        for kind, e, yk in zip(g.kinds, g.errs, yg):
            if kind == "mass":
                sig.append(e * l / _areas(g))
            elif kind == "v2":
                sig.append(2 * e * torch.maximum(yk, 1e-2 * l))
            else:
                sig.append(e * l)
    sig = torch.cat(sig)
    Y = y + 0.5 * sig * _randn(gen, y.numel())
    # measured data have a few digits: rounded, they are the same whatever the order of the sums
    return tuple(t.float().double().cpu().numpy() for t in (Y, sig, Vp, sp))


def _fit_spec(case, seed, pot=None, aniso=None, stream=0):
    """Everything of one fit: descriptors, data and the initial model on the GPU."""
    pot = pot or _potential(case)
    groups = _groups(case)
    maps = case["obs"] == "maps"
    incl = 60.0 if maps else 0.0
    flat = 0.8 if pot["kind"] in ("log", "scf") else 1.0
    g = _rng(seed, 10 * stream + 1)
    target = _realise(g, 1000000 if maps else 200000, pot, flat=flat, spin=0.3 if maps else 0.0)
    Y, sig, Vp, sp = _targets(groups, incl, target, g)
    del target
    if aniso is None:
        aniso = 1.5 if case["obs"] == "c2" and pot["kind"] == "hernquist" else 1.0
    model = _realise(_rng(seed, 10 * stream + 2), case["n"], pot, aniso=aniso, flat=flat)
    return dict(potential=pot, groups=groups, incl_deg=incl, Y=Y, sig=sig, Vp=Vp, sp=sp,
                prior=_prior(case, pot, model[0], model[1]), params=_params(case)), model


def _batch_specs(case, seed):
    g = np.random.default_rng(int(seed))
    for i, n in enumerate(_batch_counts(case)):
        u = g.random(3)
        sub = dict(case, pot="nfw", obs="c2", prior="cell", n=n)
        desc, model = _fit_spec(sub, seed, _halo(1.0 + 29.0 * u[1], 2.0 + 18.0 * u[0]), 0.7 + 0.8 * u[2], stream=i + 1)
        yield desc, model


def _load(fit, model):
    pos, vel, w = (t.contiguous() for t in model)
    torch.cuda.synchronize()
    fit.load_device(w.numel(), pos.data_ptr(), vel.data_ptr(), w.data_ptr())


def _pinned(n):
    return torch.empty(n, dtype=torch.float64, pin_memory=True)


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    if case["kind"] == "batch":
        descs, models = zip(*_batch_specs(case, seed))
        batch = B.Batch(list(descs), precision=case["precision"])
        for f, m in zip(batch.fits, models):
            _load(f, m)
        n = [m[2].numel() for m in models]
        return dict(case=case, batch=batch, w=_pinned(sum(n)), off=np.concatenate([[0], np.cumsum(n)]).tolist())
    desc, model = _fit_spec(case, seed)
    if case["kind"] == "diag":  # a finished model: uneven weights
        model = (model[0], model[1], model[2] * torch.exp(0.3 * _randn(_rng(seed, 5), case["n"])))
    fit = B.Fit(precision=case["precision"], **{"potential_desc" if k == "potential" else k: v for k, v in desc.items()})
    _load(fit, model)
    state = dict(case=case, fit=fit, w=_pinned(case["n"]))
    if case["kind"] == "diag":
        state["target"] = _host_particles(_diag_target(case, seed, desc))
    return state


def _diag_target(case, seed, desc):
    return _realise(_rng(seed, 6), DIAG_TARGET, desc["potential"], flat=0.8 if desc["potential"]["kind"] == "log" else 1.0)


def _host_particles(p):
    pos, vel, w = (t.cpu().numpy() for t in p)
    return dict(x=pos[0], y=pos[1], z=pos[2], vx=vel[0], vy=vel[1], vz=vel[2], w=w)


def _read_weights(fit, out):
    """The weights into the caller's buffer, as the C interface takes it."""
    B._check(B.lib().m2m_get_weights(fit.h, C.cast(out.data_ptr(), C.POINTER(C.c_double)), out.numel()), fit.h)
    return out


def run(state):
    case = state["case"]
    mixed = case["precision"] == "mixed"
    if case["kind"] == "diag":
        fit = state["fit"]
        sums, counts = fit.diag_kinematics(SPH)
        tsums, tcounts = fit.diag_kinematics(SPH, state["target"])
        ws, wd, cells = fit.diag_grid()
        tws, twd, tcells = fit.diag_grid(None, state["target"])
        return dict(sums=sums, counts=counts, tsums=tsums, tcounts=tcounts, ws=ws, wd=wd, cells=cells, tws=tws, twd=twd,
                    tcells=tcells)
    if case["kind"] == "batch":
        batch = state["batch"]
        batch.step(case["steps"])
        chi2 = batch.chi2()
        for i, f in enumerate(batch.fits):
            _read_weights(f, state["w"][state["off"][i]:state["off"][i + 1]])
        out = dict(chi2=chi2, w=state["w"])
        return dict(chi2=chi2.astype(np.float32), w=state["w"].float()) if mixed else out
    fit = state["fit"]
    chi2 = np.zeros(case["reads"])
    for k in range(case["reads"]):
        fit.step(case["steps"])
        chi2[k] = fit.chi2()
    ytil, y = fit.observables()
    w = _read_weights(fit, state["w"])
    out = dict(chi2=chi2, ytil=ytil, y=y, w=w)
    if case["n"] <= 20001:  # small models are looked at particle by particle
        out["pos"], out["vel"] = fit.state()
    if case["pot"] == "scf":
        ups, out["coef"] = fit.scf()
        out["ups"] = float(ups)
    if mixed:
        out = {k: v.float() if isinstance(v, torch.Tensor) else np.asarray(v, np.float32) for k, v in out.items()}
    return out


# ------------------------------------------------------------------ the method in FP64, plain torch

def _bins(idx, val, n):
    """Sums of val by idx (-1: none), over spread copies of the bins."""
    rep = max(1, min(4096, (1 << 22) // (n + 1)))
    spread = torch.arange(idx.numel(), device=idx.device) % rep
    out = torch.zeros(rep * (n + 1), device=idx.device, dtype=torch.float64)
    out.index_add_(0, spread * (n + 1) + idx + 1, val)
    return out.view(rep, n + 1).sum(0)[1:]


def _areas(g):
    if g.geometry == "annuli":
        e = torch.tensor(g.edges, device=DEV)
        return math.pi * (e[1:] ** 2 - e[:-1] ** 2)
    b = g.box
    return torch.full((g.n_ap,), (b[1] - b[0]) / g.nx * ((b[3] - b[2]) / g.ny), device=DEV, dtype=torch.float64)


def _aperture(g, incl, pos, vel):
    i = math.radians(incl)
    X, Y = pos[0], pos[1] * math.cos(i) - pos[2] * math.sin(i)
    vlos = vel[1] * math.sin(i) + vel[2] * math.cos(i)
    if g.geometry == "annuli":
        e2 = torch.tensor(np.asarray(g.edges) ** 2, device=DEV)
        p = torch.bucketize(X * X + Y * Y, e2, right=True) - 1
        return torch.where(p >= g.n_ap, torch.full_like(p, -1), p), vlos
    b = g.box
    px = torch.floor((X - b[0]) * g.nx / (b[1] - b[0]))
    py = torch.floor((Y - b[2]) * g.ny / (b[3] - b[2]))
    ok = (px >= 0) & (px < g.nx) & (py >= 0) & (py < g.ny)
    return torch.where(ok, py * g.nx + px, torch.full_like(px, -1)).long(), vlos


def _hermite(nu, top):
    h = [torch.ones_like(nu), 2 * nu]
    for n in range(1, top):
        h.append(2 * nu * h[n] - 2 * n * h[n - 1])
    return h


def _gh_const(n):
    return math.sqrt(2.0 ** (1 - n) / math.factorial(n))


def _cic(g, pos):
    e = torch.tensor(np.asarray(g.edges), device=DEV)
    r = torch.sqrt((pos * pos).sum(0))
    k = torch.bucketize(r, e, right=True)  # radii at or below r
    lo, hi = (k - 1).clamp_min(0), k.clamp_max(len(e) - 1)
    d = torch.where(hi > lo, e[hi] - e[lo], torch.ones_like(r))
    g1 = torch.where((k > 0) & (k < len(e)), (r - e[lo]) / d, torch.zeros_like(r))
    g0 = torch.where(k < len(e), 1 - g1, torch.zeros_like(r))
    return lo, hi, g0, g1


def _shell_w2(g, pos, w):
    lo, hi, g0, g1 = _cic(g, pos)
    return _bins(lo, (w * g0) ** 2, g.n_ap) + _bins(hi, (w * g1) ** 2, g.n_ap)


def _ylm(lms, pos):
    """Real spherical harmonics of unit norm, without the Condon-Shortley phase."""
    x, y, z = pos
    R2 = x * x + y * y
    R, r = torch.sqrt(R2), torch.sqrt(R2 + z * z)
    ct, st = z / r, R / r
    ph = torch.atan2(y, x)
    out = []
    for l, m in lms:
        a = abs(m)
        p0 = torch.zeros_like(r)
        p1 = st ** a * float(np.prod(np.arange(1, 2 * a, 2)) if a else 1.0)
        for j in range(a + 1, l + 1):
            p0, p1 = p1, ((2 * j - 1) * ct * p1 - (j + a - 1) * p0) / (j - a)
        nrm = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - a) / math.factorial(l + a))
        if m:
            nrm *= math.sqrt(2.0)
            p1 = p1 * (torch.cos(m * ph) if m > 0 else torch.sin(a * ph))
        out.append(nrm * p1)
    return out


def _lms(g):
    return [tuple(int(v) for v in k[4:].split("_")) for k in g.kinds]


def _observe(groups, incl, Vp, sp, pos, vel, w, slopes=False):
    """y_j, or with slopes the derivatives of the kinematic kernels with respect to ln Upsilon."""
    out, a0 = [], 0
    for g in groups:
        if g.geometry == "shells":
            lo, hi, g0, g1 = _cic(g, pos)
            for Y in _ylm(_lms(g), pos):
                out.append(_bins(lo, w * g0 * Y, g.n_ap) + _bins(hi, w * g1 * Y, g.n_ap))
            a0 += g.n_ap
            continue
        p, vlos = _aperture(g, incl, pos, vel)
        V, S = Vp[a0:a0 + g.n_ap], sp[a0:a0 + g.n_ap]
        a0 += g.n_ap
        q = p.clamp_min(0)
        gh = any(k.startswith("gh") for k in g.kinds)
        if gh:
            nu = (vlos - V[q]) / S[q]
            ex = torch.exp(-0.5 * nu * nu)
            h = _hermite(nu, 6)
        for k in g.kinds:
            if k == "mass":
                out.append(torch.zeros_like(V) if slopes else _bins(p, w, g.n_ap) / _areas(g))
            elif k == "v2":
                out.append(_bins(p, w * vlos * vlos, g.n_ap))
            else:
                n = int(k[2:])
                K = _gh_const(n) * h[n] * ex
                if slopes:
                    dh = (2 * n * h[n - 1] if n else 0.0) - nu * h[n]
                    K = 0.5 * vlos * _gh_const(n) * dh * ex / S[q]
                out.append(_bins(p, w * K, g.n_ap))
    return torch.cat(out)


def _data_force(groups, incl, Vp, sp, pos, vel, c):
    """sum_j K_ij c_j of every particle (c_j with the 1/area of the surface mass in it)."""
    F, a0, j0 = torch.zeros_like(pos[0]), 0, 0
    for g in groups:
        if g.geometry == "shells":
            lo, hi, g0, g1 = _cic(g, pos)
            for Y in _ylm(_lms(g), pos):
                cj = c[j0:j0 + g.n_ap]
                F += Y * (g0 * cj[lo] + g1 * cj[hi])
                j0 += g.n_ap
            a0 += g.n_ap
            continue
        p, vlos = _aperture(g, incl, pos, vel)
        V, S = Vp[a0:a0 + g.n_ap], sp[a0:a0 + g.n_ap]
        a0 += g.n_ap
        q, inside = p.clamp_min(0), p >= 0
        f = torch.zeros_like(F)
        if any(k.startswith("gh") for k in g.kinds):
            nu = (vlos - V[q]) / S[q]
            ex = torch.exp(-0.5 * nu * nu)
            h = _hermite(nu, 6)
        for k in g.kinds:
            cj = c[j0:j0 + g.n_ap][q]
            j0 += g.n_ap
            f += cj if k == "mass" else cj * vlos * vlos if k == "v2" else cj * _gh_const(int(k[2:])) * h[int(k[2:])] * ex
        F += torch.where(inside, f, torch.zeros_like(f))
    return F


def _mu_of(q):
    s = torch.zeros_like(q)
    for k in range(14, 1, -1):
        s = s * q + (-1.0) ** k * (k - 1) / k
    return torch.where(q < 1e-2, s * q * q, torch.log1p(q) - q / (1 + q))


def _phi(pot, pos):
    x, y, z = pos
    if pot["kind"] in ("log", "scf"):
        return 0.5 * pot["v0"] ** 2 * torch.log(pot["r0"] ** 2 + x * x + y * y + z * z / pot["q"] ** 2)
    r = torch.sqrt(x * x + y * y + z * z)
    phi = -1.0 / (r + 1.0)
    return phi - pot["Ms"] * torch.log1p(r / pot["rs"]) / r if pot["kind"] == "hernquist_nfw" else phi


def _accel(pot, pos):
    x, y, z = pos
    if pot["kind"] in ("log", "scf"):
        f = -pot["v0"] ** 2 / (pot["r0"] ** 2 + x * x + y * y + z * z / pot["q"] ** 2)
        return torch.stack([f * x, f * y, f * z / pot["q"] ** 2])
    r2 = x * x + y * y + z * z
    r = torch.sqrt(r2)
    f = 1.0 / ((r + 1.0) ** 2 * r)
    if pot["kind"] == "hernquist_nfw":
        f = f + pot["Ms"] * _mu_of(r / pot["rs"]) / (r2 * r)
    return -f * pos


class _Light:
    """The potential of thin shells carrying the particles' light (the self-consistent part)."""

    def __init__(self, pot):
        self.r = torch.tensor(np.asarray(pot["scf_r"]), device=DEV)
        self.lms = [(l, m) for l in range(pot["scf_lmax"] + 1) for m in range(-l, l + 1)]
        self.ups, self.a = pot["ups"], torch.zeros(len(self.r), len(self.lms), device=DEV, dtype=torch.float64)

    def rebuild(self, pos, w):
        rr = torch.sqrt((pos * pos).sum(0))
        n = len(self.r)
        k = torch.bucketize(rr, self.r, right=True)
        lo, hi = (k - 1).clamp_min(0), k.clamp_max(n - 1)
        d = torch.where(hi > lo, self.r[hi] - self.r[lo], torch.ones_like(rr))
        g1 = torch.where((k > 0) & (k < n), (rr - self.r[lo]) / d, torch.zeros_like(rr))
        Y = _ylm(self.lms, pos)
        self.a = torch.stack([_bins(lo, w * (1 - g1) * v, n) + _bins(hi, w * g1 * v, n) for v in Y], 1)

    def phi(self, pos):
        r = torch.sqrt((pos * pos).sum(0))
        j = torch.bucketize(r.detach(), self.r, right=True)
        n, out = len(self.r), torch.zeros_like(r)
        for q, ((l, m), Y) in enumerate(zip(self.lms, _ylm(self.lms, pos))):
            zero = torch.zeros(1, device=DEV, dtype=torch.float64)
            A = torch.cat([zero, torch.cumsum(self.a[:, q] * self.r ** l, 0)])
            s = self.a[:, q] * self.r ** -(l + 1)
            Bo = torch.cat([torch.flip(torch.cumsum(torch.flip(s, [0]), 0), [0]), zero])
            rin = torch.where(j > 0, r, torch.ones_like(r))
            out = out - 4 * math.pi / (2 * l + 1) * Y * (A[j] * rin ** -(l + 1) + Bo[j] * r ** l)
        return self.ups * out

    def accel(self, pos):
        with torch.enable_grad():
            p = pos.detach().clone().requires_grad_(True)
            (g,) = torch.autograd.grad(self.phi(p).sum(), p)
        return -g


def _circular_L(pot, light, E):
    """L of the circular orbit of energy E in the equatorial plane (0 where there is none)."""
    if pot["kind"] == "hernquist":
        u = (-1 - torch.sqrt(1 - 8 * E)) / (4 * E)
        R = u - 1
        return torch.where((E < 0) & (E > -1), R * torch.sqrt(R.clamp_min(0)) / (R + 1), torch.zeros_like(E))

    def axis(R):
        z = torch.zeros_like(R)
        p = torch.stack([R, z, z])
        ax, ph = _accel(pot, p)[0], _phi(pot, p)
        if light is not None:
            p = torch.stack([R.clamp_min(1e-300), z, z])
            ax, ph = ax + torch.where(R > 0, light.accel(p)[0], z), ph + light.phi(p)
        return -R * ax, ph

    if light is None:
        lo, hi = torch.full_like(E, math.log(1e-6)), torch.full_like(E, math.log(1e8))
        for _ in range(62):
            mid = 0.5 * (lo + hi)
            v2, ph = axis(torch.exp(mid))
            up = ph + 0.5 * v2 <= E
            lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
        R = torch.exp(0.5 * (lo + hi))
        bound = E < 0 if pot["kind"] == "hernquist_nfw" else E > pot["v0"] ** 2 * math.log(pot["r0"])
    else:
        lo, hi = torch.zeros_like(E), torch.ones_like(E)
        for _ in range(50):
            v2, ph = axis(hi)
            hi = torch.where(ph + 0.5 * v2 <= E, 2 * hi, hi)
        for _ in range(60):
            mid = 0.5 * (lo + hi)
            v2, ph = axis(mid)
            up = ph + 0.5 * v2 <= E
            lo, hi = torch.where(up, mid, lo), torch.where(up, hi, mid)
        R = 0.5 * (lo + hi)
        bound = E > axis(torch.zeros(1, device=DEV, dtype=torch.float64))[1]
    v2, _ = axis(R)
    return torch.where(bound, R * torch.sqrt(v2.clamp_min(0)), torch.zeros_like(E))


def _cells(pot, light, grid, pos, vel):
    E = 0.5 * (vel * vel).sum(0) + _phi(pot, pos)
    if light is not None:
        E = E + light.phi(pos)
    Lz = pos[0] * vel[1] - pos[1] * vel[0]
    if grid["signed_lz"]:
        L, lo = Lz, -1.0
    else:
        Lx, Ly = pos[1] * vel[2] - pos[2] * vel[1], pos[2] * vel[0] - pos[0] * vel[2]
        L, lo = torch.sqrt(Lx * Lx + Ly * Ly + Lz * Lz), 0.0
    Lc = _circular_L(pot, light, E)
    x = torch.where(Lc > 0, L / torch.where(Lc > 0, Lc, torch.ones_like(Lc)), torch.zeros_like(L)).clamp(lo, 1.0)
    if grid["e_spacing"] == "logneg":
        s0, s1 = math.log(-grid["Emin"]), math.log(-grid["Emax"])
        f = torch.where(E < 0, (torch.log((-E).clamp_min(1e-300)) - s0) / (s1 - s0), torch.ones_like(E))
    elif grid["e_spacing"] == "exp":
        s0, s1 = math.exp(grid["Emin"]), math.exp(grid["Emax"])
        f = (torch.exp(E) - s0) / (s1 - s0)
    else:
        f = (E - grid["Emin"]) / (grid["Emax"] - grid["Emin"])
    k = torch.floor(f * grid["nE"]).clamp(0, grid["nE"] - 1).long()
    l = torch.floor((x - lo) / (1.0 - lo) * grid["nx"]).clamp(0, grid["nx"] - 1).long()
    return k * grid["nx"] + l


def _window_sum(v, half):
    for dim, h in enumerate(half):
        n = v.shape[dim]
        v = torch.stack([v.narrow(dim, max(0, i - h), min(n, i + h + 1) - max(0, i - h)).sum(dim) for i in range(n)], dim)
    return v


def _advance(desc, model, steps, reads=1):
    """The fit after `reads` segments of `steps` steps, in FP64."""
    pot, groups, incl, grid, par = (desc[k] for k in ("potential", "groups", "incl_deg", "prior", "params"))
    Y, sig, Vp, sp = (torch.tensor(desc[k], device=DEV) for k in ("Y", "sig", "Vp", "sp"))
    post = torch.cat([1.0 / _areas(g) if k == "mass" else torch.ones(g.n_ap, device=DEV, dtype=torch.float64)
                      for g in groups for k in g.kinds])
    pos, vel, w = (t.clone() for t in model)
    W0, n, dt = w.sum(), w.numel(), par["dt"]
    light = None
    if pot["kind"] == "scf":
        light = _Light(pot)
        light.rebuild(pos, w)
    pull = (lambda p: _accel(pot, p) + light.accel(p)) if light is not None else (lambda p: _accel(pot, p))
    ytil = _observe(groups, incl, Vp, sp, pos, vel, w)
    chi2, prior, acc = [], None, pull(pos)
    for t in range(1, steps * reads + 1):
        vel = vel + 0.5 * dt * acc
        pos = pos + dt * vel
        acc = pull(pos)
        vel = vel + 0.5 * dt * acc
        y = _observe(groups, incl, Vp, sp, pos, vel, w)
        ytil = ytil + par["alpha"] * (y - ytil)
        delta = (ytil - Y) / sig
        c2 = (delta * delta).sum()
        if t % steps == 0:
            chi2.append(c2)
        update = (t - 1) % grid["update_every"] == 0
        if update and grid["mode"] == "mpr":
            cell = _cells(pot, light, grid, pos, vel)
            nc = grid["nE"] * grid["nx"]
            cw, cn = _bins(cell, w, nc), _bins(cell, torch.ones_like(w), nc)
            if "window" in grid:
                shape = (grid["nE"], grid["nx"])
                cw, cn = (_window_sum(v.view(shape), grid["window"]).reshape(-1) for v in (cw, cn))
            prior = torch.where(cn > 0, cw / cn.clamp_min(1), torch.zeros_like(cw))[cell]
        if update and light is not None:
            if pot["eps_ups"] > 0:
                D = _observe(groups, incl, Vp, sp, pos, vel, w, slopes=True)
                light.ups *= math.exp(-pot["eps_ups"] * grid["update_every"] * dt * float((delta / sig * D).sum()))
            light.rebuild(pos, w)
            acc = pull(pos)
        data = _data_force(groups, incl, Vp, sp, pos, vel, delta / sig * post)
        dS = -torch.log(w * n / W0) - 1 if grid["mode"] == "gwr" else -torch.log(w / prior)
        h = par["eps"] * dt * (par["mu"] * dS - data)
        w = w * (1 + h) if par["update_rule"] == "euler" else w * torch.exp(h)
        w = w * (W0 / w.sum())
    return dict(chi2=torch.stack(chi2), ytil=ytil, y=y, w=w, pos=pos, vel=vel, light=light)


def _exact_diag(case, seed):
    desc, model = _fit_spec(case, seed)
    w = model[2] * torch.exp(0.3 * _randn(_rng(seed, 5), case["n"]))
    own = tuple(t.float().double() if case["precision"] == "mixed" else t for t in (model[0], model[1], w))
    out = {}
    for tag, (pos, vel, w) in (("", own), ("t", _diag_target(case, seed, desc))):
        x, y, z = pos
        R, r = torch.sqrt(x * x + y * y), torch.sqrt((pos * pos).sum(0))
        cp, sn, ct, st = x / R, y / R, z / r, R / r
        v = [vel[0] * st * cp + vel[1] * st * sn + vel[2] * ct, vel[0] * ct * cp + vel[1] * ct * sn - vel[2] * st,
             vel[1] * cp - vel[0] * sn]
        f = (torch.log(r) - math.log(SPH["r_min"])) / math.log(SPH["r_max"] / SPH["r_min"])
        ir = torch.where(r < SPH["r_min"], torch.zeros_like(r), 1 + torch.floor(f * (SPH["n_r"] - 1))).long()
        ir = ir.clamp_max(SPH["n_r"] - 1)
        ic = torch.floor((ct + 1) * 0.5 * SPH["n_ct"]).clamp(0, SPH["n_ct"] - 1).long()
        ip = torch.floor((torch.atan2(y, x) + math.pi) / (2 * math.pi) * SPH["n_phi"]).clamp(0, SPH["n_phi"] - 1).long()
        b = torch.where(r < SPH["r_max"], (ir * SPH["n_ct"] + ic) * SPH["n_phi"] + ip, torch.full_like(ir, -1))
        nb = SPH["n_r"] * SPH["n_ct"] * SPH["n_phi"]
        out[tag + "sums"] = torch.stack([_bins(b, q, nb) for q in [w] + [w * u for u in v] + [w * u * u for u in v]], 1)
        out[tag + "counts"] = None
        cell = _cells(desc["potential"], None, desc["prior"], pos, vel)
        nc = desc["prior"]["nE"] * desc["prior"]["nx"]
        ws, cn = _bins(cell, w, nc), _bins(cell, torch.ones_like(w), nc)
        out[tag + "ws"] = ws
        # the target's weights are all alike: their deviations are rounding only
        out[tag + "wd"] = None if tag else _bins(cell, (w - (ws / cn.clamp_min(1))[cell]) ** 2, nc)
        out[tag + "cells"] = None
    return out


def exact(case, seed):
    if case["kind"] == "diag":
        return _exact_diag(case, seed)
    if case["kind"] == "batch":
        if sum(_batch_counts(case)) * case["steps"] > 3e9 or case["fits"] * case["steps"] > 4000:
            return None  # tens of seconds
        got = [_advance(desc, model, case["steps"]) for desc, model in _batch_specs(case, seed)]
        return dict(chi2=torch.cat([g["chi2"] for g in got]), w=torch.cat([g["w"] for g in got]))
    desc, model = _fit_spec(case, seed)
    got = _advance(desc, model, case["steps"], case["reads"])
    out = {k: got[k] for k in ("chi2", "ytil", "y", "w")}
    if case["n"] <= 20001:
        out["pos"], out["vel"] = got["pos"], got["vel"]
    if got["light"] is not None:
        out["coef"], out["ups"] = got["light"].a, got["light"].ups
    return out
