"""The step at the sizes where its launch and finalize change: particle counts around a warp,
a block and a full wave of blocks (the particles are shared out in whole warps), and
observable sets of 16 and 17 chunks of apertures (the finalize runs in the last block of the
step kernel up to 16 chunks and over several blocks beyond). FP64 within 1e-10 of the oracle."""
import math

import numpy as np
import pytest

import oracle as O
from paper_1202_2355_gb300 import workloads as W
from paper_1202_2355_gb300.workloads import Group

from _common import Pair, obs_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1202_2355_gb300 import build
    build.build()
    O.build()


def _edges(n):
    return np.exp(np.linspace(math.log(0.05), math.log(20.0), n + 1))


def _check(wl, targets, steps=12, **kw):
    pr = Pair(wl, prior=dict(wl.prior, update_every=5), targets=targets, precision="fp64", **kw)
    pr.step(steps)
    e = pr.errors()
    assert e["ytil"] < 1e-10 and e["yraw"] < 1e-10 and e["w"] < 1e-10, e
    pr.close()


@pytest.fixture(scope="module")
def c1_targets():
    return O.from_workload(W.make("c1", n=16, n_target=100_000))


@pytest.mark.parametrize("n", [1, 31, 33, 257, 4863, 4865, 38911, 38913])
def test_particle_counts(c1_targets, n):
    wl = W.make("c1", n=n, n_target=10)
    wl.params = dict(wl.params, eps=1e-5)
    _check(wl, c1_targets)


@pytest.mark.parametrize("n_ap", [32 * 14, 32 * 14 + 1])
def test_chunks_of_the_finalize(n_ap):
    # mass in n_ap annuli (14 or 15 chunks) and v2, h4 in 15 (2 chunks): 16 and 17 chunks
    wl = W.make("c1", n=3000, n_target=200_000)
    wl.groups = [Group("annuli", ["mass"], [0.05], edges=_edges(n_ap)), wl.groups[1]]
    wl.params = dict(wl.params, eps=1e-6)
    _check(wl, O.from_workload(wl))


def _same(a, b):
    for u, v in zip(a, b):
        assert np.array_equal(u, v)


def _read(f):
    yt, y = f.observables()
    pos, vel = f.state()
    g, cnt, cells = f.priors()
    return yt, y, f.weights(), pos, vel, g, cnt, cells, np.array([f.chi2(), f.step_count()])


CASES = {
    "c1": dict(wl="c1", n=3001),
    "c1_mixed": dict(wl="c1", n=40_001, precision="mixed"),
    "window": dict(wl="c2", n=20_000, prior=dict(nE=90, nx=30, window=(1, 1), update_every=7), precision="mixed"),
    "every_step": dict(wl="c2", n=5000, prior=dict(update_every=1)),
    "gwr_euler_relax": dict(wl="c1", n=700, prior=dict(mode="gwr"), params=dict(update_rule="euler", n_relax=9, eps=1e-5)),
    "nfw": dict(wl="c3", n=2500, precision="fp64", params=dict(eps=1e-5)),
    "one": dict(wl="c1", n=1, params=dict(eps=1e-6)),
    "wide_block": dict(wl="c1", n=9000, kw=dict(block=64, blocks_per_sm=1)),
}


def _fit(case, targets):
    from paper_1202_2355_gb300 import binding as B
    wl = W.make(case["wl"], n=case["n"], n_target=100_000)
    obs, Y, sig = targets(case["wl"])
    f = B.fit_from_workload(wl, Y, sig, obs.Vp, obs.sp, precision=case.get("precision", "fp64"),
                            prior=dict(wl.prior, **dict(dict(update_every=5), **case.get("prior", {}))),
                            params=dict(wl.params, **dict(dict(eps=1e-4), **case.get("params", {}))), **case.get("kw", {}))
    f.load(wl.model)
    return f


@pytest.fixture(scope="module")
def targets():
    made = {}

    def get(name):
        if name not in made:
            made[name] = O.from_workload(W.make(name, n=16, n_target=100_000))
        return made[name]
    return get


@pytest.mark.parametrize("name", sorted(CASES))
def test_many_steps_per_launch_are_the_same_steps(name, targets):
    """step(k) runs k steps in one launch, step(1) a launch and a finalize per step: the same
    bits, in any mixture, and with two fits taking turns on their own streams."""
    one, many, other = (_fit(CASES[name], targets) for _ in range(3))
    for _ in range(83):
        one.step(1)
    for k in (2, 1, 70, 10):
        many.step(k)
        other.step(k)
    _same(_read(one), _read(many))
    _same(_read(one), _read(other))
    for f in (one, many, other):
        f.close()


@pytest.mark.parametrize("grid", [dict(n_r=21, n_phi=8, n_ct=4, r_min=0.05, r_max=20.0),   # sums of a block in shared memory
                                  dict(n_r=30, n_phi=12, n_ct=12, r_min=1e-3, r_max=1e3),  # beyond it
                                  dict(n_r=2, n_phi=1, n_ct=1, r_min=1.0, r_max=1.0 + 1e-6)])
def test_kinematic_bins_beside_their_edges(grid, targets):
    """Counts and sums of 20,000 particles and of points 1e-9 to either side of every kind of bin
    edge, where FP32 cannot decide: the oracle's."""
    from paper_1202_2355_gb300 import synth
    p = synth.realise_spherical(3, 20_000, W.hernquist_sigma2)
    r_edges = np.concatenate([[grid["r_min"]], np.exp(np.linspace(math.log(grid["r_min"]), math.log(grid["r_max"]), grid["n_r"]))])
    rng = np.random.default_rng(5)
    ext = {k: [] for k in p}
    for side in (1 - 1e-9, 1 + 1e-9):
        for r in r_edges * side:
            for _ in range(3):
                d = rng.normal(size=3)
                d *= r / np.linalg.norm(d)
                for k, v in zip("xyz", d):
                    ext[k].append(v)
        for i in range(grid["n_phi"]):
            ph, z = (-math.pi + 2 * math.pi * (i + 0.5 * (side - 1)) / grid["n_phi"]) * 1.0 + (side - 1), rng.normal()
            for k, v in zip("xyz", (0.3 * math.cos(ph), 0.3 * math.sin(ph), z)):
                ext[k].append(v)
        for i in range(1, grid["n_ct"]):
            ct = -1 + 2 * i / grid["n_ct"] + (side - 1)
            for k, v in zip("xyz", (0.5 * math.sqrt(1 - ct * ct), 0.1 * side, 0.51 * ct / max(1e-9, 1.0))):
                ext[k].append(v)
    m = len(ext["x"])
    for k in ("vx", "vy", "vz"):
        ext[k] = list(rng.normal(size=m))
    ext["w"] = [1e-5] * m
    q = {k: np.concatenate([p[k], np.asarray(ext[k])]) for k in p}
    f = _fit(dict(wl="c1", n=10), targets)
    s, c = f.diag_kinematics(grid, particles=q)
    so, co = O.kin_sums(grid, O.ParticleSet(q))
    f.close()
    assert np.array_equal(c, co)
    assert np.all(np.abs(s - so) <= 1e-12 * (np.abs(so).max(axis=0) + 1e-300))


def test_steps_under_capture(targets):
    """Steps captured into a graph on the caller's stream, replayed: the same steps."""
    import torch
    st = torch.cuda.Stream()
    case = dict(CASES["c1"], kw=dict(stream=st.cuda_stream))
    a, b = _fit(case, targets), _fit(CASES["c1"], targets)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        a.step(3)
    with torch.cuda.stream(st):
        g.replay()
        g.replay()
    b.step(6)
    _same(_read(a), _read(b))
    a.close()
    b.close()


def test_fits_of_several_threads_take_turns(targets):
    """Two threads step their own fits at the same time: the same bits as alone."""
    import threading
    names = ["c1", "nfw"]
    alone = []
    for n in names:
        f = _fit(CASES[n], targets)
        f.step(200)
        alone.append(_read(f))
        f.close()
    fits = [_fit(CASES[n], targets) for n in names]
    ts = [threading.Thread(target=lambda f=f: [f.step(20) for _ in range(10)]) for f in fits]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for f, want in zip(fits, alone):
        _same(_read(f), want)
        f.close()
