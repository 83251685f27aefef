"""Fits whose kernels are the same and whose shared memory is not: one created, or diagnosed
by another thread, later and smaller takes nothing from the larger one."""
import threading

import numpy as np
import pytest

import oracle as O
from paper_1202_2355_gb300 import binding as B
from paper_1202_2355_gb300 import workloads as W

from test_gpu_step_shapes import _read, _same

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1202_2355_gb300 import build
    build.build()
    O.build()


def _desc(big, precision):
    wl = W.make("c1", n=2000, n_target=20_000)
    obs, Y, sig = O.from_workload(wl)
    prior = dict(wl.prior, nE=110 if big else 5, nx=30 if big else 5, update_every=5)
    return wl, dict(potential=wl.potential, groups=wl.groups, incl_deg=wl.incl_deg, Y=Y, sig=sig, Vp=obs.Vp, sp=obs.sp,
                    prior=prior, params=dict(wl.params, eps=1e-5))


def _fit(d, precision, **kw):
    return B.Fit(d["potential"], *(d[k] for k in ("groups", "incl_deg", "Y", "sig", "Vp", "sp", "prior", "params")),
                 precision, **kw)


@pytest.mark.parametrize("deposit", ["shared", "global"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_a_smaller_fit_created_later(precision, deposit):
    wl, big = _desc(True, precision)
    _, small = _desc(False, precision)
    alone = _fit(big, precision, deposit=deposit)
    alone.load(wl.model)
    for k in (1, 12):
        alone.step(k)
    want = _read(alone)
    a = _fit(big, precision, deposit=deposit)
    b = _fit(small, precision, deposit=deposit)
    for f in (a, b):
        f.load(wl.model)
        for k in (1, 12):
            f.step(k)
    _same(_read(a), want)
    for f in (a, b, alone):
        f.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_a_smaller_batch_created_later(precision):
    wl, big = _desc(True, precision)
    _, small = _desc(False, precision)
    a, b = B.Batch([big, small], precision=precision), B.Batch([small], precision=precision)
    one = _fit(big, precision)
    one.load(wl.model)
    one.step(4)
    for g in (a, b):
        for f in g.fits:
            f.load(wl.model)
        g.step(4)
    _same(_read(a.fit(0)), _read(one))
    for g in (a, b, one):
        g.close()


def test_diagnostics_of_two_threads():
    """Spherical grids of 2,520 and 8 bins (the first needs more than the default 48 KB) by turns."""
    wl, d = _desc(False, "fp64")
    grids = [dict(n_r=35, n_phi=9, n_ct=8, r_min=0.05, r_max=20.0), dict(n_r=2, n_phi=2, n_ct=2, r_min=0.05, r_max=20.0)]
    want = [O.kin_sums(g, O.ParticleSet(wl.model)) for g in grids]
    bad = []

    def work(g, w):
        f = _fit(d, "fp64")
        f.load(wl.model)
        try:
            for _ in range(200):
                s, c = f.diag_kinematics(g)
                if not (np.array_equal(c, w[1]) and np.all(np.abs(s - w[0]) <= 1e-12 * (np.abs(w[0]).max(axis=0) + 1e-300))):
                    bad.append("sums")
        except B.M2MError as e:
            bad.append(str(e))
        f.close()

    ts = [threading.Thread(target=work, args=a) for a in zip(grids, want)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad, bad[:3]
