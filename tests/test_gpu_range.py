"""A weight beyond the range of the fixed-point sums (2^24 times the loaded total in FP64, 2^12
in mixed precision) is reported as an overflow, however large it is: its words have wrapped
and the other particles' sums with them.

Two particles far from the centre on slow orbits, the first in the only pixel: with the target
at twice the surface density and an error of once it, Delta = -1 and the force of change without
entropy is 1/W0, so the weight grows by exp(eps dt) at the start of the second step."""
import math

import numpy as np
import pytest

from paper_1202_2355_gb300 import binding as B
from paper_1202_2355_gb300 import workloads as W
from paper_1202_2355_gb300.workloads import Group

pytestmark = pytest.mark.gpu

GROUPS = [Group("pixels", ["mass"], [1.0], nx=1, ny=1, box=(0.0, 50.0, -50.0, 50.0))]
AREA = 5000.0
DT = 0.01


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1202_2355_gb300 import build
    build.build()


def _particles(w):
    z = np.zeros(2)
    return dict(x=np.array([25.0, -25.0]), y=z, z=z, vx=z, vy=np.array([0.1, 0.1]), vz=z, w=np.array([w, 1e-3 * w]))


def _desc(growth, w):
    wl = W.make("c1", n=16, n_target=10)
    return dict(potential=wl.potential, groups=GROUPS, incl_deg=0.0, Y=np.array([2.0 * w / AREA]),
                sig=np.array([w / AREA]), Vp=np.zeros(1), sp=np.ones(1), prior=dict(wl.prior, mode="gwr"),
                params=dict(wl.params, dt=DT, eps=math.log(growth) / DT * w, mu=0.0, alpha=1.0, renormalize=1,
                            update_rule="exp", n_relax=0))


def _fit(d, precision):
    return B.Fit(d["potential"], *(d[k] for k in ("groups", "incl_deg", "Y", "sig", "Vp", "sp", "prior", "params")),
                 precision)


def _status(f):
    try:
        f.synchronize()
    except B.M2MError as e:
        return str(e)
    return "ok"


RANGE = {"fp64": 2.0 ** 24, "mixed": 2.0 ** 12}
GROWTH = {"fp64": [1e8, 1e9, 1e10, 1e15, 1e25, 1e30, 1e100, 1e300], "mixed": [1e4, 1e6, 1e10, 1e20, 1e30]}


def _cases():
    return [pytest.param(p, g, id=f"{p}-{g:g}") for p in RANGE for g in GROWTH[p]]


@pytest.mark.parametrize("precision,growth", _cases())
@pytest.mark.parametrize("steps", [[1, 1], [2], [1, 16]])
def test_overflow_is_reported(precision, growth, steps):
    w = 0.7
    f = _fit(_desc(growth, w), precision)
    f.load(_particles(w))
    for k in steps:
        f.step(k)
    assert "OVERFLOW" in _status(f)
    f.close()


@pytest.mark.parametrize("precision", sorted(RANGE))
def test_growth_inside_the_range(precision):
    w, growth = 0.7, RANGE[precision] / 4
    f = _fit(_desc(growth, w), precision)
    f.load(_particles(w))
    f.step(2)
    assert _status(f) == "ok"
    f.close()


@pytest.mark.parametrize("precision,growth", _cases())
def test_overflow_of_one_fit_of_a_batch(precision, growth):
    w = 0.7
    b = B.Batch([_desc(1.0, w), _desc(growth, w)], precision=precision)
    for f in b.fits:
        f.load(_particles(w))
    b.step(2)
    assert _status(b.fit(0)) == "ok" and "OVERFLOW" in _status(b.fit(1))
    b.close()


@pytest.mark.parametrize("precision,growth", [("fp64", 1e30), ("fp64", 1e300), ("mixed", 1e30)])
def test_overflow_of_one_shard_reaches_every_shard(precision, growth):
    """The shards' range words are added between the pass and the finalize: the shard whose own
    particles are in range reports the overflow too."""
    import torch
    from paper_1202_2355_gb300 import dist as D
    w = 0.7
    p = _particles(w)
    fits = [_fit(_desc(growth, w), precision) for _ in range(2)]
    parts = [{k: v[i:i + 1].copy() for k, v in p.items()} for i in range(2)]
    bounds = [f.shard_bounds(q) for f, q in zip(fits, parts)]

    def exchange():
        words = [torch.as_tensor(D._DeviceWords(*f.shard_exchange()), device="cuda") for f in fits]
        for f in fits:
            try:
                f.synchronize()
            except B.M2MError:  # the shard of the large weight may know by itself
                pass
        total = torch.stack(words).sum(0)
        for v in words:
            v.copy_(total)
        torch.cuda.synchronize()

    for f, q in zip(fits, parts):
        f.shard_set(2, sum(b[0] for b in bounds), max(b[1] for b in bounds))
        f.load(q)
    exchange()
    for f in fits:
        f.step_end()
    for _ in range(2):
        for f in fits:
            f.step_begin()
        exchange()
        for f in fits:
            f.step_end()
    assert all("OVERFLOW" in _status(f) for f in fits)
    for f in fits:
        f.close()
