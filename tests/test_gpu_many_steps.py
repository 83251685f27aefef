"""Several steps per launch where the finalize takes most room beside the block's sums: single
apertures, each of them a chunk of its own, and no prior grid. step(k) gives the bits of k
times step(1)."""
import numpy as np
import pytest

import oracle as O
from paper_1202_2355_gb300 import binding as B
from paper_1202_2355_gb300 import workloads as W
from paper_1202_2355_gb300.workloads import Group

from test_gpu_step_shapes import _read, _same

pytestmark = pytest.mark.gpu

KINDS = ["mass", "v2", "gh0", "gh1", "gh2", "gh3", "gh4", "gh5", "gh6"]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1202_2355_gb300 import build
    build.build()
    O.build()


def _pixel(k):
    return [Group("pixels", KINDS[:k], [0.05] * k, nx=1, ny=1, box=(-3.0, 3.0, -3.0, 3.0))]


def _annuli(*kinds):
    return [Group("annuli", k, [0.05] * len(k), edges=np.array([0.05, 2.0 + i])) for i, k in enumerate(kinds)]


SETS = {"pixel6": _pixel(6), "pixel7": _pixel(7), "pixel8": _pixel(8), "pixel9": _pixel(9),
        "annuli44": _annuli(["mass", "v2", "gh3", "gh4"], ["mass", "v2", "gh3", "gh4"]),
        "annuli25": _annuli(["mass", "v2"], ["mass", "gh1", "gh2", "gh3", "gh4"])}


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("name", sorted(SETS))
def test_single_apertures(name, precision):
    wl = W.make("c1", n=3001, n_target=100_000)
    wl.groups = SETS[name]
    obs, Y, sig = O.from_workload(wl)
    fits = [B.fit_from_workload(wl, Y, sig, obs.Vp, obs.sp, precision=precision, prior=dict(wl.prior, mode="gwr"),
                                params=dict(wl.params, eps=1e-4)) for _ in range(2)]
    for f in fits:
        f.load(wl.model)
    for _ in range(40):
        fits[0].step(1)
    fits[1].step(40)
    _same(_read(fits[0]), _read(fits[1]))
    for f in fits:
        f.close()
