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
