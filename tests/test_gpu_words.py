"""FP64 sums beyond 2^53 units (weights grown by more than 2^15 in a step, within the range): the
sums' integer and fraction words depend on how the particles are shared out over blocks, their
value does not. Every deposit and launch shape gives the same bits."""
import math

import numpy as np
import pytest

from paper_1202_2355_gb300 import binding as B
from paper_1202_2355_gb300 import workloads as W
from paper_1202_2355_gb300.workloads import Group

pytestmark = pytest.mark.gpu

GROUPS = [Group("pixels", ["mass", "v2", "gh2", "gh4"], [1.0] * 4, nx=3, ny=3, box=(-2.0, 2.0, -2.0, 2.0))]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1202_2355_gb300 import build
    build.build()


def _read(f):
    c2, d = f.chi2(with_delta=True)
    yt, y = f.observables()
    return yt, y, d, np.array([c2]), f.weights()


def test_sums_beyond_53_bits():
    n, dt = 30_011, 0.01
    wl = W.make("c1", n=n, n_target=10)
    args = dict(prior=dict(wl.prior, mode="gwr"), par=dict(wl.params, dt=dt, mu=0.0, alpha=1.0, renormalize=1,
                                                             update_rule="exp", n_relax=0))

    def fit(Y, sig, eps, **kw):
        f = B.Fit(wl.potential, GROUPS, 0.0, Y, sig, np.zeros(9), np.ones(9), args["prior"], dict(args["par"], eps=eps),
                  "fp64", **kw)
        f.load(wl.model)
        return f

    probe = fit(np.ones(36), np.ones(36), 0.0)
    _, y = probe.observables()
    probe.close()
    # Delta = -1 on the surface masses: the weights in pixel p grow by exp(eps dt / W_p), the most in
    # the lightest pixel, by 10^7
    Y, sig = y.copy(), np.full(36, 1e30)
    Y[:9] *= 2.0
    sig[:9] = y[:9]
    wp = y[:9] * (4.0 / 3.0) ** 2
    eps = math.log(1e7) / dt * wp.min()
    want = None
    for kw in (dict(deposit="shared"), dict(deposit="shared", block=32), dict(deposit="shared", block=96, blocks_per_sm=1),
               dict(deposit="global"), dict(deposit="global", block=64)):
        for steps in ([1, 1], [2]):
            f = fit(Y, sig, eps, **kw)
            for k in steps:
                f.step(k)
            got = _read(f)
            f.close()
            if want is None:
                want = got
                assert want[1].max() > 0 and np.all(np.isfinite(want[1]))
            for a, b in zip(got, want):
                assert np.array_equal(a, b), (kw, steps)
