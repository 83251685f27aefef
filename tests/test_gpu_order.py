"""Restored states are complete before the fit's stream uses them: a fit alternates between
two saved states and steps at once after each load, and gives the bits of the uninterrupted
run, with its own stream and with the caller's."""
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


@pytest.mark.parametrize("stream", [False, True])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_restored_states_step_at_once(precision, stream, tmp_path):
    import torch
    wl = W.make("c2", n=30_001, n_target=100_000)
    obs, Y, sig = O.from_workload(wl)
    st = torch.cuda.Stream()
    prior = dict(wl.prior, nE=90, nx=30, update_every=7)

    def fit():
        f = B.fit_from_workload(wl, Y, sig, obs.Vp, obs.sp, precision=precision, prior=prior,
                                params=dict(wl.params, eps=1e-5), stream=st.cuda_stream if stream else None)
        f.load(wl.model)
        return f

    a, b = fit(), fit()
    paths, want = [], []
    for k in (5, 9):
        a.step(k)
        paths.append(str(tmp_path / f"{k}.m2m"))
        a.save(paths[-1])
        ref = fit()
        ref.step(k if k == 5 else 14)
        ref.step(3)
        want.append(_read(ref))
        ref.close()
    for i in range(12):
        b.restore(paths[i % 2])
        b.step(3 if i % 4 < 2 else 1)
        if i % 4 >= 2:
            b.step(2)
        _same(_read(b), want[i % 2])
    a.close()
    b.close()
