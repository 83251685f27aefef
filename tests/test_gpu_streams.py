"""Fits on streams of their own do not wait for one another."""
import pytest

import oracle as O

from test_gpu_step_shapes import CASES, _fit, _read, _same, targets  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1202_2355_gb300 import build
    build.build()
    O.build()


def test_a_held_stream_holds_only_its_own_fit(targets):  # noqa: F811
    """The first fit's stream is kept busy for a second (a bounded spin); the steps and chi^2 of
    the second come through meanwhile, and both are the steps they would be alone."""
    import torch
    st = torch.cuda.Stream()
    case = dict(CASES["c1"], kw=dict(stream=st.cuda_stream))
    a, b, alone = _fit(case, targets), _fit(CASES["c1"], targets), _fit(CASES["c1"], targets)
    for k in (3, 20, 70):
        alone.step(k)
    want = _read(alone)
    done = torch.cuda.Event()
    for f in (a, b):
        f.step(3)
        f.synchronize()
    with torch.cuda.stream(st):
        torch.cuda._sleep(2_000_000_000)
    a.step(20)
    done.record(st)
    b.step(20)
    b.chi2()
    assert not done.query()
    a.step(70)
    b.step(70)
    _same(_read(b), want)
    _same(_read(a), want)
    for f in (a, b, alone):
        f.close()


def test_interleaved_fits_of_one_thread(targets):  # noqa: F811
    """Four fits stepped in turn without a wait between them, their work on the GPU at once."""
    names = ["c1", "nfw", "c1_mixed", "gwr_euler_relax"]
    alone = []
    for n in names:
        f = _fit(CASES[n], targets)
        f.step(150)
        alone.append(_read(f))
        f.close()
    fits = [_fit(CASES[n], targets) for n in names]
    for k in (2, 40, 1, 64, 43):
        for f in fits:
            f.step(k)
    for f, want in zip(fits, alone):
        _same(_read(f), want)
        f.close()


def test_steps_while_another_thread_captures(targets):  # noqa: F811
    """Two fits step in turn while another thread holds a capture in the global mode open."""
    import threading
    import torch
    fits = [_fit(CASES["c1"], targets) for _ in range(2)]
    alone = _fit(CASES["c1"], targets)
    alone.step(90)
    opened, close, out = threading.Event(), threading.Event(), []

    def capture():
        g = torch.cuda.CUDAGraph()
        x = torch.zeros(8, device="cuda")
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=torch.cuda.Stream(), capture_error_mode="global"):
            x += 1
            opened.set()
            close.wait(20)
        g.replay()
        torch.cuda.synchronize()
        out.append(float(x[0]))

    t = threading.Thread(target=capture)
    t.start()
    assert opened.wait(20)
    try:
        for _ in range(3):
            for f in fits:
                f.step(30)
    finally:
        close.set()
        t.join()
    assert out == [1.0]
    for f in fits:
        _same(_read(f), _read(alone))
        f.close()
    alone.close()
