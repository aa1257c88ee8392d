"""Steps captured by the caller into a CUDA graph of its own.  Every replay
continues from the state it finds: replays equal direct steps bit for bit,
whether the state was in the populations or in the 12 stored values per cell
when the call was captured, and with direct steps, reads, loads and writes
between the replays.  A capture by itself changes nothing."""
import numpy as np
import pytest

from paper_1906_03065_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1906_03065_gb300 import build
    build.build()


def _bare(wl):
    wl.membranes = []
    return wl


def _general(wl):
    wl.params.tau = 0.8
    return wl


CASES = {
    "2d_f64": lambda: W.small_2d("f64"),
    "3d_f32": lambda: W.small_3d("f32"),
    "3d_f16": lambda: W.small_sweep_3d(1, seed=4, storage="f16")[0],
    "3d_f32_general": lambda: _general(W.small_3d("f32")),
    "3d_f32_bare": lambda: _bare(W.small_3d("f32")),
    "3d_bf16_bare": lambda: _bare(W.small_3d("bf16")),
}


def _sim(wl):
    import torch
    from paper_1906_03065_gb300 import Simulation
    return Simulation(wl, stream=torch.cuda.Stream())


def _start(s):
    C0, u0 = W.random_fields(s.p, seed=5)
    return s.init(C0, u0)


def _captured(s, n):
    import torch
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s.stream):
        s.step(n)
    return g


def _replay(s, g, times):
    import torch
    with torch.cuda.stream(s.stream):
        for _ in range(times):
            g.replay()


def _same(a, b):
    assert np.array_equal(a.pops(), b.pops())
    assert np.array_equal(a.field("I"), b.field("I"))
    for m in range(a.n_mem):
        assert np.array_equal(a.nodes(m), b.nodes(m))


@pytest.mark.parametrize("name", CASES)
def test_replays_equal_direct_steps(name):
    a, b = _start(_sim(CASES[name]())), _start(_sim(CASES[name]()))
    g = _captured(a, 2)
    _replay(a, g, 5)
    b.step(10)
    _same(a, b)


@pytest.mark.parametrize("name", CASES)
def test_a_capture_alone_changes_nothing(name):
    a, b = _start(_sim(CASES[name]())), _start(_sim(CASES[name]()))
    g = _captured(a, 2)
    _same(a, b)
    a.step(40)
    b.step(40)
    _same(a, b)
    del g


@pytest.mark.parametrize("name", CASES)
def test_replays_among_other_calls(name):
    """A capture after earlier steps, and replays between direct steps, reads,
    a restored checkpoint, written populations, markers set from outside and a
    new start."""
    a, b = _start(_sim(CASES[name]())), _start(_sim(CASES[name]()))
    a.step(4)
    b.step(4)
    blob = b.save()
    g = _captured(a, 4)

    def both(n):
        _replay(a, g, n)
        b.step(4 * n)

    both(2)
    _same(a, b)
    a.step(2)
    b.step(2)
    both(1)
    a.step(40)
    b.step(40)
    both(1)
    P = b.pops()
    for s in (a, b):
        s.load(blob)
    both(2)
    _same(a, b)
    for s in (a, b):
        s.set_pops(P)
        for m in range(s.n_mem):
            s.set_nodes(m, s.nodes(m) + 0.37)
    both(2)
    _same(a, b)
    for s in (a, b):
        _start(s)
    both(2)
    a.step(1)
    b.step(1)
    _same(a, b)


def test_replays_between_collide_variants():
    """At tau = 1 the caller may go over to the general collide, which keeps
    the populations, and back."""
    a, b = _start(_sim(W.small_3d("f32"))), _start(_sim(W.small_3d("f32")))
    g = _captured(a, 2)
    _replay(a, g, 2)
    b.step(4)
    for s in (a, b):
        s.set_tile(3, 8)
        s.step(2)
    _replay(a, g, 1)  # (captured with the default variant)
    b.set_tile(14, 8)
    b.step(2)
    _same(a, b)


def test_batch_calls_are_refused_in_a_capture():
    """A batch uploads its argument tables in each call, which no graph can
    hold: the calls are refused before anything is enqueued."""
    import torch
    from paper_1906_03065_gb300 import Batch, TLBError
    wls = W.small_sweep_3d(2, seed=9, storage="f32")
    s = torch.cuda.Stream()
    a, b = Batch(wls, stream=s).init(), Batch(wls).init()
    a.step(3)
    b.step(3)
    g = torch.cuda.CUDAGraph()
    x = torch.zeros(4, device="cuda")
    with torch.cuda.graph(g, stream=s):
        x += 1
        for call in (lambda: a.step(2), lambda: a.profile(2), a.autotune, lambda: a.run(4, 2, 0.0)):
            with pytest.raises(TLBError, match="captur"):
                call()
    a.step(4)
    b.step(4)
    for i in range(2):
        assert np.array_equal(a[i].pops(), b[i].pops()), i


def test_batch_steps_after_captured_steps_of_an_instance():
    import torch
    from paper_1906_03065_gb300 import Batch
    wls = W.small_sweep_3d(2, seed=9, storage="f32")
    a, b = Batch(wls, stream=torch.cuda.Stream()).init(), Batch(wls).init()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=a.stream):
        a[1].step(2)
    _replay(a, g, 2)
    b[1].step(4)
    a.step(3)
    b.step(3)
    _replay(a, g, 1)
    b[1].step(2)
    a.step(2)
    b.step(2)
    for i in range(2):
        assert np.array_equal(a[i].pops(), b[i].pops()), i
