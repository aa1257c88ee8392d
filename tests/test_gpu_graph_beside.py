"""Steps of a context while the program captures another stream (as PyTorch
captures a training step): the library's own capture keeps out of it."""
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


@pytest.mark.parametrize("name", ["3d_f32", "2d_f64"])
def test_steps_beside_a_capture_of_another_stream(name):
    import torch
    from paper_1906_03065_gb300 import Simulation
    wl = {"3d_f32": lambda: W.small_3d("f32"), "2d_f64": lambda: W.small_2d("f64")}[name]()
    s, other = torch.cuda.Stream(), torch.cuda.Stream()
    a, b = Simulation(wl, stream=s).init(), Simulation(wl).init()
    b.set_graphs(False)
    x = torch.zeros(8, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=other):
        x += 1
        a.step(70)
        a.set_tile(16, 5)
        a.step(40)
        x += 1
    b.step(70)
    b.set_tile(16, 5)
    b.step(40)
    assert np.array_equal(a.pops(), b.pops())
    assert np.array_equal(a.nodes(0), b.nodes(0))
    g.replay()
    torch.cuda.synchronize()
    assert float(x[0]) == 2.0
