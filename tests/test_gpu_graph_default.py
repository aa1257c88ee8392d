"""The default rule for step graphs (calls long enough to pay for a capture)
changes no bits: runs in calls of any length equal those with graphs off."""
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


def _general(n):
    wl = W.capsule_3d("f32", n=n, level=2, radius=9.0)
    wl.params.tau = wl.params.tau_phi = wl.params.tau_psi = 0.8
    return wl


CASES = {"2d_f64": lambda: W.small_2d("f64"), "3d_f32": lambda: W.small_3d("f32"),
         "3d_f16": lambda: W.small_sweep_3d(1, seed=4, storage="f16")[0],
         "3d_general": lambda: _general(48), "3d_general_large": lambda: _general(128)}


@pytest.mark.parametrize("name", CASES)
def test_default_calls_equal_direct_launches(name):
    from paper_1906_03065_gb300 import Simulation
    runs = []
    for off in (False, True):
        s = Simulation(CASES[name]()).init()
        if off:
            s.set_graphs(False)
        for n in (8, 31, 32, 7, 33, 64, 9, 71, 8):
            s.step(n)
        s.set_nodes(0, s.nodes(0) + 0.2)
        s.step(40)
        runs.append((s.field("C1"), s.field("C3"), s.field("u"), s.nodes(0)))
    for x, y in zip(*runs):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("storage,tau", [("f32", 1.0), ("bf16", 1.0), ("f32", 0.8)])
def test_graphs_asked_for_without_membranes(storage, tau):
    from paper_1906_03065_gb300 import Simulation
    p = W.Params(dim=3, nx=33, ny=20, nz=18, wall_last=1, storage=storage, alpha=1.0, interface_pos=9.0, tau=tau)
    C0, u0 = W.random_fields(p, seed=2)
    runs = []
    for on in (False, True):
        s = Simulation(W.Workload("fluid", p, [])).init(C0, u0)
        s.set_graphs(on)
        for n in (8, 9, 40, 3, 16):
            s.step(n)
        s.set_pops(s.pops())
        s.step(17)
        runs.append((s.launches(), s.pops()))
    assert runs[0][0] == runs[1][0]
    assert np.array_equal(runs[0][1], runs[1][1])
