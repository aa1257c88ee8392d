"""Calls that use the idle population buffer as scratch (contact angles, the
autotuners) leave the run as it was: the steps after them give the same bits."""
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


def _general(wl):
    wl.params.tau = 0.8
    return wl


CASES = {"2d_f64": lambda: W.small_2d("f64"), "3d_f32": lambda: W.small_3d("f32"),
         "3d_f16": lambda: W.small_sweep_3d(1, seed=4, storage="f16")[0],
         "3d_general": lambda: _general(W.small_3d("f32"))}


@pytest.mark.parametrize("name", CASES)
def test_scratch_between_steps(name):
    from paper_1906_03065_gb300 import Simulation
    a, b = Simulation(CASES[name]()).init(), Simulation(CASES[name]()).init()
    tile = (3, 8) if name == "3d_general" else (14, 8)
    for s in (a, b):
        s.set_tile(*tile)
        s.step(5)
    a.contact_angle()
    a.step(40)
    a.autotune()
    a.set_tile(*tile)
    a.contact_angle()
    assert np.array_equal(a.residual(), (b.step(40), b.residual())[1])
    a.step(6)
    b.step(6)
    assert np.array_equal(a.pops(), b.pops())
    assert np.array_equal(a.nodes(0), b.nodes(0))


def test_tau1_and_general_steps_in_turn():
    """Odd numbers of general steps move the state, and with it the tau = 1
    state, between the two buffers."""
    from paper_1906_03065_gb300 import Simulation
    a, b = (Simulation(W.small_2d("f64")).init() for _ in range(2))
    for s, cut in ((a, False), (b, True)):
        for n, tile in ((3, (14, 8)), (1, (3, 8)), (40, (14, 8)), (2, (3, 8)), (5, (14, 8)), (33, (3, 8)), (7, (14, 8))):
            s.set_tile(*tile)
            s.step(n)
            if cut:
                s.contact_angle()
                s.load(s.save())
    assert np.array_equal(a.pops(), b.pops())
    assert np.array_equal(a.nodes(0), b.nodes(0))


def test_batch_autotune_between_steps():
    from paper_1906_03065_gb300 import Batch
    wls = W.small_sweep_3d(2, seed=9, storage="f32")
    a, b = Batch(wls).init(), Batch(wls).init()
    for s in (a, b):
        s.step(3)
    a.autotune()
    a[1].contact_angle()
    for s in (a, b):
        s.step(4)
    for i in range(2):
        assert np.array_equal(a[i].field("I"), b[i].field("I"))
        assert np.abs(a[i].pops() - b[i].pops()).max() < 1e-6


def test_contact_angle_of_a_dense_ring():
    """A ring whose scratch does not fit past the state: the state moves over."""
    from paper_1906_03065_gb300 import Simulation
    wl = W.small_2d("f64", nx=24, ny=24, nodes=1200, radius=6.0, centre=(12.2, 11.9))
    wl.params.interface_pos = 12.0
    wl.membranes[0].kb = 0.0
    a, b = Simulation(wl).init(), Simulation(wl).init()
    for s in (a, b):
        s.step(3)
    assert a.contact_angle()[0, 3] == 2
    for s in (a, b):
        s.step(4)
    assert np.array_equal(a.pops(), b.pops())
    assert np.array_equal(a.nodes(0), b.nodes(0))
    assert np.isfinite(a.pops()).all()
