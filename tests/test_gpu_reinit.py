"""A context that has taken steps starts again: tlb_init_fields replaces its
state whatever was read in between, so the steps after it equal those of a
fresh context, bit for bit."""
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


def _cases():
    general = W.small_3d("f32")
    general.params.tau = 0.8
    return [W.small_2d("f64"), W.small_3d("f32"), W.small_sweep_3d(1, seed=4, storage="f16")[0], general]


@pytest.mark.parametrize("wl", _cases(), ids=["2d_f64", "3d_f32", "3d_f16", "3d_f32_general"])
@pytest.mark.parametrize("read", [False, True])
def test_init_after_steps_starts_again(wl, read):
    from paper_1906_03065_gb300 import Simulation
    C0, u0 = W.random_fields(wl.params, seed=3)
    a, b = Simulation(wl).init(), Simulation(wl).init(C0, u0)
    X0 = a.nodes(0)
    a.step(6)
    if read:
        a.pops()
    a.set_nodes(0, X0)
    a.init(C0, u0)
    ra, rb = a.residual(), b.residual()
    assert np.array_equal(ra, rb)
    assert np.array_equal(a.pops(), b.pops())
    a.step(5)
    b.step(5)
    assert np.array_equal(a.pops(), b.pops())
    assert np.array_equal(a.nodes(0), b.nodes(0))


def test_batch_instances_start_again():
    from paper_1906_03065_gb300 import Batch
    wls = [W.small_2d("f64"), W.small_2d("f64", nx=44, ny=40, centre=(21.1, 19.7))]
    a, b = Batch(wls).init(), Batch(wls).init()
    X0 = [a[i].nodes(0) for i in range(2)]
    a.step(6)
    for i in range(2):
        a[i].set_nodes(0, X0[i])
    a.init()
    a.step(5)
    b.step(5)
    for i in range(2):
        assert np.array_equal(a[i].pops(), b[i].pops()), i
        assert np.array_equal(a[i].nodes(0), b[i].nodes(0)), i
