"""The membrane profile after the state or the markers were replaced: the
profile of the whole lattice belongs to the markers as they are, and nothing
is left of where the membrane has been before."""
import numpy as np
import pytest

import oracle
from paper_1906_03065_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1906_03065_gb300 import build
    build.build()
    oracle.build()


def _drifting():
    """A capsule that a uniform flow carries 0.15 cells a step along x."""
    wl = W.small_3d("f32", nx=72, ny=28, nz=26, level=2, radius=5.0, centre=(14.2, 14.1, 13.3), wall=0)
    wl.params.u0 = (0.15, 0.0, 0.0)
    wl.params.interface_pos = -1.0
    return wl


def _single(wl):
    from paper_1906_03065_gb300 import Simulation
    s = Simulation(wl).init()
    return s, s.step


def _batched(wl):
    from paper_1906_03065_gb300 import Batch
    b = Batch([wl, wl]).init()
    return b[1], b.step


@pytest.mark.parametrize("make", [_single, _batched])
def test_markers_set_far_away_leave_nothing_behind(make):
    """I over the whole lattice within 4e-6 of the oracle's brute force (FP32
    distances of up to 8 cells, dI/dd at most 1/4)."""
    s, step = make(_drifting())
    step(2)
    X = s.nodes(0)
    X[:, 0] += 36.0
    s.set_nodes(0, X)
    step(1)
    o = oracle.Oracle(_drifting())
    I, _, _ = o.iprofile(X)
    assert np.abs(s.field("I") - I).max() < 4e-6


@pytest.mark.parametrize("make", [_single, _batched])
def test_a_loaded_checkpoint_resumes_beside_the_old_band(make):
    """A run that drifts more than its profile box, then goes back to an
    earlier checkpoint, passes where the membrane was before: the profile
    equals that of a context which has not been there, bit for bit."""
    wl = _drifting()
    s, step = make(wl)
    blob = s.save()
    step(130)
    assert s.nodes(0)[:, 0].mean() > 14.2 + 10 + 5
    s.load(blob)
    fresh, fresh_step = make(wl)
    fresh.load(blob)
    for _ in range(6):
        step(12)
        fresh_step(12)
        assert np.array_equal(s.field("I"), fresh.field("I"))
    assert np.array_equal(s.pops(), fresh.pops())
    assert np.array_equal(s.nodes(0), fresh.nodes(0))


@pytest.mark.parametrize("make", [_single, _batched])
def test_a_new_start_resumes_beside_the_old_band(make):
    wl = _drifting()
    s, step = make(wl)
    X0 = s.nodes(0)
    step(130)
    s.set_nodes(0, X0)
    s.init()
    fresh, fresh_step = make(wl)
    assert np.array_equal(s.field("I"), fresh.field("I"))
    for _ in range(6):
        step(12)
        fresh_step(12)
        assert np.array_equal(s.field("I"), fresh.field("I"))
    assert np.array_equal(s.pops(), fresh.pops())
