"""The plane sweeps of the collide and of the moments rebuild at the sizes
where they can go wrong: tiles wider than the lattice, ragged last tiles,
chunks of one plane, a last chunk of one plane, walls and periodic ends.  A
cell's result does not depend on the tile or chunk that computes it, so every
split gives the same bits; the fields are checked against the FP64 oracle.
Also the profile of strongly deformed capsules against the oracle's brute
force, and a batch whose markers are set from outside between steps."""
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


def _fluid(n, storage, wall, tau=1.0):
    dim = 2 if len(n) == 2 else 3
    nz = n[2] if dim == 3 else 1
    p = W.Params(dim=dim, nx=n[0], ny=n[1], nz=nz, wall_last=wall, storage=storage, alpha=1.0, tau=tau,
                 gamma_phi=0.2, gamma_psi=0.2, interface_pos=n[-1] / 2.0)
    return W.Workload("fluid", p, [])


CASES = [((4, 4, 4), "f32", 0), ((5, 4, 7), "f32", 1), ((33, 5, 9), "f32", 1), ((32, 8, 17), "f32", 0),
         ((65, 17, 6), "f32", 1), ((31, 6, 5), "f16", 1), ((34, 5, 9), "bf16", 0), ((5, 4), "f64", 0),
         ((67, 9), "f64", 1), ((129, 33), "f32", 0)]


@pytest.mark.parametrize("n,storage,wall", CASES)
def test_every_split_gives_the_same_bits(n, storage, wall):
    from paper_1906_03065_gb300 import Simulation
    wl = _fluid(n, storage, wall)
    C0, u0 = W.random_fields(wl.params, seed=3)
    ref = Simulation(wl).init(C0, u0)
    ref.step(4)
    P = ref.pops()
    for variant in (13, 14, 15, 16, 28, 29):
        for zc in sorted({1, 2, 3, n[-1] - 1, n[-1]}):
            s = Simulation(wl).init(C0, u0)
            s.set_tile(variant, zc)
            s.step(4)
            assert np.array_equal(s.pops(), P), (variant, zc)
    # FP32: 4 steps from O(1) fields, each adding a few roundings of 6e-8
    bound = {"f64": 1e-12, "f32": 5e-6, "f16": 3e-3, "bf16": 3e-2}[storage]
    o = oracle.Oracle(wl, Cf=C0, u=u0)
    o.step(4)
    for name in ("C1", "C2", "C3"):
        assert np.abs(ref.field(name) - o.field(name)).max() < bound, name


@pytest.mark.parametrize("n,wall", [((5, 4, 7), 1), ((33, 5, 9), 0), ((65, 9, 6), 1)])
def test_general_collide_splits(n, wall):
    from paper_1906_03065_gb300 import Simulation
    wl = _fluid(n, "f32", wall, tau=0.8)
    C0, u0 = W.random_fields(wl.params, seed=4)
    ref = Simulation(wl).init(C0, u0)
    ref.step(3)
    for variant, zc in ((0, 1), (1, 2), (2, n[2]), (4, n[2] - 1), (6, 3), (9, 1), (12, 2)):
        s = Simulation(wl).init(C0, u0)
        s.set_tile(variant, zc)
        s.step(3)
        assert np.abs(s.pops() - ref.pops()).max() < 1e-6, (variant, zc)
    o = oracle.Oracle(wl, Cf=C0, u=u0)
    o.step(3)
    for name in ("C1", "C2", "C3"):
        assert np.abs(ref.field(name) - o.field(name)).max() < 5e-6, name


@pytest.mark.parametrize("level,radius,jitter", [(1, 6.0, 0.0), (2, 7.0, 0.3), (2, 7.0, 0.6), (3, 9.0, 0.2)])
def test_profile_of_deformed_capsules(level, radius, jitter):
    """I within 4e-6 of the oracle's: FP32 distances of up to 8 cells carry
    about 1e-6, and dI/dd is at most 1/(4 alpha)."""
    from paper_1906_03065_gb300 import Simulation
    wl = W.small_3d("f32", nx=44, ny=40, nz=42, level=level, radius=radius, centre=(22.0, 20.0, 21.0))
    wl.membranes[0] = W.jitter_nodes(wl.membranes[0], jitter, seed=6)
    s = Simulation(wl).init()
    s.step(1)
    o = oracle.Oracle(wl)
    I, _, _ = o.iprofile(o.nodes(0))
    assert np.abs(s.field("I") - I).max() < 4e-6


def test_batch_follows_markers_set_from_outside():
    from paper_1906_03065_gb300 import Batch, Simulation
    wls = W.small_sweep_3d(3, seed=9, storage="f32")
    b = Batch(wls).init()
    alone = [Simulation(wl).init() for wl in wls]
    b.step(5)
    for s in alone:
        s.step(5)
    X = b[1].nodes(0)
    X[:, 0] += 0.4
    b[1].set_nodes(0, X)
    alone[1].set_nodes(0, X)
    b.step(6)
    for i, s in enumerate(alone):
        s.step(6)
        assert np.abs(b[i].field("I") - s.field("I")).max() < 1e-6, i
        assert np.abs(b[i].nodes(0) - s.nodes(0)).max() < 1e-7, i
