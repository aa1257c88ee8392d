"""Readers of the tau = 1 state: what they see are the populations that the
state stands for, in every storage type."""
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


def _peskin(r):
    x = np.abs(r)
    near = (3 - 2 * x + np.sqrt(np.maximum(0, 1 + 4 * x - 4 * x * x))) / 8
    far = (5 - 2 * x - np.sqrt(np.maximum(0, -7 + 12 * x - 4 * x * x))) / 8
    return np.where(x <= 1, near, np.where(x <= 2, far, 0.0))


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_markers_move_with_the_readable_populations(storage):
    """One step of a fluid with no force at all (every modulus and kappa 0) and
    strong random flow: each marker's displacement is the kernel-weighted
    velocity of the streamed populations as read back.  FP32 arithmetic:
    weights to a few units of 6e-8 each and sums of 19 terms below 0.1, so
    2e-7 on a displacement below 0.5; one population off by a unit of its
    storage type moves a marker by up to 1e-5."""
    import oracle
    from paper_1906_03065_gb300 import Simulation
    oracle.build()
    n = (40, 38, 36)
    p = W.Params(dim=3, nx=n[0], ny=n[1], nz=n[2], storage=storage, alpha=1.0, kappa1=0.0, kappa2=0.0, kappa3=0.0,
                 kappa_c=0.0, dc=8.0, interface_pos=18.0)
    m = W.icosphere(4, 11.0, (20.2, 19.1, 18.3))
    m.G = m.kb = 0.0
    wl = W.Workload("flow", p, [m])
    rng = np.random.default_rng(12)
    C0, _ = W.random_fields(p, seed=12, amp=0.2)
    u0 = rng.uniform(-0.25, 0.25, (3, p.ncells))
    s = Simulation(wl).init(C0, u0)
    X0 = s.nodes(0)
    s.step(1)
    U = s.nodes(0) - X0
    c, w = oracle.Oracle(wl, init=False).lattice()
    f = s.pops()[0]
    rho = f.sum(0)
    v = (np.tensordot(c.T.astype(float), f, 1) / rho).reshape(3, n[2], n[1], n[0])
    ref = np.zeros_like(U)
    base = np.floor(X0).astype(int) - 1
    for k in range(4):
        for j in range(4):
            for i in range(4):
                cell = base + np.array([i, j, k])
                wt = _peskin(cell - X0).prod(axis=1)
                q = cell % np.array(n)
                ref += wt[:, None] * v[:, q[:, 2], q[:, 1], q[:, 0]].T
    assert np.abs(U).max() < 0.5
    assert np.abs(U - ref).max() < 2e-7


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_moment_state_equals_the_population_scheme(storage):
    """From populations written by the caller, one step of the tau = 1 collide
    (state in 12 values per cell, pulled this once) and a second one (rebuilt
    from them) give the populations of the general collide, which stores and
    pulls them: the collisions round differently in FP32 (a few units of 6e-8
    of values up to 1), and each of the two roundings to the storage type may
    then fall on either side."""
    import oracle
    from paper_1906_03065_gb300 import Simulation
    oracle.build()
    wl = W.small_3d(storage)
    o = oracle.Oracle(wl, init=False)
    C0, u0 = W.random_fields(wl.params, seed=4)
    c, w = o.lattice()
    a, b = Simulation(wl).init(C0, u0), Simulation(wl).init(C0, u0)
    b.set_tile(3, 8)
    rng = np.random.default_rng(5)
    P = a.pops() + 1e-3 * rng.standard_normal((3, o.Q, o.N)) * w[None, :, None]
    eps = {"f32": 0.0, "f16": 2.0 ** -10, "bf16": 2.0 ** -7}[storage]
    for s in (a, b):
        s.set_pops(P)
    a.step(1)
    b.step(1)
    Pa, Pb = a.pops(), b.pops()
    stored = np.abs(Pb)
    stored[0] -= w[:, None]
    stored = np.abs(stored)
    stored[1:, 0] = 0.0  # the rest populations of the order parameters are FP32
    assert np.all(np.abs(Pa - Pb) <= eps * stored + 1e-6)
    assert np.abs(a.nodes(0) - b.nodes(0)).max() < (1e-6 if storage == "f32" else 2e-3)
    # the second step from the same stored state in both schemes
    blob = a.save()
    b.load(blob)
    assert np.array_equal(b.pops(), Pa)
    a.step(1)
    b.step(1)
    Pa, Pb = a.pops(), b.pops()
    stored = np.abs(np.stack([Pb[0] - w[:, None], Pb[1], Pb[2]]))
    stored[1:, 0] = 0.0
    assert np.all(np.abs(Pa - Pb) <= eps * stored + 1e-6)
    da, db = a.diagnostics(), b.diagnostics()
    assert np.allclose(da.mass[:], db.mass[:], rtol=0, atol=(1e-6 + eps * 0.05) * o.N)


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("general", [False, True])
def test_network_input_of_a_stepped_context(storage, general):
    """The network's input tensor holds the phi and psi that the last step
    started from (bf16, to half a unit beside FP32 rounding), those of the
    start before any step, and those of the new start after another one."""
    import torch
    from paper_1906_03065_gb300 import Simulation, WarmStartNet
    n = 48
    p = W.Params(dim=3, nx=n, ny=n, nz=n, wall_last=1, storage=storage, alpha=1.0, dc=8.0, interface_pos=24.0,
                 tau=0.8 if general else 1.0)
    m = W.icosphere(2, 8.0, (24.2, 24.1, 23.7))
    m.G, m.kb = 0.01, 0.005
    s = Simulation(W.Workload("cap", p, [m]))
    C0, u0 = W.random_fields(p, seed=8)
    s.init(C0, u0)
    net = WarmStartNet(n, 16, 4, 1)

    def check(phi, psi):
        x = net.input(s, np.zeros(5))
        torch.cuda.synchronize()
        x = x.float().cpu().numpy().astype(float)
        for k, ref in ((0, phi), (1, psi)):
            assert np.all(np.abs(x[:, k] - ref) <= 2.0 ** -8 * np.abs(ref) + 1e-6), k

    def order(s):
        return s.field("phi"), s.field("psi")

    check(C0[0] - C0[1], C0[2])
    s.step(2)
    ref = order(s)
    s.step(1)
    check(*ref)
    ref = order(s)
    s.step(1)
    check(*ref)
    s.step(39)
    ref = order(s)
    s.step(1)
    check(*ref)
    C1, u1 = W.random_fields(p, seed=9)
    s.init(C1, u1)
    check(C1[0] - C1[1], C1[2])
