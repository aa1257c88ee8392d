"""Coupling sums over their whole range: a cell's contribution to a marker is
held in fixed point up to +-4096, far beyond what the 32-bit parts of the
common case hold."""
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


@pytest.mark.parametrize("kappa_c,psi", [(0.02, 0.0), (40.0, 0.0), (400.0, 0.0), (2500.0, 0.0), (2500.0, 1.0)])
def test_first_step_of_a_strongly_coupled_capsule(kappa_c, psi):
    """From rest with no free-energy force (kappa 0, psi constant), one step:
    the fluid's momentum comes from the spread coupling force, whose
    contributions of one cell reach kappa_c / 7 at psi = 1.  Against the FP64
    oracle, relative to the largest momentum: the populations of a cell are up
    to |u| (500 here) times larger than the momentum left of them, each rounded
    to 6e-8: 1e-4."""
    from paper_1906_03065_gb300 import Simulation
    n = (30, 28, 26)
    p = W.Params(dim=3, nx=n[0], ny=n[1], nz=n[2], storage="f32", alpha=1.0, kappa1=0.0, kappa2=0.0, kappa3=0.0,
                 kappa_c=kappa_c, dc=8.0, interface_pos=13.0, gamma_phi=0.0, gamma_psi=0.0)
    m = W.icosphere(2, 6.0, (15.2, 14.1, 13.3))
    m.G = m.kb = 0.0
    wl = W.Workload("coupled", p, [m])
    C0 = np.zeros((3, p.ncells))
    C0[0] = 1.0 - psi
    C0[2] = psi
    u0 = np.zeros((3, p.ncells))
    s, o = Simulation(wl).init(C0, u0), oracle.Oracle(wl, Cf=C0, u=u0)
    s.step(1)
    o.step(1)
    c, _ = o.lattice()
    j, jo = (np.tensordot(c.T.astype(float), q.pops()[0], 1) for q in (s, o))
    assert np.abs(j - jo).max() < 1e-4 * np.abs(jo).max()
