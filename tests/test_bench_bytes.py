"""The bytes per cell that the bench's rooflines are made of, for the kernels
that a step runs (no GPU needed)."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def bench():
    sys.path.insert(0, ROOT)
    import bench
    return bench


def test_bytes_of_a_tau_1_step(bench):
    """FP32 arithmetic: the rebuild reads the 12 stored values and writes rho -
    1, phi, psi and j (6); the collide reads those and I and writes 12 values.
    The same for every storage type."""
    assert bench.state_kernel_bytes() == {"k_moments_recon": 72, "k_collide": 76}
    for storage in ("f32", "f16", "bf16"):
        assert bench.moved_bytes(storage, True) == 148
        assert [(n, p) for n, p, _ in bench.lattice_kernels(storage, True)] == [
            ("k_moments_recon", "ms_moments"), ("k_collide", "ms_collide")]


def test_bytes_of_a_general_step(bench):
    """Populations pulled by both kernels and stored by one (228 B in FP32, 118
    with 16-bit storage), rho - 1, phi, psi written and read, I read."""
    assert bench.moved_bytes("f32", False) == 3 * 228 + 12 + 16
    assert bench.moved_bytes("f16", False) == bench.moved_bytes("bf16", False) == 3 * 118 + 12 + 16
