"""Arena sizes (host-only): the tau = 1 scheme's state takes no memory of its
own, so a lattice or batch that fits at any other tau fits at tau = 1."""
import ctypes

import pytest

from paper_1906_03065_gb300 import workloads as W


def _bytes(wl):
    import paper_1906_03065_gb300 as T
    from paper_1906_03065_gb300 import build
    build.build()
    cp = T.make_params(wl.params)
    keep = []
    n = ctypes.c_size_t(0)
    T._check(T.lib().tlb_state_bytes(ctypes.byref(cp), T._marshal_membranes(wl, keep), len(wl.membranes),
                                     ctypes.byref(n)))
    return n.value


@pytest.mark.parametrize("make", [lambda: W.small_2d("f64"), lambda: W.small_2d("f32"), lambda: W.small_3d("f32"),
                                  lambda: W.capsule_3d("f16"), lambda: W.capsule_3d("bf16")])
def test_the_state_at_tau_1_lies_in_the_population_buffers(make):
    one, other = make(), make()
    other.params.tau = other.params.tau_phi = other.params.tau_psi = 0.9
    assert _bytes(one) == _bytes(other)


@pytest.mark.parametrize("q,real,store", [(9, 8, 8), (9, 4, 4), (19, 4, 4), (19, 4, 2)])
def test_a_population_buffer_holds_the_state(q, real, store):
    assert (12 + 2) * real <= (3 * q - 2) * store
