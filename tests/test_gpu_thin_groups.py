"""The FP16 step copies the part of a work group's data blocks that holds nodes, in pieces of eight
lanes: groups of every remainder, alone and beside others, against the node-by-node step (a context
whose import lists failed to be allocated, on the host), bit for bit in each kernel.
"""
import numpy as np
import pytest

from paper_1611_02445_gb300 import inputs as I
from paper_1611_02445_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _no_injection_left():
    yield
    lbm.testing_fail_allocation(-1)


def _without_lists(nt, periodic):
    live0 = lbm.testing_live_allocations()
    with lbm.Lattice(nt, "f16s", periodic):
        full = lbm.testing_live_allocations() - live0
    for k in range(200):
        lbm.testing_fail_allocation(k)
        try:
            L = lbm.Lattice(nt, "f16s", periodic)
        except lbm.LBMError:
            continue
        finally:
            lbm.testing_fail_allocation(-1)
        assert lbm.testing_live_allocations() - live0 == full - 1
        return L
    raise AssertionError("no context without lists")


@pytest.mark.parametrize("nodes", [1, 2, 7, 8, 9, 15, 16, 17, 31, 33, 64, 127, 129, 200, 255, 256])
@pytest.mark.parametrize("boxes", [1, 3])
def test_groups_of_any_size(nodes, boxes):
    rng = np.random.default_rng(nodes)
    nt = np.zeros((4, 4, 16 * boxes), np.uint8)     # four tiles: one work group, if full
    for b in range(boxes):
        part = np.zeros(256, np.uint8)
        part[rng.permutation(256)[:max(1, nodes - 3 * b)]] = lbm.FLUID
        nt[:, :, 16 * b:16 * b + 16] = part.reshape(4, 4, 16)
    f0 = I.random_populations(nt, 0.1, seed=7)
    g = (2e-5, -1e-5, 1e-5)
    out = []
    for make in (lambda: lbm.Lattice(nt, "f16s", 0b111), lambda: _without_lists(nt, 0b111)):
        with make() as L:
            L.set_params(0.8, g)
            for kernel in (lbm.KERNEL_FULL, lbm.KERNEL_PROPAGATE, lbm.KERNEL_RW):
                L.set_f(f0)
                L.step_kernel(kernel, 5)
                out.append(L.get_f()[:, nt != 0])
    assert all(np.array_equal(a, b) for a, b in zip(out[:3], out[3:]))
