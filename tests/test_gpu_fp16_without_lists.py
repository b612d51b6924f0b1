"""An FP16 context whose import lists (60 B a node beside 76 B of populations) do not fit the device
is built without them: its step pulls node by node, to the same bits, and so does its adjoint's
forward. Every allocation of lbm_create is made to fail on the host, one at a time.
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


def _results(L, nt, f0, dtype):
    L.set_params(0.8, (1e-5, 0, 0), None, (0.03, 0, 0), 1.0)
    L.set_f(f0)
    L.step(23)
    out = [L.get_f()[:, nt != 0]]
    if dtype == "f16s":
        loss, dg, dtau = L.adjoint(7, 3, 5)
        out += [loss, dg, dtau]
    return out


@pytest.mark.parametrize("dtype", ["f16s", "f16sr"])
def test_a_failed_list_allocation_takes_the_node_by_node_step(dtype):
    nt = I.random_box(24, 20, 28, p_solid=0.3, seed=95, boundary=True)
    f0 = I.random_populations(nt, 0.05, seed=96)
    live0 = lbm.testing_live_allocations()
    with lbm.Lattice(nt, dtype, 0b110) as L:
        full = lbm.testing_live_allocations() - live0
        ref = _results(L, nt, f0, dtype)
    without = 0
    for k in range(200):
        lbm.testing_fail_allocation(k)
        try:
            L = lbm.Lattice(nt, dtype, 0b110)
        except lbm.LBMError as e:
            assert e.status == 2, (k, str(e))                   # LBM_ENOMEM
            assert lbm.testing_live_allocations() == live0, k
            continue
        finally:
            lbm.testing_fail_allocation(-1)
        with L:
            held = lbm.testing_live_allocations() - live0
            got = _results(L, nt, f0, dtype)
        assert lbm.testing_live_allocations() == live0
        assert all(np.array_equal(a, b) for a, b in zip(ref, got)), k
        if held == full:   # k lies beyond the last allocation
            break
        assert held == full - 1, k
        without += 1
    assert without == 1
