"""Device memory that really runs out (the tests of test_gpu_failures.py fake the failure on the
host): the call reports it, and the calls after it work."""
import numpy as np
import pytest

from paper_1611_02445_gb300 import inputs as I
from paper_1611_02445_gb300 import lbm

pytestmark = pytest.mark.gpu


def test_an_adjoint_too_large_for_the_device_leaves_the_context_usable():
    """Checkpoints of twice the device's memory: LBM_ENOMEM before any work, and the state can
    be reduced, exported and stepped as if the call had not been made."""
    import torch
    nt = I.random_box(96, 96, 96, p_solid=0.3, seed=91)
    total = torch.cuda.get_device_properties(0).total_memory

    def run(with_failure):
        with lbm.Lattice(nt, "f64", 0b111) as L:
            L.set_params(0.8, (1e-5, 0, 0))
            L.init_equilibrium()
            L.step(3)
            if with_failure:
                T = 2 * total // L.info()["copy_bytes"]
                with pytest.raises(lbm.LBMError) as e:
                    L.adjoint(T, T, 5)
                assert e.value.status == 2                     # LBM_ENOMEM
            first = L.reduce()
            L.step(20)
            return first, L.reduce(), L.get_f()

    (m0, p0), (m1, p1), f = run(False)
    (n0, q0), (n1, q1), g = run(True)
    assert m0 == n0 and m1 == n1 and np.array_equal(p0, q0) and np.array_equal(p1, q1)
    assert np.array_equal(f, g, equal_nan=True)
