"""A chained step lets the next one start at once or at its end and takes its groups in index order or
reversed, by the number of groups for its CTAs. One call of many steps equals single calls (never
chained) bit for bit in every regime of that rule: fewer CTAs than half the places, between half and
two thirds, places nearly full, one to five groups a CTA with fewer and with more than half of the
CTAs one group ahead, five and more, and Zou-He nodes.
"""
import numpy as np
import pytest

from paper_1611_02445_gb300 import lbm

pytestmark = pytest.mark.gpu


def _run(nt, dtype, calls, zou_he):
    with lbm.Lattice(nt, dtype, 0) as L:
        L.set_params(0.7, (2e-5, 1e-5, 0.0), None, (0.01, 0.0, 0.0), 1.0)
        if zou_he:
            L.set_bc(lbm.BC_ZOU_HE, 0, 1)
        L.init_equilibrium(1.0, (0.01, -0.02, 0.03))
        for n in calls:
            L.step(n)
        return L.save_state()


@pytest.mark.parametrize("side", [33, 40, 45, 50, 56, 61, 70, 95])
@pytest.mark.parametrize("dtype", ["f64", "f64n", "f32", "f16s"])
def test_any_number_of_groups(dtype, side):
    nt = np.ones((side, side, side), np.uint8)
    assert _run(nt, dtype, [37], False) == _run(nt, dtype, [1] * 37, False)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("shape", [(40, 50, 90), (44, 50, 100)])
def test_zou_he_duct(dtype, shape):
    nt = np.ones(shape, np.uint8)
    nt[:, :, 0], nt[:, :, -1] = lbm.INLET, lbm.OUTLET
    nt[:, 0, :] = nt[:, -1, :] = lbm.SOLID
    assert _run(nt, dtype, [37], True) == _run(nt, dtype, [1] * 37, True)
