"""The FP32 incompressible LBGK kernel against the oracle: fluid nodes through the pair form with 1
in place of 1 / rho, inlet and outlet nodes by both boundary schemes, uniform and per-node
forces. Bar: that of the FP32 model tests (4e-6 of w).
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1611_02445_gb300 import inputs as I
from paper_1611_02445_gb300 import lbm

pytestmark = pytest.mark.gpu
_, W, _ = O.lattice()


@pytest.mark.parametrize("bc", ["none", "equilibrium", "zou_he"])
@pytest.mark.parametrize("field", [False, True])
@pytest.mark.parametrize("shape", [(4, 4, 4), (9, 10, 17)])
def test_incompressible_f32_matches_oracle(shape, field, bc):
    nt = np.ones(shape, np.uint8)
    if shape != (4, 4, 4):
        nt[:, 0] = nt[:, -1] = 0
    if bc != "none":
        nt[:, 1:-1, 0] = 2
        nt[:, 1:-1, -1] = 3
    f0 = I.random_populations(nt, 0.02, seed=6)
    gf = I.body_force_field(nt, 2e-5, 1e-6) if field else None
    g, u_in, steps = (1e-5, -2e-5, 3e-5), (0.03, 0.004, -0.002), 12
    with lbm.Lattice(nt, "f32", 0) as L:
        L.set_params(0.75, g, gf, u_in, 1.01)
        L.set_model(O.EQ_INCOMPR, O.COLL_BGK)
        if bc == "zou_he":
            L.set_bc(lbm.BC_ZOU_HE, 0, 1)
        L.set_f(f0)
        L.step(steps)
        fg = L.get_f()
    fo = O.run_m(f0, nt, steps, 0, 0.75, g, gf, u_in, 1.01, eq=O.EQ_INCOMPR, coll=O.COLL_BGK,
                 bc=O.BC_ZOU_HE if bc == "zou_he" else 0, in_face=0, out_face=1)
    on = nt != 0
    assert float((np.abs(fg[:, on] - fo[:, on]) / W[:, None]).max()) <= 4e-6
