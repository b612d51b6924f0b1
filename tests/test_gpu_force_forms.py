"""The FP64 steps' forms by model and force: a force along x (F_y = F_z = 0) or a general one,
uniform or per node, with inlet and outlet nodes by both boundary schemes, for the
incompressible LBGK (the hybrid collision in a kernel of its own) and MRT, against the oracle.

Bar: that of the model tests, |f_gpu - f_oracle| / w_i <= 1e-12.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1611_02445_gb300 import inputs as I
from paper_1611_02445_gb300 import lbm

pytestmark = pytest.mark.gpu
_, W, _ = O.lattice()


@pytest.mark.parametrize("bc", ["none", "equilibrium", "zou_he"])
@pytest.mark.parametrize("force", ["zero", "x", "general", "field_x", "field_general"])
@pytest.mark.parametrize("eq,coll", [(O.EQ_INCOMPR, O.COLL_BGK), (O.EQ_QCOMPR, O.COLL_MRT), (O.EQ_INCOMPR, O.COLL_MRT)])
def test_forms_match_oracle(eq, coll, force, bc):
    nt = np.ones((9, 10, 17), np.uint8)
    nt[:, 0] = nt[:, -1] = 0
    nt[4:6, 3:5, 6:9] = 0
    if bc != "none":
        nt[:, 1:-1, 0] = 2
        nt[:, 1:-1, -1] = 3
    f0 = I.random_populations(nt, 0.02, seed=6)
    g = {"zero": (0.0, 0.0, 0.0), "x": (3e-5, 0.0, 0.0), "field_x": (0.0, 0.0, 0.0)}.get(force, (1e-5, -2e-5, 3e-5))
    gf = I.body_force_field(nt, 2e-5, 1e-6) if force.startswith("field") else None
    u_in, rho_out, steps = (0.03, 0.004, -0.002), 1.01, 12
    with lbm.Lattice(nt, "f64", 0) as L:
        L.set_params(0.75, g, gf, u_in, rho_out)
        L.set_model(eq, coll)
        if bc == "zou_he":
            L.set_bc(lbm.BC_ZOU_HE, 0, 1)
        L.set_f(f0)
        L.step(steps)
        fg = L.get_f()
    fo = O.run_m(f0, nt, steps, 0, 0.75, g, gf, u_in, rho_out, eq=eq, coll=coll,
                 rates=O.mrt_rates(0.75) if coll else None, bc=O.BC_ZOU_HE if bc == "zou_he" else 0, in_face=0, out_face=1)
    on = nt != 0
    err = float((np.abs(fg[:, on] - fo[:, on]) / W[:, None]).max())
    print(f"{eq},{coll} {force} {bc}: {err:.3e}")
    assert err <= 1e-12
