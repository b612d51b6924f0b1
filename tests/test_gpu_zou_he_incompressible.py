"""Zou-He inlets and outlets of the incompressible LBGK in FP64 storage are completed and collided
in FP64: after one step their populations agree with the FP64 oracle to FP64 rounding, on every
face, with and without forces, also where an inlet meets walls and in small ragged boxes.

Bars: the rounding errors of such a node in FP64 are 3e-16 of w, rms over the boundary populations
(LBM_F64_NATIVE against long double), so two FP64 evaluations in different order differ by
less than 1e-15 rms; the worst case of the 14- and 19-term sums is 1.5e-14 of w.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1611_02445_gb300 import inputs as I
from paper_1611_02445_gb300 import lbm

pytestmark = pytest.mark.gpu
_, W, _ = O.lattice()


def _duct(axis, flip, shape):
    """Inlet and outlet on opposite faces of the axis, walls on the faces of the next axis."""
    nt = np.ones(shape, np.uint8)
    wall = [slice(None)] * 3
    for at in (0, -1):
        wall[2 - (axis + 1) % 3] = at
        nt[tuple(wall)] = lbm.SOLID
    face = [slice(None)] * 3
    for at, kind in ((0, lbm.INLET), (-1, lbm.OUTLET)):
        face[2 - axis] = -1 - at if flip else at
        part = nt[tuple(face)]
        part[part != lbm.SOLID] = kind
    return nt, (2 * axis + 1, 2 * axis) if flip else (2 * axis, 2 * axis + 1)


@pytest.mark.parametrize("g,field", [((0.0, 0.0, 0.0), False), ((1e-4, 0.0, 0.0), False), ((1e-4, -2e-5, 3e-5), False),
                                     ((0.0, 0.0, 0.0), True), ((0.0, 2e-5, 0.0), True)])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("flip", [False, True])
def test_boundary_nodes_collide_in_fp64(axis, flip, g, field):
    nt, (fi, fo) = _duct(axis, flip, (13, 22, 17))
    f0 = I.random_populations(nt, 0.05, seed=41)
    gf = I.body_force_field(nt, 1e-4, 1e-5) if field else None
    u_in, tau = (0.04, 0.01, -0.02), 0.6
    with lbm.Lattice(nt, "f64", 0) as L:
        L.set_params(tau, g, gf, u_in, 1.01)
        L.set_model(lbm.EQ_INCOMPR, lbm.COLL_BGK)
        L.set_bc(lbm.BC_ZOU_HE, fi, fo)
        L.set_f(f0)
        L.step(1)
        fg = L.get_f()
    fr = O.step_m(f0, nt, 0, tau, g, gf, u_in, 1.01, eq=O.EQ_INCOMPR, bc=O.BC_ZOU_HE, in_face=fi, out_face=fo)
    e = np.abs(fg - fr) / W[:, None, None, None]
    boundary = (nt == lbm.INLET) | (nt == lbm.OUTLET)
    assert boundary.sum() > 100
    assert float(np.sqrt((e[:, boundary] ** 2).mean())) <= 1e-15
    assert float(e[:, boundary].max()) <= 1.5e-14
    assert float(e[:, nt == lbm.FLUID].max()) <= 1e-12
