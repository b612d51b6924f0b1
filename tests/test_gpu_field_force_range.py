"""The velocity field under a per-node force of any size: FP32 results of FP64 storage form the force
in pairs, which hold [2^-60, 2), and other nodes in FP64. Reference and bars as in test_fields.py
(the result rounds once, the fixed-point momentum to 19 2^-59). At rest the momentum is exactly 0
and the velocity -F / (2 rho), to the rounding of the result alone."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1611_02445_gb300 import inputs as I
from paper_1611_02445_gb300 import lbm

pytestmark = pytest.mark.gpu
FORCES = [0.0, -0.0, 1e-300, 2.0 ** -61, -(2.0 ** -60), 1e-19, 1e-5, -0.3, np.nextafter(2.0, 0.0), 2.0, -2.5, 4.0, 300.0, -1e9]


@pytest.mark.parametrize("eq", [O.EQ_QCOMPR, O.EQ_INCOMPR])
@pytest.mark.parametrize("out64", [False, True])
@pytest.mark.parametrize("dtype", ["f64", "f64n", "f32"])
def test_velocity_under_any_force(dtype, out64, eq):
    nt = np.ones((6, 7, 9), np.uint8)
    f0 = I.random_populations(nt, 0.05, seed=3)
    gf = np.resize(np.array(FORCES), nt.shape)
    with lbm.Lattice(nt, dtype, 0) as L:
        L.set_params(0.8, None, gf)
        L.set_model(eq, 0)
        L.set_f(f0)
        f = L.get_f().astype(np.longdouble)
        rho, u = L.macroscopic(out64)
    F = (gf.astype(np.float32) if dtype == "f32" else gf).astype(np.longdouble)
    c = np.asarray(O.lattice()[0]).reshape(-1, 3)[:, 0].astype(np.longdouble)
    r = f.sum(0)
    want = (np.tensordot(c, f, 1) - F / 2) / (r if eq == O.EQ_QCOMPR else 1)
    ulp = 2.0 ** -52 if out64 else 2.0 ** -23
    a64 = 2.0 ** -44 if dtype == "f32" else 19 * 2.0 ** -59
    assert (np.abs(rho - r) <= ulp * np.abs(r) + a64).all()
    assert (np.abs(u[0] - want) <= ulp * np.abs(want) + 4 * a64).all()


@pytest.mark.parametrize("eq", [O.EQ_QCOMPR, O.EQ_INCOMPR])
@pytest.mark.parametrize("out64", [False, True])
@pytest.mark.parametrize("dtype", ["f64", "f64n"])
def test_velocity_at_rest_under_any_force(dtype, out64, eq):
    nt = np.ones((6, 7, 9), np.uint8)
    gf = np.resize(np.array(FORCES + [1e30, 2.0 ** 130]), nt.shape)
    with lbm.Lattice(nt, dtype, 0) as L:
        L.set_params(0.8, None, gf)
        L.set_model(eq, 0)
        L.set_f(np.broadcast_to(O.lattice()[1][:, None, None, None], (19,) + nt.shape))
        r = L.get_f().astype(np.longdouble).sum(0)
        rho, u = L.macroscopic(out64)
    want = -gf.astype(np.longdouble) / 2 / (r if eq == O.EQ_QCOMPR else 1)
    with np.errstate(over="ignore", under="ignore"):
        fits = np.abs(want) < (1e300 if out64 else 3e38)
        bar = (2.0 ** -52 if out64 else 2.0 ** -23) * np.abs(want) + (0 if out64 else 2.0 ** -149)
        assert (np.abs(u[0] - want)[fits] <= bar[fits]).all()
        assert (u[0][~fits] == -np.inf).all()
