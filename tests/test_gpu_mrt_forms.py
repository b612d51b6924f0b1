"""The forms of the MRT collision against the oracle, over the range of states each takes.

FP64 storage forms the moments in 64-bit fixed point for populations in [2^-6, 2) and a
density below 3, and in FP64 for any other node; FP32 through shared sums; FP16 through the
products written out. States scaled so that nodes lie inside, outside and on both sides of
those limits (also with negative and large single populations), forces on every axis, both
equilibria, sizes with partly filled and several work groups.

Bars: those of the model tests (1e-12 of w for FP64, 4e-6 for FP32, 3e-3 for FP16), times the
scale of the populations.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1611_02445_gb300 import inputs as I
from paper_1611_02445_gb300 import lbm

pytestmark = pytest.mark.gpu
_, W, _ = O.lattice()
TOL = {"f64": 1e-12, "f64n": 1e-12, "f32": 4e-6, "f16s": 3e-3}


@pytest.mark.parametrize("dtype", ["f64", "f64n", "f32", "f16s"])
@pytest.mark.parametrize("eq", [O.EQ_QCOMPR, O.EQ_INCOMPR])
@pytest.mark.parametrize("state", ["near", "thin", "dense", "denser", "mixed"])
@pytest.mark.parametrize("shape", [(4, 4, 4), (5, 9, 7), (16, 12, 20)])
def test_mrt_matches_oracle(shape, state, eq, dtype):
    nx, ny, nz = shape
    nt = I.random_box(nx, ny, nz, 0.2 if nx == 16 else 0.0, seed=3)
    f0 = I.random_populations(nt, 0.05, seed=4)
    scale = {"near": 1.0, "thin": 0.4, "dense": 1.72, "denser": 3.3, "mixed": 1.0}[state]
    f0 *= scale
    if state == "mixed":
        rng = np.random.default_rng(5)
        hit = rng.random(nt.shape) < 0.1
        f0[0][hit] += 2.1          # rest population outside the fixed-point range
        f0[9][rng.random(nt.shape) < 0.1] = -1e-3
        scale = 3.1
    steps = 6
    g = (1e-5, -2e-5, 3e-5)
    with lbm.Lattice(nt, dtype, 0) as L:
        L.set_params(0.8, g)
        L.set_model(eq, O.COLL_MRT)
        L.set_f(f0)
        L.step(steps)
        fg = L.get_f()
    fo = O.run_m(f0, nt, steps, 0, 0.8, g, eq=eq, coll=O.COLL_MRT, rates=O.mrt_rates(0.8))
    on = nt != 0
    err = float((np.abs(fg[:, on] - fo[:, on]) / W[:, None]).max())
    print(f"{state} {dtype}: {err:.3e}")
    assert err <= TOL[dtype] * scale
