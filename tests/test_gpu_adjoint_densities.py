"""lbm_adjoint over the densities and populations its FP64 arithmetic tells apart: populations
below 2^-6 and of 1 and more (moments in FP64 instead of 64-bit fixed point, which holds values
below 32), densities outside [5/8, 7/4) (1 / rho by division), and sums of 32 and more. FP64
arithmetic throughout ("f64n") takes any density; the double-float forward of "f64" is for
densities near 1 and is tested up to 3.

Bars: those of test_gpu_adjoint.py, gradients to 1e-10 of their largest entry; the velocity in
the loss does not scale with the density.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1611_02445_gb300 import inputs as I
from paper_1611_02445_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,rho", [("f64", 0.3), ("f64", 1.8), ("f64", 3.0), ("f64n", 0.3), ("f64n", 1.8),
                                       ("f64n", 3.0), ("f64n", 7.0), ("f64n", 15.5), ("f64n", 31.0), ("f64n", 33.0),
                                       ("f64n", 40.0), ("f64n", 47.0), ("f64n", 60.0), ("f64n", 100.0)])
@pytest.mark.parametrize("g", [(0.0, 0.0, 0.0), (0.0, 1e-4, -2e-4)])
def test_adjoint_matches_oracle_at_density(dtype, rho, g):
    nt = I.random_box(12, 8, 8, p_solid=0.25, seed=31)
    f0 = rho * I.random_populations(nt, 0.05, seed=32)
    gf = 1e-3 * (1 + 0.1 * np.random.default_rng(33).standard_normal(nt.shape))
    T, K, plane, tau = 7, 3, 11, 0.8
    with lbm.Lattice(nt, dtype, 0b111) as L:
        L.set_params(tau, g, gf)
        L.set_f(f0)
        Lg, dg, dtau = L.adjoint(T, K, plane)
    Lo, dg_o, _, dtau_o = O.adjoint(nt, T, plane, 0b111, tau, g, gf, f0=f0)
    on = nt != 0
    assert np.abs(dg[on] - dg_o[on]).max() <= 1e-10 * np.abs(dg_o[on]).max()
    assert abs(dtau - dtau_o) <= 1e-10 * abs(dtau_o)
    assert abs(Lg - Lo) <= 1e-12 / 3.0
