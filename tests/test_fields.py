"""Density, velocity, mass and momentum from the stored populations.

The fields are formed per lane of a work group: FP64 storage through exact fixed-point
moments widened with integer instructions, the other formats through FP32 pairs, and nodes
whose density lies outside those forms' ranges in plain FP64. Sizes cover one lane, the
edges of a work group and several of them; scales cover both forms and the change between
them; the reference sums the exported populations in long double.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import oracle as O
from paper_1611_02445_gb300 import inputs as I

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fixed_point_to_double_is_the_nearest(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "fields_host_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-o", exe,
                    os.path.join(ROOT, "tests", "fields_host_check.cpp")], check=True, capture_output=True)
    assert subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout.strip() == "0"


def _geometry(size):
    if size == "one":
        nt = np.zeros((4, 4, 4), np.uint8)
        nt[2, 1, 3] = 1
        return nt
    if size == "full":            # four full tiles: every lane of one work group
        return np.ones((4, 4, 16), np.uint8)
    if size == "ragged":          # full tiles that do not fill groups, cut at every end
        return np.ones((9, 7, 13), np.uint8)
    return I.random_box(24, 20, 28, 0.45, seed=4)


@pytest.mark.gpu
@pytest.mark.parametrize("eq", [O.EQ_QCOMPR, O.EQ_INCOMPR])
@pytest.mark.parametrize("scale", [1.0, 0.3, 1.72, 2.6])
@pytest.mark.parametrize("size", ["one", "full", "ragged", "sparse"])
@pytest.mark.parametrize("dtype", ["f64", "f32", "f16s"])
def test_fields_match_long_double_sums(dtype, size, scale, eq):
    from paper_1611_02445_gb300 import lbm
    nt = _geometry(size)
    f0 = scale * I.random_populations(nt, 0.08, seed=9)
    g = (3e-5, -2e-5, 1e-5)
    gf = I.body_force_field(nt, 2e-5, 1e-6) if scale == 1.0 else None
    with lbm.Lattice(nt, dtype, 0) as L:
        L.set_params(0.8, g, gf)
        L.set_model(eq, 0)
        L.set_f(f0)
        f = L.get_f().astype(np.longdouble)
        fields = {out: L.macroscopic(out) for out in (True, False)}
        mass, mom = L.reduce()
    on = nt != 0
    c = np.array([v for v in O.lattice()[0]], dtype=np.longdouble).reshape(-1, 3)
    Fx = (gf if dtype == "f64" else gf.astype(np.float32).astype(np.float64)) if gf is not None else np.full(nt.shape, g[0])
    F = [Fx.astype(np.longdouble), np.longdouble(g[1]), np.longdouble(g[2])]
    rho = np.where(on, f.sum(0), 0)
    mo = [np.where(on, np.tensordot(c[:, a], f, 1) - F[a] / 2, 0) for a in range(3)]
    u = np.stack([m if eq == O.EQ_INCOMPR else np.divide(m, rho, where=on, out=np.zeros_like(m)) for m in mo])
    # moments: FP64 storage rounds a population outside [2^-6, 16) to 2^-59 and the result
    # once; the pairs keep 2^-44 of sum |h| (the exported f = w + h itself is rounded to
    # 2^-53, 19 times). The division and the FP32 result round once each.
    habs = float(np.abs(f - O.lattice()[1].reshape(-1, 1, 1, 1))[:, on].sum(0).max())
    a64 = 19 * 2.0 ** -59 if dtype == "f64" else 2.0 ** -44 * habs + 19 * 2.0 ** -54
    for out64 in (True, False):
        r, v = fields[out64]
        ulp = 2.0 ** -52 if out64 else 2.0 ** -23
        assert (r[~on] == 0).all() and (v[:, ~on] == 0).all()
        assert (np.abs(r - rho) <= ulp * np.abs(rho) + a64).all()
        lo = float(rho[on].min()) if eq == O.EQ_QCOMPR else 1.0
        assert (np.abs(v - u) <= ulp * np.abs(u) + 2 * a64 / lo).all()
    n = int(on.sum())
    assert abs(mass - float(rho.sum())) <= n * (a64 + 2.0 ** -52 * float(rho[on].max()))
    for a in range(3):
        assert abs(mom[a] - float(mo[a].sum())) <= n * (a64 + 2.0 ** -52 * float(np.abs(mo[a]).max()))


@pytest.mark.gpu
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_a_non_finite_population_shows_in_its_node_alone(dtype, bad):
    from paper_1611_02445_gb300 import lbm
    nt = _geometry("ragged")
    f0 = I.random_populations(nt, 0.05, seed=2)
    f0[7, 3, 2, 5] = bad
    with lbm.Lattice(nt, dtype, 0) as L:
        L.set_params(0.8)
        L.set_f(f0)
        for out in (True, False):
            rho, u = L.macroscopic(out)
            here = np.zeros(nt.shape, bool)
            here[3, 2, 5] = True
            assert not np.isfinite(rho[here]).any() and np.isfinite(rho[~here]).all()
            assert np.isfinite(u[:, ~here]).all()
        with pytest.raises(lbm.LBMError, match="LBM_ENONFINITE"):
            L.reduce()
