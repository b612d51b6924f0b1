"""The FP16 step stages each work group's data blocks whole and gathers only the pulls from other
groups; a geometry in which some group has more of those than fit its list takes the pulls
node by node. Both against the oracle, in the step and the propagation kernel: one node, one
group, ragged and sparse boxes, a box whose layers cross tile faces everywhere (too many
imports for the lists), with walls, inlets and outlets, and a slab's ghost planes.

Bars: FP16 rounding of the model tests (3e-3 of w); propagation moves stored values, exactly.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1611_02445_gb300 import inputs as I
from paper_1611_02445_gb300 import lbm

pytestmark = pytest.mark.gpu
_, W, _ = O.lattice()


def _geometry(name):
    if name == "one":
        nt = np.zeros((4, 4, 4), np.uint8)
        nt[1, 2, 3] = 1
        return nt, 0
    if name == "group":
        return np.ones((4, 4, 16), np.uint8), 0b111
    if name == "ragged":
        return np.ones((13, 9, 22), np.uint8), 0
    if name == "boundary":
        return I.random_box(28, 24, 20, 0.3, seed=3, boundary=True), 0b101
    if name == "sparse":
        return I.random_box(40, 36, 32, 0.85, seed=4), 0b111
    nt = np.ones((24, 24, 64), np.uint8)     # layers: y = 3 and 0 of neighbouring tiles
    nt[:, 1::4] = nt[:, 2::4] = 0
    return nt, 0b111


@pytest.mark.parametrize("name", ["one", "group", "ragged", "boundary", "sparse", "layers"])
def test_fp16_step_matches_oracle(name):
    nt, per = _geometry(name)
    f0 = I.random_populations(nt, 0.03, seed=5)
    g, u_in = (2e-5, -1e-5, 1e-5), (0.02, 0.0, 0.0)
    with lbm.Lattice(nt, "f16s", per) as L:
        L.set_params(0.8, g, None, u_in, 1.0)
        L.set_f(f0)
        L.step(9)
        fg = L.get_f()
    fo = O.run(f0, nt, 9, per, 0.8, g, None, u_in, 1.0)
    on = nt != 0
    assert float((np.abs(fg[:, on] - fo[:, on]) / W[:, None]).max()) <= 3e-3


@pytest.mark.parametrize("name", ["one", "group", "ragged", "boundary", "sparse", "layers"])
def test_fp16_propagation_moves_stored_values(name):
    nt, per = _geometry(name)
    f0 = I.random_populations(nt, 0.2, seed=6)
    f0[:, nt == 0] = np.nan
    with lbm.Lattice(nt, "f16s", per) as L:
        L.set_params(0.8)
        L.set_f(f0)
        s = L.get_f()                                  # as stored
        L.step_kernel(lbm.KERNEL_PROPAGATE, 3)
        fg = L.get_f()
    c = np.asarray(O.lattice()[0]).reshape(-1, 3)
    opp = [int(np.flatnonzero((c == -v).all(1))[0]) for v in c]
    on = nt != 0
    for _ in range(3):
        new = s.copy()
        for i in range(1, 19):
            src = np.roll(s[i], tuple(c[i][::-1]), (0, 1, 2))
            ok = np.roll(on, tuple(c[i][::-1]), (0, 1, 2))
            for a in range(3):
                if c[i][a] and not per >> a & 1:
                    sl = [slice(None)] * 3
                    sl[2 - a] = 0 if c[i][a] > 0 else -1
                    ok[tuple(sl)] = False
            # a bounced value keeps its stored h = f - w of the opposite direction (same weight)
            new[i] = np.where(ok, src, s[opp[i]])
        s = np.where(on, new, np.nan)
    assert np.array_equal(fg[:, on], s[:, on])
