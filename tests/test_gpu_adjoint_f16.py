"""lbm_adjoint of FP16 storage, whose forward and recomputed steps run on the staged runs of the
workspace's copies: with import lists, on thin groups, and on a geometry whose lists overflow
(layers crossing tile faces). Checkpoint spacing changes nothing, the call ends in lbm_step's
state, and the gradients are those of the oracle's reverse steps through the states that the
context stored.

Bar: FP32 arithmetic, about 20 roundings of 2^-24 a reverse step of a value that all 12 steps
carry on: 1.5e-5 of the largest gradient. (dL/dtau is a sum of terms of both signs, whose rounding has
no such bound relative to the sum; the spacing test compares it bit for bit.)
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1611_02445_gb300 import inputs as I
from paper_1611_02445_gb300 import lbm

pytestmark = pytest.mark.gpu


def _geometry(name):
    if name == "lists":
        return I.sphere_pack(32, 5.0, 0.5, seed=8), 0b111
    if name == "boundary":
        return I.random_box(28, 24, 20, 0.3, seed=3, boundary=True), 0b110
    if name == "thin":
        return I.random_box(32, 32, 32, 0.95, seed=4), 0b111
    nt = np.ones((24, 24, 64), np.uint8)
    nt[:, 1::4] = nt[:, 2::4] = 0
    return nt, 0b111


@pytest.mark.parametrize("name", ["lists", "boundary", "thin", "layers"])
@pytest.mark.parametrize("every", [1, 5, 50])
def test_checkpoint_spacing_is_bitwise_the_same(name, every):
    nt, per = _geometry(name)
    out = []
    for k in (every, 7):
        with lbm.Lattice(nt, "f16s", per) as L:
            L.set_params(0.8, (0.0, 1e-5, 0.0), I.body_force_field(nt), (0.02, 0.0, 0.0), 1.0)
            L.init_equilibrium()
            loss, dg, dtau = L.adjoint(22, k, nt.shape[2] - 1)
            out.append((loss, dg, dtau, L.save_state()))
            L.init_equilibrium()
            L.step(22)
            assert L.save_state() == out[-1][3]
    assert out[0][0] == out[1][0] and out[0][2] == out[1][2] and np.array_equal(out[0][1], out[1][1])
    assert out[0][3] == out[1][3]


@pytest.mark.parametrize("name", ["lists", "boundary", "thin", "layers"])
def test_gradients_match_the_oracle_through_the_stored_states(name):
    nt, per = _geometry(name)
    T, plane, tau = 12, nt.shape[2] - 1, 0.8
    on = nt != 0
    gf = (I.body_force_field(nt, 1e-4, 1e-5)).astype(np.float32).astype(np.float64)
    g, u_in, rho_out = (0.0, 1e-4, -2e-4), (0.02, 0.01, 0.0), 1.01
    with lbm.Lattice(nt, "f16s", per) as L:
        L.set_params(tau, g, gf, u_in, rho_out)
        L.set_f(I.random_populations(nt, 0.05, seed=9))
        start = L.save_state()
        states = [L.get_f()]
        for _ in range(T):
            L.step(1)
            states.append(L.get_f())
        L.load_state(start)
        loss, dg, _ = L.adjoint(T, 5, plane)
    gb, g3, tb = np.zeros(nt.shape), np.zeros(3), np.zeros(1)
    want, lam = O.loss(states[T], nt, plane, g, gf, gb, g3)
    for t in range(T - 1, -1, -1):
        lam = O.step_adj(states[t], lam, nt, per, tau, g, gf, u_in, rho_out, gb, g3, tb)
    assert abs(loss - want) <= 1e-12
    assert np.abs(dg[on] - gb[on]).max() <= 1.5e-5 * np.abs(gb[on]).max()
    assert (dg[~on] == 0).all()
