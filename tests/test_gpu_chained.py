"""Steps of one call are chained launches: each may start before the one before it has ended.
A run in one call equals the same steps in calls of one each (never chained) bit for bit, in
graph replays and outside them, for geometries of one work group, of fewer groups than
resident CTAs and of several per CTA, in every storage format; so does a run on another
stream, and the adjoint, whose launches are chained across its two kernels, repeats itself.
"""
import numpy as np
import pytest

from paper_1611_02445_gb300 import inputs as I
from paper_1611_02445_gb300 import lbm

pytestmark = pytest.mark.gpu


def _run(nt, dtype, calls, stream=None):
    with lbm.Lattice(nt, dtype, 0b111, stream) as L:
        L.set_params(0.7, (2e-5, 1e-5, 0.0))
        L.init_equilibrium(1.0, (0.01, -0.02, 0.03))
        for n in calls:
            L.step(n)
        return L.save_state()


@pytest.mark.parametrize("n", [4, 24, 96])
@pytest.mark.parametrize("dtype", ["f64", "f64n", "f32", "f16s", "f16sr"])
def test_chained_steps_equal_single_steps(dtype, n):
    import torch
    nt = np.ones((n, n, n), np.uint8) if n == 4 else I.sphere_pack(n, 5.0, 0.5, seed=7)
    one = _run(nt, dtype, [1] * 37)
    assert _run(nt, dtype, [37]) == one              # two graph replays and five chained launches
    assert _run(nt, dtype, [15, 15, 7]) == one       # chained launches only
    assert _run(nt, dtype, [37], torch.cuda.Stream()) == one


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("every", [1, 4, 11, 50])
def test_adjoint_checkpoint_spacing_is_bitwise_the_same(dtype, every):
    nt = I.sphere_pack(32, 5.0, 0.5, seed=8)
    out = []
    for k in (every, 7):
        with lbm.Lattice(nt, dtype, 0b111) as L:
            L.set_params(0.8, (1e-5, 0, 0), I.body_force_field(nt))
            L.init_equilibrium()
            loss, dg, dtau = L.adjoint(22, k, 31)
            out.append((loss, dg, dtau, L.save_state()))
            L.init_equilibrium()
            L.step(22)
            assert L.save_state() == out[-1][3]      # the call ends in s_T, as lbm_step
    assert out[0][0] == out[1][0] and out[0][2] == out[1][2] and np.array_equal(out[0][1], out[1][1])
    assert out[0][3] == out[1][3]
