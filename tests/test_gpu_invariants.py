"""The last digits of lbm_reduce, against exactly rounded sums of the stored populations.

Mass: the final rounding is half a unit in the last place, at most 2^-53 of the mass; the rounding
of the blocks' partial sums and of their tree (errors kept over its last three levels) is random
and stays below half of that again. Momentum: a state whose momentum cancels exactly, pair of
nodes by pair, leaves only the half force, rounded a few times.
"""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_1611_02445_gb300 import inputs as I
from paper_1611_02445_gb300 import lbm

pytestmark = pytest.mark.gpu
C, W, OPP = O.lattice()
C = np.asarray(C).reshape(-1, 3)


def _stored(f, dtype):
    """What the context keeps of f [19, n], as doubles: f itself, or h = f - w rounded."""
    if dtype == "f64":
        return f
    h = f - W[:, None]
    if dtype == "f32":
        return h.astype(np.float32).astype(np.float64)
    return (h * 4096.0).astype(np.float16).astype(np.float64) / 4096.0


@pytest.mark.parametrize("dtype", ["f64", "f32", "f16s"])
@pytest.mark.parametrize("size,seed", [((4, 4, 4), 1), ((9, 7, 13), 2), ((40, 40, 40), 3), ((52, 44, 60), 4),
                                       ((60, 60, 61), 5), ((72, 70, 66), 6), ((80, 80, 80), 7), ((96, 64, 96), 8)])
def test_mass_is_rounded_about_once(dtype, size, seed):
    nt = I.random_box(*size, p_solid=0.3, seed=seed)
    f0 = I.random_populations(nt, 0.05, seed=seed + 20)
    with lbm.Lattice(nt, dtype, 0) as L:
        L.set_params(0.8, (1e-5, 0, 0))
        L.set_f(f0)
        mass, _ = L.reduce()
    on = nt != 0
    v = _stored(f0[:, on], dtype)
    n = 0 if dtype == "f64" else int(on.sum())
    exact = math.fsum([float(n)] + v.ravel().tolist())
    assert abs(mass - exact) <= 1.5 * 2.0 ** -53 * exact


@pytest.mark.parametrize("dtype", ["f64", "f64n", "f32", "f16s"])
@pytest.mark.parametrize("size", [(32, 32, 32), (64, 64, 64), (128, 128, 64)])
def test_momentum_that_cancels_leaves_the_half_force(dtype, size):
    nx, ny, nz = size
    nt = np.ones((nz, ny, nx), np.uint8)
    rng = np.random.default_rng(7)
    a = W * (1.0 + 0.1 * (2.0 * rng.random(19) - 1.0))
    f0 = np.empty((19, nz, ny, nx))
    f0[..., 0::2] = a[:, None, None, None]
    f0[..., 1::2] = a[list(OPP)][:, None, None, None]    # the opposite momentum
    g = (1.1e-5, -0.7e-5, 0.3e-5)
    with lbm.Lattice(nt, dtype, 0) as L:
        L.set_params(0.8, g)
        L.set_f(f0)
        _, momentum = L.reduce()
    for c in range(3):
        exact = -0.5 * nx * ny * nz * g[c]
        assert abs(momentum[c] - exact) <= 4 * 2.0 ** -53 * abs(exact)


@pytest.mark.parametrize("n", [24, 100, 128])
def test_small_fp32_populations_beside_large_ones_keep_their_bits(n):
    """Populations h from 1e-9 to 5e-3 of either sign. The FP64 sum of n^3 node momenta of standard
    deviation sqrt(10) s (s of h) in about 20 levels rounds by about 2^-54 sqrt(20) times the
    random walk sqrt(10) s n^1.5, 7 units of 2^-53 s n^1.5; the bar is four times that."""
    rng = np.random.default_rng(n)
    h = 10.0 ** rng.uniform(-9, -2.3, (19, n, n, n)) * rng.choice([-1.0, 1.0], (19, n, n, n))
    f0 = W[:, None, None, None] + h
    with lbm.Lattice(np.ones((n, n, n), np.uint8), "f32", 0b111) as L:
        L.set_params(0.8)
        L.set_f(f0)
        _, momentum = L.reduce()
    v = _stored(f0.reshape(19, -1), "f32")
    for c in range(3):
        terms = np.concatenate([C[i, c] * v[i] for i in range(19) if C[i, c]])
        exact = math.fsum(terms)
        assert abs(momentum[c] - exact) <= 28 * 2.0 ** -53 * float(v.std()) * n ** 1.5
