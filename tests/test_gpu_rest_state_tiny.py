"""Densities whose population w rho of the diagonal directions rounds to 0 while that of the axes or of
the rest population does not (FP32 below 1e-43, FP64 below 1e-321): every stored population is the
rounded product w_i rho, as numpy forms it, also where only one component is that small."""
import numpy as np
import pytest

from paper_2505_22256_gb300 import lbm, lbm3d, scenarios as S

pytestmark = pytest.mark.gpu

W9 = [4.0 / 9.0] + [1.0 / 9.0] * 4 + [1.0 / 36.0] * 4
W19 = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
REAL = {"f64": (np.float64, 5e-324), "f32": (np.float32, 1.4e-45)}


def densities(shape, least, seed):
    """Multiples of the least denormal, ordinary values and zeros."""
    rng = np.random.default_rng(seed)
    r = least * rng.integers(1, 64, shape).astype(np.float64)
    u = rng.random(shape)
    r[u < 0.3] = rng.uniform(0.1, 1.0, shape)[u < 0.3]
    r[u > 0.9] = 0.0
    return r


@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_tiny_densities_2d(storage):
    real, least = REAL[storage]
    solid = (np.random.default_rng(1).random((19, 130)) < 0.15).astype(np.uint8)
    a, b = densities(solid.shape, least, 2), densities(solid.shape, least, 3)
    lat = lbm.Lattice(S.Scenario("tiny", solid, np.ones(solid.shape), np.ones(solid.shape), bc_x="periodic", bc_y="wall"), storage)
    lbm.lbm_set_densities_all(lat.ctx, a, b)
    want = np.stack([[(w * r * (solid == 0)).astype(real).astype(np.float64) for w in W9] for r in (a, b)])
    assert np.array_equal(lat.populations(), want)


@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_tiny_densities_3d(storage):
    real, least = REAL[storage]
    solid = (np.random.default_rng(4).random((18, 9, 33)) < 0.15).astype(np.uint8)
    a, b = densities(solid.shape, least, 5), densities(solid.shape, least, 6)
    lat = lbm3d.Lattice3(solid, np.ones(solid.shape), np.ones(solid.shape), {}, storage)
    lat.set_densities(a, b)
    want = np.stack([[(w * r * (solid == 0)).astype(real).astype(np.float64) for w in W19] for r in (a, b)])
    assert np.array_equal(lat.populations(), want)
