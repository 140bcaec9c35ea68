"""The state that new densities give, f = f^eq(rho_k, 0), against numpy's products w_i rho_k: the same
bits in FP64 and FP32 storage, on lattices whose width, height and depth sit at the edges of the
setter's tiles (126 columns by 16 rows; 32 x 8 columns by 16 planes), with densities from ordinary
ones down to the smallest normal FP32 values."""
import numpy as np
import pytest

from paper_2505_22256_gb300 import lbm, lbm3d, scenarios as S

pytestmark = pytest.mark.gpu

W9 = [4.0 / 9.0] + [1.0 / 9.0] * 4 + [1.0 / 36.0] * 4
W19 = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
REAL = {"f64": np.float64, "f32": np.float32}


def densities(shape, seed):
    rng = np.random.default_rng(seed)
    r = rng.uniform(0.02, 1.1, shape)
    small = rng.random(shape) < 0.1
    r[small] = 10.0 ** rng.uniform(-37.0, -25.0, int(small.sum()))
    return r


def mask(shape, seed):
    return (np.random.default_rng(seed).random(shape) < 0.15).astype(np.uint8)


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny,bc_x,bc_y", [(5, 5, "periodic", "periodic"), (7, 16, "periodic", "wall"),
                                             (125, 17, "wall", "periodic"), (126, 33, "periodic", "wall"),
                                             (127, 15, "wall", "wall"), (253, 6, "periodic", "periodic")])
def test_rest_state_2d(nx, ny, bc_x, bc_y, storage):
    solid = mask((ny, nx), nx)
    solid[2, 2] = 0
    a, b = densities((ny, nx), 1), densities((ny, nx), 2)
    sc = S.Scenario("rest", solid, np.ones((ny, nx)), np.ones((ny, nx)), bc_x=bc_x, bc_y=bc_y)
    lats = [lbm.Lattice(sc, storage) for _ in range(2)]
    lbm.lbm_set_densities(lats[0].ctx, 0, a, b)
    lbm.lbm_set_densities_all(lats[1].ctx, a, b)
    want = np.stack([[(w * r * (solid == 0)).astype(REAL[storage]).astype(np.float64) for w in W9] for r in (a, b)])
    for lat in lats:
        assert np.array_equal(lat.populations(), want)


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny,nz", [(5, 5, 5), (31, 8, 16), (32, 9, 17), (33, 7, 33), (64, 16, 6)])
def test_rest_state_3d(nx, ny, nz, storage):
    solid = mask((nz, ny, nx), nx)
    solid[2, 2, 2] = 0
    a, b = densities((nz, ny, nx), 3), densities((nz, ny, nx), 4)
    lat = lbm3d.Lattice3(solid, np.ones(solid.shape), np.ones(solid.shape), {}, storage)
    lat.set_densities(a, b)
    want = np.stack([[(w * r * (solid == 0)).astype(REAL[storage]).astype(np.float64) for w in W19] for r in (a, b)])
    assert np.array_equal(lat.populations(), want)
