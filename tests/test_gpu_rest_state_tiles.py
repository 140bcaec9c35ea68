"""The setter's tiles: blocks of 128 or, on narrow lattices, 32 columns by 1 to 16 rows (3-D: 1 to 16 planes),
as many as fill the GPU.  A small lattice is spread over one block per row, and the state is numpy's products at the
edges of every tile shape."""
import numpy as np
import pytest

from paper_2505_22256_gb300 import lbm, lbm3d, scenarios as S

pytestmark = pytest.mark.gpu

W9 = [4.0 / 9.0] + [1.0 / 9.0] * 4 + [1.0 / 36.0] * 4
W19 = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
REAL = {"f64": np.float64, "f32": np.float32}


def made(shape, seed):
    rng = np.random.default_rng(seed)
    solid = (rng.random(shape) < 0.15).astype(np.uint8)
    solid[tuple(n // 2 for n in shape)] = 0
    return solid, rng.uniform(0.02, 1.1, shape), rng.uniform(0.02, 1.1, shape)


# rows per block on 152 SMs: 1, 1, 1; 2, 16 (32 columns); 2, 8, 16 (128 columns)
@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny", [(29, 40), (30, 61), (31, 61), (30, 9731), (17, 80001), (126, 2437), (127, 5003), (601, 4001)])
def test_tiles_2d(nx, ny, storage):
    solid, a, b = made((ny, nx), nx)
    lat = lbm.Lattice(S.Scenario("tiles", solid, np.ones(a.shape), np.ones(a.shape), bc_x="periodic", bc_y="periodic"), storage)
    lbm.lbm_set_densities(lat.ctx, 0, a, b)
    f = lat.populations()
    for k, r in enumerate((a, b)):
        for i, w in enumerate(W9):
            assert np.array_equal(f[k, i], (w * r * (solid == 0)).astype(REAL[storage]).astype(np.float64)), (k, i)


@pytest.mark.parametrize("storage", ["f64", "f32"])
@pytest.mark.parametrize("nx,ny,nz", [(33, 9, 40), (64, 65, 31), (100, 99, 141)])
def test_tiles_3d(nx, ny, nz, storage):
    solid, a, b = made((nz, ny, nx), nx)
    lat = lbm3d.Lattice3(solid, np.ones(a.shape), np.ones(a.shape), {}, storage)
    lat.set_densities(a, b)
    f = lat.populations()
    for k, r in enumerate((a, b)):
        for i, w in enumerate(W19):
            assert np.array_equal(f[k, i], (w * r * (solid == 0)).astype(REAL[storage]).astype(np.float64)), (k, i)


@pytest.mark.parametrize("nx,ny", [(40, 300), (96, 96), (9, 120), (350, 100)])
def test_small_lattices_take_a_block_per_row(nx, ny):
    import torch
    from capture_util import launches

    solid, a, b = made((ny, nx), 1)
    stream = torch.cuda.Stream()
    lat = lbm.Lattice(S.Scenario("rows", solid, a, b), "f32", stream.cuda_stream)
    da, db = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    torch.cuda.synchronize()
    (_, blocks, threads), = launches(stream, lambda: lbm.lbm_set_densities_all(lat.ctx, da, db, on_device=True))
    assert blocks == ny * -(-nx // (threads - 2))
    lat.close()
