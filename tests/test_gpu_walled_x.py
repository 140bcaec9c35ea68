"""Closed x (bc_x = wall) on lattices wider than one column window: the last window reaches columns
beyond the wall and beyond the ghost columns of the flags, which are solid like the wall itself."""
import numpy as np
import pytest

import oracle
from paper_2505_22256_gb300 import lbm, scenarios as S

pytestmark = pytest.mark.gpu

# absolute, densities up to 1.3: 30 steps x 9 populations x one rounding of the type, doubled by the forces
# (FP64: the bar of the narrow lattices); FP16: a storage rounding of the largest population (0.6) per step
BAR = {"f64": 1e-12, "f32": 30 * 9 * 2.0 ** -24 * 1.3 * 2, "f16": 30 * 2.0 ** -11 * 0.6}


def scenario(nx, ny):
    solid = np.zeros((ny, nx), np.uint8)
    solid[3:6, nx // 2 - 1:nx // 2 + 2] = 1
    solid[ny - 2, nx - 1] = 1
    y, x = np.mgrid[:ny, :nx]
    a = np.where((np.abs(x - 0.7 * nx) < 0.3 * nx) & (y > 7), 0.06, 1.0)
    rng = np.random.default_rng(nx)
    rho = np.stack([a, 1.06 - a]) * (1 + 1e-3 * rng.standard_normal((2, ny, nx))) * (solid == 0)
    return S.Scenario("walled", solid, rho[0], rho[1], bc_x="wall", bc_y="wall", lam=0.6)


@pytest.mark.parametrize("storage", ["f64", "f32", "f16"])
@pytest.mark.parametrize("width", [64, 128])
@pytest.mark.parametrize("nx", [5, 56, 97, 113, 121, 150, 233, 500, 1210])
def test_walled_x_matches_oracle(nx, width, storage):
    sc = scenario(nx, 21)
    lat = lbm.Lattice(sc, storage)
    lbm.lbm_set_launch(lat.ctx, width, 0)
    lat.step(30)
    rA, rB, ux, uy = lat.fields()
    d = lat.diagnostics()
    lat.close()
    cfg = oracle.Config(nx=nx, ny=21, **sc.params())
    f = oracle.run(cfg, sc.solid, oracle.init(cfg, sc.solid, sc.rhoA0, sc.rhoB0), 30)
    oA, oB, oux, ouy = oracle.fields(cfg, sc.solid, f)
    fl = sc.solid == 0
    assert max(np.max(np.abs(rA - oA)[fl]), np.max(np.abs(rB - oB)[fl])) <= BAR[storage]
    assert max(np.max(np.abs(ux - oux)), np.max(np.abs(uy - ouy))) <= BAR[storage]
    assert d["n_fluid"] == int(fl.sum())
