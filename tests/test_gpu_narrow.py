"""Periodic lattices narrower than the ghost columns of both sides together: every node within four
columns of an edge is repeated beyond the opposite edge, for both edges where it lies near both."""
import numpy as np
import pytest

import oracle
from paper_2505_22256_gb300 import lbm, scenarios as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [1, 16])
@pytest.mark.parametrize("nx", [5, 6, 7, 8])
def test_narrow_periodic_lattice_matches_oracle(nx, rows):
    rng, ny = np.random.default_rng(nx), 24
    solid = np.zeros((ny, nx), np.uint8)
    solid[0] = solid[-1] = 1
    solid[11, 2] = 1
    r = rng.uniform(0.3, 0.8, (2, ny, nx)) * (solid == 0)
    sc = S.Scenario("narrow", solid, r[0], r[1], bc_x="periodic", bc_y="wall")
    lat = lbm.Lattice(sc, "f64")
    lbm.lbm_set_launch(lat.ctx, 64, rows)
    lat.step(9)
    cfg = oracle.Config(nx=nx, ny=ny, **sc.params())
    f = oracle.run(cfg, solid, oracle.init(cfg, solid, r[0], r[1]), 9)
    assert np.max(np.abs(lat.populations() - f)) <= 1e-12
