"""The default form of the wall-list correction: called where cases with sliding walls, or narrow periodic
ones, hold most of the nodes; elsewhere inlined by size or by the share of wall-list nodes."""
import numpy as np
import pytest

from paper_2505_22256_gb300 import lbm, scenarios as S

pytestmark = pytest.mark.gpu


def narrow(nx, ny):
    r = np.random.default_rng(nx).uniform(0.3, 0.8, (2, ny, nx))
    return S.Scenario("narrow", np.zeros((ny, nx), np.uint8), r[0], r[1], bc_x="periodic", bc_y="wall")


@pytest.mark.parametrize("make,expect", [
    (lambda: [S.couette_channel(160, 200) for _ in range(12)], 0),  # more than 2^18 nodes
    (lambda: [S.couette_channel(50, 64)], 0),                       # 6 % wall-list nodes
    (lambda: [narrow(7, 60000)], 0),
    (lambda: [narrow(8, 60000)], 1),
    (lambda: [S.cylinder_droplet(600), S.couette_channel(50, 100)], 1),
    (lambda: [S.cylinder_droplet(96)] + [S.couette_channel(50, 400)], 0)])
def test_default_form(make, expect):
    lat = lbm.Lattice(make(), "f32")
    assert lat.info()["wall_inline"] == expect
    lat.close()
