"""FP64 lists in 64-column blocks.  Three such blocks run on an SM in little more than the time of one, so lattices
with rows enough for that take the shorter items, and every list gives the state of one long item per window."""
import numpy as np
import pytest

from paper_2505_22256_gb300 import lbm, scenarios as S

pytestmark = pytest.mark.gpu


def box(nx, ny):
    solid = np.zeros((ny, nx), np.uint8)
    solid[ny // 3:ny // 3 + 4, nx // 2:nx // 2 + 4] = 1
    r = np.random.default_rng(nx).uniform(0.3, 0.8, (2, ny, nx)) * (solid == 0)
    return S.Scenario("box", solid, r[0], r[1], bc_x="periodic", bc_y="wall", lam=0.6)


@pytest.mark.parametrize("shapes", [[(50, 100)] * 64, [(602, 581)], [(56, 588)] * 11, [(56, 4000)]])
def test_short_items_fill_the_sms(shapes):
    import torch

    scs = [box(*s) for s in shapes]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    out = []
    for rows in (0, 8192):
        lat = lbm.Lattice(scs, "f64")
        assert lat.info()["block_threads"] == 64
        if rows:
            lbm.lbm_set_launch(lat.ctx, 64, rows)
        else:
            assert 2.5 * sms <= lat.info()["work_items"] <= 3 * sms, lat.info()
        lat.step(3)
        out.append([lat.populations(i) for i in range(len(scs))])
        lat.close()
    for a, b in zip(*out):  # three steps of sums in another order: a few roundings of the largest value each
        assert np.max(np.abs(a - b)) <= 3 * 4 * 2.0 ** -52 * np.max(np.abs(b))
