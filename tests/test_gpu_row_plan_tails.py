"""Default lists that run more items than are resident at once: the guided list with 16-row tails, or with 8-row
tails where those promise at least 2 %; items are claimed from the counter, and the state is the one of a single
long item per column window, to the rounding of the row order."""
import numpy as np
import pytest

from paper_2505_22256_gb300 import lbm, scenarios as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make,storage,tail", [
    (lambda: [S.cylinder_droplet(1024, seed=k) for k in range(7)], "f16", -16),
    (lambda: [S.cylinder_droplet(1024, seed=k) for k in range(7)], "f32", -16),
    (lambda: [S.cylinder_in_box(seed=k) for k in range(14)], "f32", -8),
    (lambda: [S.cylinder_in_box(seed=k) for k in range(14)], "f16", -8)])
def test_guided_default(make, storage, tail):
    scs = make()
    lat = lbm.Lattice(scs, storage)
    info = lat.info()
    assert info["work_items"] > info["grid_blocks"]  # not all resident at once: the rest are claimed
    lat.step(3)
    got = [lat.populations(i) for i in range(len(scs))]
    lbm.lbm_set_launch(lat.ctx, info["block_threads"], tail)
    same = lat.info()
    assert (same["block_rows"], same["work_items"]) == (info["block_rows"], info["work_items"])
    lat.close()
    one = lbm.Lattice(scs, storage)
    lbm.lbm_set_launch(one.ctx, info["block_threads"], 4096)
    one.step(3)
    # three steps of sums in another order; in 16-bit storage a value near a rounding boundary moves by one
    # unit in the last place (2^-11 of at most 0.6), and its neighbours' next values by less
    tol = 3 * 4 * 2.0 ** -23 if storage == "f32" else 3 * 2.0 ** -11
    for i, a in enumerate(got):
        b = one.populations(i)
        assert np.max(np.abs(a - b)) <= tol * np.max(np.abs(b)), i
    one.close()


@pytest.mark.parametrize("make", [lambda: [S.cylinder_droplet(96)], lambda: [S.cylinder_droplet(640, nx=1500, R=90, r=100)],
                                  lambda: [S.flat_droplet(64, 48, r=12), S.cylinder_droplet(300)]])
def test_small_default_runs_all_items_at_once(make):
    lat = lbm.Lattice(make(), "f32")
    assert lat.info()["work_items"] == lat.info()["grid_blocks"]
    lat.close()
