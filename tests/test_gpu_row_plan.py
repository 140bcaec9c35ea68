"""The default work list: short uniform items for lattices that cannot fill the GPU otherwise, a guided
list for large ones.  Whatever it picks, the state is the one that a single long item per column
window gives, to FP32 rounding of the row order, and the per-case lists of the fields pass cover every node once."""
import numpy as np
import pytest

from paper_2505_22256_gb300 import lbm, scenarios as S

pytestmark = pytest.mark.gpu

CASES = {
    "one_window": lambda: [S.cylinder_droplet(96, lam=0.6)],
    "two_rows_over": lambda: [S.cylinder_droplet(131, nx=121, R=12, r=15)],
    "narrow": lambda: [S.couette_channel(nx=9, ny=150)],
    "flat": lambda: [S.flat_droplet(900, 9, r=3.0)],
    "uneven": lambda: [S.flat_droplet(64, 48, r=12), S.cylinder_droplet(300), S.couette_channel(50, 7)],
    "guided": lambda: [S.cylinder_droplet(640, nx=1500, R=90, r=100)],
}


@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("name", list(CASES))
def test_default_list_matches_one_item_per_window(name, storage):
    scs = CASES[name]()
    if storage == "f64" and name == "guided":
        pytest.skip("FP64 on a large lattice only repeats the smaller ones")
    out = []
    for rows in (None, 1024):
        lat = lbm.Lattice(scs, storage)
        if rows:
            lbm.lbm_set_launch(lat.ctx, lat.info()["block_threads"], rows)
        info = lat.info()
        assert info["grid_blocks"] <= info["work_items"] and info["block_rows"] >= 1
        lat.step(21)
        out.append([[lat.populations(i) for i in range(len(scs))], [np.stack(f) for f in lat.fields_all()],
                    [lat.diagnostics(i) for i in range(len(scs))]])
        lat.close()
    # 21 steps of sums whose terms come in another order: a few roundings of the largest value per step
    tol = 21 * 4 * np.finfo(np.float64 if storage == "f64" else np.float32).eps
    for i, sc in enumerate(scs):
        a, b = out[0][0][i], out[1][0][i]
        assert np.max(np.abs(a - b)) <= tol * np.max(np.abs(b)), name
        fa, fb = out[0][1][i], out[1][1][i]
        assert np.max(np.abs(fa - fb)) <= tol * np.max(np.abs(fb)), name
        assert out[0][2][i]["n_fluid"] == int((sc.solid == 0).sum()) == out[1][2][i]["n_fluid"]
