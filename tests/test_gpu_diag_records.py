"""Diagnostics of cases whose lists hold few and very many items (the reduction takes 256 records at a time,
a lane 8): sums, extrema and counts of the fields that the same state gives."""
import numpy as np
import pytest

from paper_2505_22256_gb300 import lbm, scenarios as S

pytestmark = pytest.mark.gpu


def scenario(nx, ny):
    rng = np.random.default_rng(nx * ny)
    solid = (rng.random((ny, nx)) < 0.05).astype(np.uint8)
    solid[ny // 2, nx // 2] = 0
    a = rng.uniform(0.2, 0.9, (2, ny, nx)) * (solid == 0)
    return S.Scenario("records", solid, a[0], a[1], bc_x="periodic", bc_y="wall", lam=0.6)


@pytest.mark.parametrize("storage", ["f64", "f32", "f16"])
@pytest.mark.parametrize("shapes", [[(9, 5000)], [(56, 257), (57, 3000), (5, 5)], [(30, 256)], [(2000, 40), (8, 9)]])
def test_diagnostics_of_long_lists(shapes, storage):
    scs = [scenario(*s) for s in shapes]
    lat = lbm.Lattice(scs, storage)
    lat.step(5)
    d, fields = lat.diagnostics_all(allow_unstable=True), lat.fields_all()
    for i, (sc, one) in enumerate(zip(scs, d)):
        fl = sc.solid == 0
        rA, rB, ux, uy = (f[fl] for f in fields[i])
        n = int(fl.sum())
        tot = rA + rB
        assert one["n_fluid"] == n and one == lat.diagnostics(i, allow_unstable=True)
        # FP64 sums of n values in two orders; rho_A + rho_B is rounded in the compute type before it weighs u
        eps = n * 2.0 ** -53
        lane = 2.0 ** -24 if storage != "f64" else 2.0 ** -53
        assert abs(one["mass_A"] - rA.sum()) <= eps * rA.sum() and abs(one["mass_B"] - rB.sum()) <= eps * rB.sum()
        for key, u in (("mom_x", ux), ("mom_y", uy)):
            assert abs(one[key] - (tot * u).sum()) <= (eps + lane) * (tot * np.abs(u)).sum()
        assert (one["rhoA_min"], one["rhoA_max"], one["rhoB_min"], one["rhoB_max"]) == (rA.min(), rA.max(), rB.min(), rB.max())
        speed = np.sqrt(ux * ux + uy * uy).max()
        assert abs(one["umax"] - speed) <= 4 * lane * speed
    lat.close()
