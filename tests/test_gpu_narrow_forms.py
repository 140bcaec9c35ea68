"""Lattices narrower than the ghost columns of both sides, beyond the FP64 state of a single one: FP32 and 16-bit
storage, both block widths, the fields pass and diagnostics, and an ensemble that puts a wide case into the same
form of the kernel."""
import numpy as np
import pytest

import oracle
from paper_2505_22256_gb300 import lbm, scenarios as S

pytestmark = pytest.mark.gpu

STEPS = 9
# absolute, densities up to 0.8: nine populations rounded once a step, doubled by the forces; 16-bit types: a storage
# rounding of the largest population (0.36 - w rho0, half a unit of 2^-11, 2^-8) in each of nine directions a step
BAR = {"f64": 1e-12, "f32": STEPS * 9 * 2.0 ** -24 * 2, "f16": STEPS * 9 * 2.0 ** -12 * 0.36, "bf16": STEPS * 9 * 2.0 ** -9 * 0.36}


def narrow(nx, ny=24):
    rng = np.random.default_rng(nx)
    solid = np.zeros((ny, nx), np.uint8)
    solid[0] = solid[-1] = 1
    solid[11, 2] = 1
    r = rng.uniform(0.3, 0.8, (2, ny, nx)) * (solid == 0)
    return S.Scenario("narrow", solid, r[0], r[1], bc_x="periodic", bc_y="wall", lam=0.8)


def check(lat, i, sc, bar):
    cfg = oracle.Config(nx=sc.nx, ny=sc.ny, **sc.params())
    f = oracle.run(cfg, sc.solid, oracle.init(cfg, sc.solid, sc.rhoA0, sc.rhoB0), STEPS)
    assert np.max(np.abs(lat.populations(i) - f)) <= bar
    want = oracle.fields(cfg, sc.solid, f)
    fl = sc.solid == 0
    for got, o in zip(lat.fields(i)[:2], want[:2]):
        assert np.max(np.abs(got - o)[fl]) <= bar
    d = lat.diagnostics(i)
    assert abs(d["mass_A"] - want[0][fl].sum()) <= bar * fl.sum() and d["n_fluid"] == int(fl.sum())


@pytest.mark.parametrize("storage", list(BAR))
@pytest.mark.parametrize("width", [64, 128])
@pytest.mark.parametrize("nx", [5, 6, 7, 8])
def test_narrow_lattice_in_every_storage(nx, width, storage):
    sc = narrow(nx)
    lat = lbm.Lattice(sc, storage)
    lbm.lbm_set_launch(lat.ctx, width, 0)
    lat.step(STEPS)
    check(lat, 0, sc, BAR[storage])
    lat.close()


@pytest.mark.parametrize("wall_inline", [0, 1])
@pytest.mark.parametrize("storage", list(BAR))
def test_narrow_case_beside_a_wide_one(storage, wall_inline):
    wide = S.cylinder_droplet(77, nx=131, R=12, r=15, lam=1.4)
    scs = [narrow(6), wide, narrow(5, 40)]
    lat = lbm.Lattice(scs, storage)
    lbm.lbm_set_wall_path(lat.ctx, wall_inline)
    lat.step(STEPS)
    for i in (0, 2):
        check(lat, i, scs[i], BAR[storage])
    alone = lbm.Lattice(wide, storage)  # the ordinary form
    lbm.lbm_set_wall_path(alone.ctx, wall_inline)
    alone.step(STEPS)
    a, b = lat.populations(1), alone.populations()
    assert np.max(np.abs(a - b)) <= BAR[storage]
    lat.close()
    alone.close()
