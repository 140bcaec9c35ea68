"""The setter's state against an independent way to the same one: lbm_set_populations of w_i rho formed in FP64 on the host
(the general state kernel: its own bounce-back, outlet and shift rules).  Populations, the populations after three steps
(which pull the ghost columns) and the fields agree bit for bit, in 16-bit storage with a shift, without one and with
unequal ones, with open columns whose last two hold solid nodes, and over uneven ensembles."""
import numpy as np
import pytest

from paper_2505_22256_gb300 import lbm, lbm3d, scenarios as S

pytestmark = pytest.mark.gpu

W9 = np.array([4.0 / 9.0] + [1.0 / 9.0] * 4 + [1.0 / 36.0] * 4)
W19 = np.array([1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12)


def case(nx, ny, bc_x, bc_y, seed, **kw):
    rng = np.random.default_rng(seed)
    solid = (rng.random((ny, nx)) < 0.12).astype(np.uint8)
    solid[ny // 2] = 0
    if bc_x == "open":
        solid[:, :2] = 0
        solid[::3, nx - 2] = 1
        solid[1::4, nx - 1] = 1
    rho = rng.uniform(0.03, 1.1, (2, ny, nx)) * (solid == 0)
    return S.Scenario("pin", solid, rho[0], rho[1], bc_x=bc_x, bc_y=bc_y, lam=0.7, **kw)


OPEN = dict(u_in=0.01, rho_in=(0.06, 1.0))
CASES = {
    "periodic": [(131, 37, "periodic", "periodic", {})],
    "walled": [(254, 18, "wall", "wall", {})],
    "open_copy": [(150, 33, "open", "wall", OPEN)],
    "open_pressure": [(40, 21, "open", "periodic", dict(OPEN, outlet="pressure"))],
    "narrow": [(6, 50, "periodic", "wall", {})],
    "sliding": [(50, 30, "periodic", "wall", dict(u_wall=(-0.01, 0.02)))],
    "uneven": [(131, 77, "periodic", "wall", {}), (8, 8, "periodic", "periodic", {}), (300, 20, "open", "wall", OPEN),
               (29, 200, "wall", "wall", {}), (6, 31, "periodic", "wall", {})],
    "all_narrow": [(30, 17, "periodic", "wall", {}), (5, 90, "wall", "periodic", {}), (29, 31, "open", "wall", OPEN)],
}
SHIFTS = [("f64", (0.0, 0.0)), ("f32", (0.06, 0.06)), ("f16", (0.06, 0.06)), ("f16", (0.0, 0.0)), ("bf16", (0.37, 0.11)), ("bf16", (0.0, 1.0))]


@pytest.mark.parametrize("storage,shift", SHIFTS)
@pytest.mark.parametrize("name", list(CASES))
def test_densities_equal_populations_2d(name, storage, shift):
    scs = [case(nx, ny, bx, by, 10 * k + 1, rho0_store=shift, **kw) for k, (nx, ny, bx, by, kw) in enumerate(CASES[name])]
    plain = [case(nx, ny, bx, by, 10 * k + 1, rho0_store=shift, **kw) for k, (nx, ny, bx, by, kw) in enumerate(CASES[name])]
    for p in plain:  # every state below replaces this one
        p.rhoA0, p.rhoB0 = 0.5 * (p.solid == 0), 0.4 * (p.solid == 0)
    one, batch, ref, made = (lbm.Lattice(x, storage) for x in (plain, plain, plain, scs))
    for i, sc in enumerate(scs):
        lbm.lbm_set_densities(one.ctx, i, sc.rhoA0, sc.rhoB0)
        ref.set_populations(np.stack([W9[:, None, None] * r for r in (sc.rhoA0, sc.rhoB0)]), i)
    lbm.lbm_set_densities_all(batch.ctx, *(np.concatenate([getattr(sc, k).ravel() for sc in scs]) for k in ("rhoA0", "rhoB0")))
    for steps in (0, 3):
        for lat in (one, batch, ref, made):
            lat.step(steps)
        for i in range(len(scs)):
            want, fields = ref.populations(i), ref.fields(i)
            for lat in (one, batch, made):
                assert np.array_equal(lat.populations(i), want), (steps, i)
                assert all(np.array_equal(a, b) for a, b in zip(lat.fields(i), fields)), (steps, i)
    for lat in (one, batch, ref, made):
        lat.close()


@pytest.mark.parametrize("storage,shift", SHIFTS)
@pytest.mark.parametrize("nx,ny,nz", [(33, 9, 18), (5, 40, 7), (64, 8, 33)])
def test_densities_equal_populations_3d(nx, ny, nz, storage, shift):
    rng = np.random.default_rng(nx)
    solid = (rng.random((nz, ny, nx)) < 0.12).astype(np.uint8)
    rho = rng.uniform(0.03, 1.1, (2, nz, ny, nx)) * (solid == 0)
    params = {"lam": 0.7, "rho0_store": shift}
    flat = [c * (solid == 0) for c in (0.5, 0.4)]
    lat, ref = (lbm3d.Lattice3(solid, *flat, params, storage) for _ in range(2))
    made = lbm3d.Lattice3(solid, *rho, params, storage)
    lat.set_densities(*rho)
    ref.set_populations(np.stack([W19[:, None, None, None] * r for r in rho]))
    for steps in (0, 2):
        for x in (lat, ref, made):
            x.step(steps)
        want = ref.populations()
        assert np.array_equal(lat.populations(), want) and np.array_equal(made.populations(), want)
