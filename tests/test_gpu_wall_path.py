"""lbm_set_wall_path chooses the kernel that steps in every context: also where walls slide or a periodic
lattice is narrower than its ghost columns, which step in a form of the kernel of their own."""
import numpy as np
import pytest

from paper_2505_22256_gb300 import lbm, scenarios as S

pytestmark = pytest.mark.gpu


def narrow(nx=6, ny=40):
    solid = np.zeros((ny, nx), np.uint8)
    solid[17:20, 2] = 1
    r = np.random.default_rng(nx).uniform(0.3, 0.8, (2, ny, nx)) * (solid == 0)
    return S.Scenario("narrow", solid, r[0], r[1], bc_x="periodic", bc_y="wall", lam=0.6)


CASES = {"ordinary": lambda: [S.cylinder_droplet(96, lam=0.6)],
         "sliding": lambda: [S.couette_channel(50, 40, lam=0.6)],
         "narrow": lambda: [narrow()],
         "sliding_beside_ordinary": lambda: [S.couette_channel(50, 40, lam=0.6), S.cylinder_droplet(96, lam=0.6)]}


@pytest.mark.parametrize("storage", ["f32", "f16", "f64"])
@pytest.mark.parametrize("name", list(CASES))
def test_wall_path_picks_the_kernel(name, storage):
    import torch
    from capture_util import launches

    stream = torch.cuda.Stream()
    kernels, states = [], []
    for inline in (0, 1):
        lat = lbm.Lattice(CASES[name](), storage, stream.cuda_stream)
        lbm.lbm_set_wall_path(lat.ctx, inline)
        assert lat.info()["wall_inline"] == inline
        lat.step(20)
        states.append(np.concatenate([lat.populations(i).ravel() for i in range(lat.info()["ncases"])]))
        kernels.append(launches(stream, lambda: lat.step(1)))
        lat.close()
    assert [len(k) for k in kernels] == [1, 1]
    assert kernels[0][0][0] != kernels[1][0][0], kernels
    # 20 steps of sums associated in two ways; in 16-bit storage a value near a rounding boundary moves by
    # one unit of the last place of f - w rho0 (2^-11 of at most 1), and later steps average it away
    tol = {"f64": 20 * 4 * 2.0 ** -52, "f32": 20 * 4 * 2.0 ** -23, "f16": 20 * 2.0 ** -11}[storage]
    assert np.max(np.abs(states[0] - states[1])) <= tol * np.max(np.abs(states[0]))
