"""Steps inside a user's own stream capture.  The step chain is launched as programmatic dependent
launches; captured behind a copy and a setter and before a fields pass and a copy, and replayed three
times, it gives the bits of the uncaptured calls (2-D with a sliding-wall case, 3-D)."""
import numpy as np
import pytest

from paper_2505_22256_gb300 import lbm, lbm3d, scenarios as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_captured_steps_2d(storage):
    import torch

    scs = [S.cylinder_droplet(96, lam=0.6), S.couette_channel(50, 40)]
    stream = torch.cuda.Stream()
    ref, lat = lbm.Lattice(scs, storage), lbm.Lattice(scs, storage, stream.cuda_stream)
    src = [torch.from_numpy(np.concatenate([getattr(s, k).ravel() for s in scs])).cuda() for k in ("rhoA0", "rhoB0")]
    dst = [torch.empty_like(x) for x in src]
    out = torch.zeros(4, src[0].numel(), dtype=torch.float64, device="cuda")
    last = torch.zeros_like(out)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        for d, x in zip(dst, src):
            d.copy_(x)
        lbm.lbm_set_densities_all(lat.ctx, *dst, on_device=True)
        lat.step(18)
        lbm.lbm_fields_all(lat.ctx, *out, on_device=True)
        last.copy_(out)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    ref.step(18)
    want = np.stack([np.concatenate([f[q].ravel() for f in ref.fields_all()]) for q in range(4)])
    assert np.array_equal(last.cpu().numpy(), want)


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_captured_steps_3d(storage):
    import torch

    sc = S.sphere_droplet_3d_small(24, lam=0.6)
    stream = torch.cuda.Stream()
    ref = lbm3d.Lattice3(sc.solid, sc.rhoA0, sc.rhoB0, sc.params(), storage)
    lat = lbm3d.Lattice3(sc.solid, sc.rhoA0, sc.rhoB0, sc.params(), storage, stream.cuda_stream)
    a, b = (torch.from_numpy(x.copy()).cuda() for x in (sc.rhoA0, sc.rhoB0))
    out = torch.zeros(5, a.numel(), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        lat.set_densities(a, b, on_device=True)
        lat.step(6)
        assert lbm.load_library().lbm3d_fields(lat.ctx, *[o.data_ptr() for o in out], 1) == lbm.LBM_OK
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    ref.step(6)
    assert np.array_equal(out.cpu().numpy(), np.stack([x.ravel() for x in ref.fields()]))
