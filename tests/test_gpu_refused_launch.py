"""A step whose launch the runtime refuses (its stream's capture has been invalidated: an error on the host,
nothing runs) reports that once and leaves the context as it was: the calls after it succeed and the state is the one
before."""
import ctypes

import numpy as np
import pytest

from paper_2505_22256_gb300 import lbm, lbm3d, scenarios as S

pytestmark = pytest.mark.gpu


def refused(stream, call):
    """call() inside a capture of `stream` that a synchronisation has invalidated; the capture is ended."""
    import torch

    try:
        rt = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    except OSError:
        pytest.skip("no shared CUDA runtime")
    handle, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(handle, 1) == 0
    assert rt.cudaStreamSynchronize(handle) != 0
    try:
        with pytest.raises(lbm.LbmError):
            call()
    finally:
        rt.cudaStreamEndCapture(handle, ctypes.byref(graph))
        rt.cudaGetLastError()


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_refused_step_2d(storage):
    import torch

    sc, stream = S.cylinder_droplet(96, lam=0.6), torch.cuda.Stream()
    lat, ref = lbm.Lattice(sc, storage, stream.cuda_stream), lbm.Lattice(sc, storage)
    a, b = torch.from_numpy(sc.rhoA0.copy()).cuda(), torch.from_numpy(sc.rhoB0.copy()).cuda()
    torch.cuda.synchronize()
    lat.step(3)
    ref.step(3)
    torch.cuda.synchronize()
    before = lat.populations()
    refused(stream, lambda: lat.step(1))
    assert np.array_equal(lat.populations(), before)
    refused(stream, lambda: lat.step(1))
    lbm.lbm_set_densities_all(lat.ctx, a, b, on_device=True)  # the first launch after the refusal
    lat.step(4)
    lbm.lbm_set_densities_all(ref.ctx, a, b, on_device=True)
    ref.step(4)
    assert np.array_equal(lat.populations(), ref.populations())


@pytest.mark.parametrize("storage", ["f32", "f64"])
def test_refused_step_3d(storage):
    import torch

    sc, stream = S.sphere_droplet_3d_small(24, lam=0.6), torch.cuda.Stream()
    lat = lbm3d.Lattice3(sc.solid, sc.rhoA0, sc.rhoB0, sc.params(), storage, stream.cuda_stream)
    ref = lbm3d.Lattice3(sc.solid, sc.rhoA0, sc.rhoB0, sc.params(), storage)
    a, b = torch.from_numpy(sc.rhoA0.copy()).cuda(), torch.from_numpy(sc.rhoB0.copy()).cuda()
    torch.cuda.synchronize()
    lat.step(3)
    torch.cuda.synchronize()
    before = lat.populations()
    refused(stream, lambda: lat.step(1))
    assert np.array_equal(lat.populations(), before)
    refused(stream, lambda: lat.step(1))
    lat.set_densities(a, b, on_device=True)
    lat.step(2)
    ref.step(2)
    assert np.array_equal(lat.populations(), ref.populations())
