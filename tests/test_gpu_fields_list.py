"""The work list of the fields pass is sized by the blocks that pass holds on an SM, not by the step's:
where uniform items of up to 16 rows can all run at once, they do, with a block for every item.  Where
they cannot, the pass runs on as many blocks as fit."""
import pytest

from paper_2505_22256_gb300 import lbm, scenarios as S

pytestmark = pytest.mark.gpu

CASES = {"throat": lambda: [S.throat_channel(2048, 512, R=180, r=120)],
         "seven": lambda: [S.cylinder_droplet(331, R=50, r=60) for _ in range(7)],
         "uneven": lambda: [S.cylinder_droplet(n, R=n // 7, r=n // 5) for n in (700, 96, 500, 210)]}


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("name", list(CASES))
def test_fields_items_all_run_at_once(name, storage):
    import torch
    from capture_util import launches

    scs = CASES[name]()
    stream = torch.cuda.Stream()
    lat = lbm.Lattice(scs, storage, stream.cuda_stream)
    out = torch.zeros(4, sum(s.nx * s.ny for s in scs), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    (_, blocks, threads), = launches(stream, lambda: lbm.lbm_fields_all(lat.ctx, *out, on_device=True))
    cols = threads - 8
    heights = [sum(-(-s.nx // cols) * -(-s.ny // h) for s in scs) for h in range(1, 17)]
    fit = (3 if storage == "f32" else 4) * 128 // threads * torch.cuda.get_device_properties(0).multi_processor_count
    if min(heights) <= fit:
        assert blocks in heights, (blocks, heights)  # as many blocks as a list of some height has items
    else:
        assert blocks == fit
    lat.close()
