"""The batched forward's float instance for tables of light bodies (one band, or
Haar of at most 3), on both sides of its rule: every entry equals the
single-scene call bit for bit, on the three row layouts, with items of the
default height and of one row."""
import pytest
import torch

from paper_1803_00737_gb300 import D4, HAAR, _C, fuse

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("table", [[(HAAR, 1), (D4, 1)], [(HAAR, 3), (HAAR, 2), (D4, 1)], [(HAAR, 3), (D4, 2)],
                                   [(HAAR, 4), (D4, 1)], [(D4, 1)], [(HAAR, 3)]])
@pytest.mark.parametrize("rows", [0, 1])
def test_light_tables_equal_single_scenes(table, rows):
    g = torch.Generator(device=DEV).manual_seed(len(table) + rows)
    scenes, keep = [], []
    for W, offset in ((388, 0), (390, 0), (390, 2), (260, 0)):
        for wav, bands in table:
            buf = torch.zeros(46 * W + offset, device=DEV)
            p = buf[offset:].view(46, W)
            p.copy_(torch.randint(0, 256, (46, W), generator=g, device=DEV, dtype=torch.uint8))
            m = torch.randint(0, 256, (bands, 23, W // 2), generator=g, device=DEV, dtype=torch.uint8).float()
            f = torch.full((bands, 46, W), float("nan"), device=DEV)
            u = torch.zeros((bands, 46, W), dtype=torch.uint8, device=DEV)
            scenes.append(_C.make_scene(p, m, wav, f, u))
            keep.append((wav, p, m, f, u))
    ws = torch.zeros(_C.dwtfuse_batched_workspace_size(), dtype=torch.uint8, device=DEV)
    _C.dwtfuse_fuse_batched(scenes, ws, rows)
    torch.cuda.synchronize()
    assert _C.dwtfuse_get_last_device_status(ws) == _C.OK
    for wav, p, m, f, u in keep:
        ef, eu = fuse(p, m, wav, f32=True, u8=True)
        assert torch.equal(f, ef) and torch.equal(u, eu), (wav, tuple(p.shape), len(m))
