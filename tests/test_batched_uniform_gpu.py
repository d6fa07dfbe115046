"""Batches laid out by the library (dense batch tensors) against the same
scenes given one by one: bit for bit, for both input types and wavelets, and
for more scenes than one table holds."""
import pytest
import torch

from paper_1803_00737_gb300 import D4, HAAR, _C

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("n,bands,H,W", [(1, 1, 4, 4), (3, 8, 34, 130), (130, 2, 6, 18)])
@pytest.mark.parametrize("wav", [HAAR, D4])
@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
def test_uniform_batch_equals_single_scenes(n, bands, H, W, wav, dtype):
    g = torch.Generator(device=DEV).manual_seed(n + bands)
    pan = torch.randint(0, 256, (n, H, W), generator=g, device=DEV).to(dtype)
    ms = torch.randint(0, 256, (n, bands, H // 2, W // 2), generator=g, device=DEV).to(dtype)
    f = torch.full((n, bands, H, W), float("nan"), device=DEV)
    u = torch.zeros((n, bands, H, W), dtype=torch.uint8, device=DEV)
    ws = torch.zeros(_C.dwtfuse_batched_workspace_size(), dtype=torch.uint8, device=DEV)
    _C.dwtfuse_fuse_batched_uniform(pan, ms, wav, f, u, ws)
    grad = torch.randn((n, bands, H, W), generator=g, device=DEV)
    gp = torch.full((n, H, W), float("nan"), device=DEV)
    gm = torch.full((n, bands, H // 2, W // 2), float("nan"), device=DEV)
    _C.dwtfuse_fuse_backward_batched_uniform(grad, wav, gp, gm, ws)
    for i in range(n):
        ef, eu = torch.empty_like(f[i]), torch.empty_like(u[i])
        _C.dwtfuse_fuse(pan[i], list(ms[i]), wav, ef, eu)
        ep, em = torch.empty_like(gp[i]), torch.empty_like(gm[i])
        _C.dwtfuse_fuse_backward(grad[i], wav, ep, list(em))
        assert torch.equal(f[i], ef) and torch.equal(u[i], eu), i
        assert torch.equal(gp[i], ep) and torch.equal(gm[i], em), i


def test_uniform_batch_refuses_what_the_table_call_refuses():
    ws = torch.zeros(_C.dwtfuse_batched_workspace_size(), dtype=torch.uint8, device=DEV)
    pan = torch.zeros((2, 8, 8), device=DEV)
    out = torch.zeros((2, 9, 8, 8), device=DEV)
    with pytest.raises(_C.DwtfuseError) as e:  # 9 bands in a batched call
        _C.dwtfuse_fuse_batched_uniform(pan, torch.zeros((2, 9, 4, 4), device=DEV), D4, out, None, ws)
    assert e.value.status == _C.ESHAPE
    with pytest.raises(ValueError):
        _C.dwtfuse_fuse_batched_uniform(pan, torch.zeros((2, 3, 4, 5), device=DEV), D4, out[:, :3], None, ws)
    with pytest.raises(_C.DwtfuseError) as e:
        _C.dwtfuse_fuse_batched_uniform(pan, torch.zeros((2, 9, 4, 4), device=DEV)[:, :8].contiguous(), D4, None,
                                        None, ws)
    assert e.value.status == _C.EINVAL
