"""The adjoint of an empty batch: nothing to do, on the host (no library call
that would refuse zero scenes)."""
import torch

from paper_1803_00737_gb300 import D4, autograd, tune


def test_adjoint_of_an_empty_batch_returns(monkeypatch, tmp_path):
    monkeypatch.setenv("DWTFUSE_AUTOTUNE", "0")
    monkeypatch.setenv("DWTFUSE_TUNE_CACHE", str(tmp_path / "none.json"))
    monkeypatch.setattr(tune, "current_device_key", lambda: "dev")
    g = torch.zeros((0, 3, 8, 12))
    gp, gm = torch.zeros((0, 8, 12)), torch.zeros((0, 3, 4, 6))
    autograd.fuse_batch_backward(g, D4, gp, gm)
    assert gp.shape == (0, 8, 12) and gm.shape == (0, 3, 4, 6)
