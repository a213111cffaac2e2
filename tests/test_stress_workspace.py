"""Workspaces of the FP32 stress: bounded at any size, and calls that go on
where the device has no room for them."""
import pytest
import torch

import synth
from helpers import stress_moments, to_gpu
from test_gpu_stress import G_TOL, L_TOL, row_err


@pytest.mark.parametrize("n", [1 << 22, 1 << 25, 1 << 28])
@pytest.mark.parametrize("d", [1, 3, 96])
def test_workspace_bounded(n, d):
    """FP32 gradients took no workspace before the tensor cores: at sizes whose
    scan alone would take hundreds of GB they have to do without."""
    import paper_1610_07394_gb300 as sx
    assert sx.simplex_workspace_bytes("stress_bwd", n, d) <= 16 << 30


@pytest.mark.gpu
def test_no_room(gpu, monkeypatch):
    n, d = 3000, 16
    x = synth.normal(n, d, 1)
    y = synth.perturbed(x, 0.1, 2)
    L, G = stress_moments(x, y)
    small = 8 * (gpu.simplex_grid_blocks(2, -(-n // 64), "lambda") + 1024)

    def full(op, n, d, map="lambda", prec="fp32", device="cuda"):
        if gpu.simplex_workspace_bytes(op, n, d, map, prec) > small:
            raise torch.OutOfMemoryError("no room")
        return torch.empty(small, dtype=torch.uint8, device=device)

    monkeypatch.setattr(gpu, "workspace", full)
    xt, yt = to_gpu(x), to_gpu(y)
    loss, g = gpu.stress_fwd_bwd(xt, yt)
    for v in (loss, gpu.stress_fwd(xt, yt)[0]):
        assert abs(v.item() - L) <= L_TOL * L
    for v in (g, gpu.stress_bwd(xt, yt)):
        assert row_err(v.double().cpu().numpy(), G).max() <= G_TOL
    with pytest.raises(torch.OutOfMemoryError):
        gpu.stress_bwd(to_gpu(synth.normal(n, 64, 1)), to_gpu(synth.normal(n, 64, 2)), 1.0, "lambda", "bf16x3")
