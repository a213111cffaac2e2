"""prec = fp32 of the stress loss and gradient where the pair products run on
the tensor cores (FP16 hi + lo splits): edges of its sizes, widths that are
padded, alignments, workspaces and clouds away from the origin, against the
FP64 moment identity (pinned against the oracle's pairwise loops) with the
FP32 tolerances: loss 1e-5, gradient 1e-4 per row."""
import numpy as np
import pytest
import torch

import synth
from helpers import stress_moments, to_gpu
from test_gpu_stress import G_TOL, L_TOL, row_err

pytestmark = pytest.mark.gpu


def check(gpu, x, y, mp, xt=None):
    xt = to_gpu(x) if xt is None else xt
    yt = to_gpu(y)
    L, G = stress_moments(x, y)
    loss, _ = gpu.stress_fwd(xt, yt, mp)
    lb, gb = gpu.stress_fwd_bwd(xt, yt, 2.5, mp)
    g = gpu.stress_bwd(xt, yt, 1.0, mp)
    gpu.simplex_device_errors()
    e = row_err(g.double().cpu().numpy(), G)
    print(f"{mp} n={len(x)} d={x.shape[1]}: loss {abs(loss.item() / L - 1):.1e}, gradient row max {e.max():.1e}")
    assert abs(loss.item() - L) <= L_TOL * L and abs(lb.item() - L) <= L_TOL * L
    assert e.max() <= G_TOL
    assert row_err(gb.double().cpu().numpy(), 2.5 * G).max() <= G_TOL


@pytest.mark.parametrize("mp,n,d", [("lambda", 1345, 64), ("lambda", 2049, 96), ("bbox", 3072, 95), ("linear", 4097, 1), ("rb", 4224, 3),
                                    ("lambda", 3000, 31), ("lambda", 2816, 64), ("linear", 3001, 33),
                                    ("lambda", 2600, 97)])
def test_f16_edges(gpu, mp, n, d):
    """One point past a tile, odd numbers of row blocks, widths at and beside
    the padding to 32, d = 97 (kept in FP32)."""
    x = synth.normal(n, d, seed=n + d)
    check(gpu, x, synth.perturbed(x, 0.1, seed=n + d + 1), mp)


@pytest.mark.parametrize("scale,shift", [(1e-3, 0.0), (1e4, 0.0), (0.05, 3.0)])
def test_f16_scales(gpu, scale, shift):
    """Clouds of other sizes, and one away from the origin."""
    x = (scale * synth.normal(3000, 20, 5).astype(np.float64) + shift).astype(np.float32)
    check(gpu, x, synth.perturbed(x, 0.1 * scale, 6), "lambda")


def test_f16_outlier(gpu):
    """One point a thousand widths away: it carries the loss and every row."""
    x = synth.normal(3000, 16, 7)
    x[1234] *= 1000
    check(gpu, x, synth.perturbed(x, 0.1, 8), "lambda")


def test_f16_alignment_and_zero(gpu):
    """Points 4-byte aligned only (a view one float in), and y = x: loss and
    gradient exactly 0."""
    n, d = 3000, 33
    x = synth.normal(n, d, 9)
    buf = torch.empty(n * d + 1, device="cuda")
    xt = buf[1:].view(n, d)
    xt.copy_(to_gpu(x))
    check(gpu, x, synth.perturbed(x, 0.1, 10), "lambda", xt)
    loss, g = gpu.stress_fwd_bwd(xt, xt)
    assert loss.item() == 0.0 and bool((g == 0).all())


def test_f16_smaller_workspace(gpu):
    """The workspaces that FP32 needed without the tensor cores are enough."""
    n, d = 3000, 16
    x, y = synth.normal(n, d, 11), synth.perturbed(synth.normal(n, d, 11), 0.1, 12)
    xt, yt = to_gpu(x), to_gpu(y)
    L, G = stress_moments(x, y)
    small = 8 * (gpu.simplex_grid_blocks(2, -(-n // 64), "lambda") + 1024)
    assert small < gpu.simplex_workspace_bytes("stress_fwd_bwd", n, d)
    ws = torch.empty(small, dtype=torch.uint8, device="cuda")
    loss, g = torch.empty((), dtype=torch.float64, device="cuda"), torch.empty_like(xt)
    gpu.simplex_stress_fwd(xt, yt, None, loss, workspace=ws)
    assert abs(loss.item() - L) <= L_TOL * L
    gpu.simplex_stress_fwd_bwd(xt, yt, 1.0, g, loss, workspace=ws)
    assert abs(loss.item() - L) <= L_TOL * L and row_err(g.double().cpu().numpy(), G).max() <= G_TOL
    gpu.simplex_stress_bwd(xt, yt, 1.0, g)
    assert row_err(g.double().cpu().numpy(), G).max() <= G_TOL


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_f16_not_finite(gpu, bad):
    x = synth.normal(3000, 16, 13)
    y = synth.perturbed(x, 0.1, 14)
    x[5, 3] = bad
    loss, g = gpu.stress_fwd_bwd(to_gpu(x), to_gpu(y))
    assert not torch.isfinite(loss) and not torch.isfinite(g).any(dim=1).all()


def test_tensor_maps_on_a_new_thread(gpu):
    """The first library call of a thread that has bound no CUDA context yet
    (autograd workers): every buffer is there already."""
    import threading
    n, d = 3000, 64
    x = to_gpu(synth.normal(n, d, 15))
    y = to_gpu(synth.perturbed(synth.normal(n, d, 15), 0.1, 16))
    for prec in ("fp32", "bf16x3"):
        want = gpu.stress_bwd(x, y, 1.0, "lambda", prec)
        g = torch.empty_like(x)
        ws = gpu.workspace("stress_bwd", n, d, "lambda", prec)
        stream = torch.cuda.current_stream().cuda_stream
        torch.cuda.synchronize()
        failed = []

        def call():
            try:
                gpu.simplex_stress_bwd(x, y, 1.0, g, "lambda", prec, ws, stream)
            except Exception as e:
                failed.append(e)

        t = threading.Thread(target=call)
        t.start()
        t.join()
        assert not failed, failed
        assert (g - want).abs().max().item() <= 1e-5 * want.abs().max().item()
