"""FP32 EDM in register-blocked tiles (edge 64 and 128) at the edges of its
sizes, against the FP64 oracle within 1e-5 (diagonal exactly 0), and against
sub-matrices small enough for the 32 x 32 tiles, whose entries it has to give
bit for bit (the same operations in the same order)."""
import numpy as np
import pytest
import torch

import synth
from helpers import packed_index, rel_err, to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mp", ["lambda", "bbox", "linear", "rb"])
@pytest.mark.parametrize("n,d", [(512, 8), (513, 17), (577, 100), (3073, 1), (4608, 7), (4737, 19)])
def test_wide_rows(gpu, oracle, mp, n, d):
    x = synth.normal(n, d, seed=n + d)
    D = gpu.edm_packed(to_gpu(x), mp, "fp32")
    got = D.cpu().numpy()
    i = np.arange(n)
    assert (got[packed_index(i, i)] == 0).all()
    pr = synth.sample_pairs(100000, n, seed=3)
    pr = pr[pr[:, 0] != pr[:, 1]]
    assert rel_err(got[packed_index(pr[:, 0], pr[:, 1])], oracle.edm_pairs(x, pr)).max() <= 1e-5
    # the last 200 points alone take the 32 x 32 tiles
    sub = gpu.edm_packed(to_gpu(x[-200:]), mp, "fp32").cpu().numpy()
    a, b = np.tril_indices(200)
    assert np.array_equal(got[packed_index(a + n - 200, b + n - 200)], sub)


@pytest.mark.parametrize("mp,n,d", [("lambda", 2560, 4), ("bbox", 2561, 33), ("linear", 2687, 130), ("rb", 2689, 2)])
def test_wide_tiles(gpu, mp, n, d):
    """Tile layout: every float written (diagonal tiles whole, padding 0), the
    lower entries those of the packed rows."""
    x = to_gpu(synth.normal(n, d, seed=n))
    rows = gpu.edm_packed(x, mp, "fp32")
    out = torch.full((gpu.simplex_edm_tiles_len(n),), float("nan"), device="cuda")
    gpu.simplex_edm_tiles(x, out, mp, "fp32")
    nt = -(-n // 128)
    t = out.view(-1, 128, 128)
    full = torch.zeros((nt * 128, nt * 128), device="cuda")
    for I in range(nt):
        s = I * (I + 1) // 2
        full[128 * I:128 * I + 128, :128 * (I + 1)] = t[s:s + I + 1].permute(1, 0, 2).reshape(128, -1)
    assert not torch.isnan(out).any()
    low = torch.tril_indices(n, n, device="cuda")
    assert torch.equal(full[low[0], low[1]], rows)
    assert (full[n:] == 0).all() and (full[:, n:] == 0).all()
    for I in range(nt):   # diagonal tiles hold the whole square
        q = t[I * (I + 1) // 2 + I]
        assert torch.equal(q, q.T)


def test_wide_unaligned(gpu):
    """d a multiple of 4 but x only 4-byte aligned: the scalar loads."""
    n, d = 600, 12
    buf = torch.randn(n * d + 1, device="cuda")
    x = buf[1:].view(n, d)
    assert torch.equal(gpu.edm_packed(x, "lambda", "fp32"), gpu.edm_packed(x.clone(), "lambda", "fp32"))
