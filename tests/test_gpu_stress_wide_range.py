"""prec = fp32 of the stress on the tensor cores (FP16 hi + lo operands) for
clouds whose coordinates or points differ in size by orders of magnitude:
wide axes that x and y share, groups far apart, single large points.  Against
64 bits and against the FP32 kernels, which a call with a smaller workspace
runs.  The operands keep 22 bits, so an error may exceed twice the FP32
kernels' by 2^-22 of the value (2^-21 where two operands' errors add up:
loss, single columns).  Rows pass 1e-4 only where their terms cancel (at most
one in a thousand); the worst row is measured by its terms, and within what 22
bits in place of 24 can make of the FP32 kernels' (four times)."""
import numpy as np
import pytest
import torch

from test_gpu_stress import G_TOL

pytestmark = pytest.mark.gpu


def exact(x, y):
    """Loss and gradient in 64 bits, the residuals formed pair by pair from
    centred points."""
    x, y = x.double(), y.double()
    x, y = x - x.mean(0), y - y.mean(0)
    S, D = x + y, x - y
    a = (S * D).sum(1)
    loss, g = torch.zeros((), dtype=torch.float64, device=x.device), torch.empty_like(x)
    for b in range(0, len(x), 1024):
        q = slice(b, b + 1024)
        r = a[q, None] + a[None] - S[q] @ D.T - D[q] @ S.T
        i = torch.arange(r.shape[0], device=x.device)
        r[i, b + i] = 0.0
        loss += 0.5 * (r * r).sum()
        g[q] = 4 * (x[q] * r.sum(1)[:, None] - r @ x)
    return loss.item(), g


def row_terms(x, y):
    """Per row 4 sqrt(sum_j (rho_ij |x_i - x_j|)^2), rho_ij = sum_t (|S_i| +
    |S_j|)(|Delta_i| + |Delta_j|), the size of what is rounded in r_ij."""
    x, y = x.double(), y.double()
    S, D = (x - x.mean(0) + y - y.mean(0)).abs(), (x - y).abs()
    out = torch.empty(len(x), dtype=torch.float64, device=x.device)
    a = (S * D).sum(1)
    for b in range(0, len(x), 512):
        q = slice(b, b + 512)
        rho = a[q, None] + a[None] + S[q] @ D.T + D[q] @ S.T
        out[q] = 4 * (rho * torch.cdist(x[q], x)).square().sum(1).sqrt()
    return out


def cloud(kind, n, d, k):
    g = np.random.default_rng(n + d + int(k))
    x, e = g.standard_normal((n, d)), 0.1 * g.standard_normal((n, d))
    if kind == "axis":          # one wide column, equal in x and y
        x[:, 0] *= k
        e[:, 0] = 0
    elif kind == "plane":       # all columns wide and equal but the last
        x[:, :-1] *= k
        e[:, :-1] = 0
    elif kind == "groups":      # two groups k apart along a shared axis
        x[n // 2:, 0] += k
        e[:, 0] = 0
    elif kind == "points":      # one far point equal in both, one with a large displacement
        x[n // 3] *= k
        e[n // 3] = 0
        e[n // 5] *= 10 * k
    elif kind == "columns":     # columns over six orders of magnitude
        s = np.logspace(-3, 3, d)
        x *= s
        e *= s * np.abs(x / s)
    x = x.astype(np.float32)
    return torch.from_numpy(x).cuda(), torch.from_numpy((x + e).astype(np.float32)).cuda()


@pytest.mark.parametrize("kind,n,d,k", [
    ("axis", 4096, 3, 1e2), ("axis", 4096, 3, 1e4), ("axis", 2600, 16, 1e3), ("axis", 4097, 64, 1e3),
    ("plane", 4096, 3, 1e2), ("plane", 4096, 3, 1e3), ("plane", 4096, 3, 1e4), ("plane", 3000, 96, 1e3),
    ("groups", 4096, 3, 1e3), ("groups", 3000, 16, 1e3), ("points", 4096, 3, 1e3), ("points", 3000, 33, 1e3),
    ("columns", 4096, 16, 1), ("plain", 4096, 3, 1), ("plain", 3000, 64, 1)])
def test_wide_range(gpu, kind, n, d, k):
    x, y = cloud(kind, n, d, k)
    L, G = exact(x, y)
    terms = row_terms(x, y)

    def errors(loss, g):
        e = g.double() - G
        rows = e.norm(dim=1) / G.norm(dim=1)
        return {"loss": abs(loss.item() / L - 1), "norm": (e.norm() / G.norm()).item(), "median": rows.median().item(),
                "columns": (e.norm(dim=0) / G.norm(dim=0)).max().item(), "rows": (rows > G_TOL).double().mean().item(), "worst": (e.norm(dim=1) / terms).max().item()}

    ws = torch.empty(8 * (gpu.simplex_grid_blocks(2, -(-n // 64), "lambda") + 1024), dtype=torch.uint8, device="cuda")
    assert ws.numel() < gpu.simplex_workspace_bytes("stress_fwd_bwd", n, d)
    loss, g = torch.empty((), dtype=torch.float64, device="cuda"), torch.empty_like(x)
    gpu.simplex_stress_fwd_bwd(x, y, 1.0, g, loss, workspace=ws)
    ref = errors(loss, g)
    loss, g = gpu.stress_fwd_bwd(x, y)
    got = errors(loss, g)
    got["loss alone"] = abs(gpu.stress_fwd(x, y)[0].item() / L - 1)
    gpu.simplex_device_errors()
    print(kind, n, d, k, {a: f"{v:.1e}" for a, v in got.items()}, "FP32 kernels", {a: f"{v:.1e}" for a, v in ref.items()})
    assert max(got["loss"], got["loss alone"]) <= 2 * ref["loss"] + 2.0 ** -21
    assert got["norm"] <= 2 * ref["norm"] + 2.0 ** -22
    assert got["median"] <= 2 * ref["median"] + 2.0 ** -22
    assert got["columns"] <= 2 * ref["columns"] + 2.0 ** -21
    assert got["rows"] <= 1e-3
    assert got["worst"] <= 4 * ref["worst"]


@pytest.mark.parametrize("scale", [2.0 ** -36, 2.0 ** 26])
def test_extreme_sizes(gpu, scale):
    """Clouds near the ends of what the gradient's FP32 values span: the
    gradient of the cloud of unit size, scaled (within 1e-6 of its largest
    entry: what rounds in FP16 hi + lo and FP32 is the same at any size)."""
    x, y = cloud("plain", 3000, 8, 1)
    G = 0.3 * exact(x, y)[1]
    g = gpu.stress_bwd(x * scale, y * scale, 0.3).double() / scale / scale / scale
    assert (g - G).abs().max().item() <= 1e-6 * G.abs().max().item()


@pytest.mark.parametrize("side", ["x", "y"])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_not_finite_rows(gpu, side, bad):
    """A coordinate that is not finite belongs to a residual of every row."""
    x, y = cloud("plain", 3000, 16, 1)
    (x if side == "x" else y)[5, 3] = bad
    loss, g = gpu.stress_fwd_bwd(x, y)
    assert not torch.isfinite(loss) and not torch.isfinite(gpu.stress_fwd(x, y)[0])
    assert not torch.isfinite(g).any()
