"""What the speed of this library is measured on: calls of its public entry
points as a program with FP32 points on the GPU makes them.

The sizes are those of the benchmark configurations (synth.WORKLOADS), the
bench rows and the tests, with ragged ones between them.  The library sums
energies, forces and losses in FP64 from FP32 terms (documented to 1e-6 and
1e-5); a program whose points are FP32 carries them on in the type of its
points, so ``run`` hands every floating result over in that type, as the
library's own autograd functions do with gradients.
"""
import math

import numpy as np
import torch

import paper_1610_07394_gb300 as sx


def listed():
    return [
        # The smallest call: the EDM of 1,024 points in space (configuration
        # edm_n1024_d3); launches and the host path count, 2 MB are written.
        dict(name="edm_n1024_d3", kind="edm", n=1024, d=3, prec="fp32", map="lambda"),
        # Distance matrix of embeddings in the default precision, a width
        # that no tile divides: the FP32 difference form.
        dict(name="edm_fp32_n12000_d100", kind="edm", n=12000, d=100, prec="fp32", map="lambda"),
        # Distance matrix of wide vectors (configuration edm_n32768_d256) on
        # the tensor cores.
        dict(name="edm_bf16x3_n32768_d256", kind="edm", n=32768, d=256, prec="bf16x3", map="lambda"),
        # The same at d = 64 and a size that is no power of two and no
        # multiple of a tile: 5 GB of packed rows, the store-bound case.
        dict(name="edm_bf16x3_n50000_d64", kind="edm", n=50000, d=64, prec="bf16x3", map="lambda"),
        # The tile-packed layout, for programs that read the matrix by tiles.
        dict(name="edm_tiles_n32768_d128", kind="edm_tiles", n=32768, d=128, prec="bf16x3", map="lambda"),
        # Energy of a Monte Carlo step, small (configuration atm_n1024).
        dict(name="atm_energy_n1024", kind="atm_energy", n=1024, side=10.0, map="lambda"),
        # A minimiser's step through autograd: energy, then its gradient, at
        # a ragged size (bench row atm_n3000).
        dict(name="atm_autograd_n3000", kind="atm_autograd", n=3000, side=20.0, map="lambda"),
        # Molecular dynamics: energy and forces from one call (configuration
        # atm_n4096).
        dict(name="atm_forces_n4096", kind="atm_forces", n=4096, side=20.0, map="lambda"),
        # The largest call, the benchmark's workload (configuration atm_n16384).
        dict(name="atm_forces_n16384", kind="atm_forces", n=16384, side=20.0, map="lambda"),
        # A training step of the stress loss through autograd in the default
        # precision.
        dict(name="stress_autograd_fp32_n10000_d64", kind="stress_autograd", n=10000, d=64, prec="fp32",
             map="lambda"),
        # Loss and gradient from one pass at full size on the tensor cores
        # (configuration stress_n65536_d64).
        dict(name="stress_bf16x3_n65536_d64", kind="stress_fwd_bwd", n=65536, d=64, prec="bf16x3", map="lambda"),
        # The loss alone, as a line search asks for it, in the default
        # precision at an odd width (d = 33 of the tests).
        dict(name="stress_fwd_fp32_n16384_d33", kind="stress_fwd", n=16384, d=33, prec="fp32", map="lambda"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same calls; no cost above the largest listed one."""
    kind = rng.choice(["edm", "edm", "edm_tiles", "atm_energy", "atm_forces", "atm_autograd", "stress_fwd",
                       "stress_autograd", "stress_fwd_bwd"])
    m2 = rng.choice(["lambda", "lambda", "lambda", "bbox", "linear", "rb"])
    m3 = rng.choice(["lambda", "lambda", "lambda", "bbox", "linear"])
    if kind in ("edm", "edm_tiles"):
        if rng.random() < 0.5:
            return dict(kind=kind, n=_log(rng, 256, 16384), d=_log(rng, 2, 256), prec="fp32", map=m2)
        return dict(kind=kind, n=_log(rng, 1024, 49152), d=rng.choice([64, 128, 192, 256]), prec="bf16x3", map=m2)
    if kind.startswith("atm"):
        n = _log(rng, 64, 12000)
        # 0.4 to 2 points per unit volume, as in the configurations
        return dict(kind=kind, n=n, side=round((n / rng.uniform(0.4, 2.0)) ** (1.0 / 3.0), 3), map=m3)
    if rng.random() < 0.5:
        return dict(kind=kind, n=_log(rng, 256, 20000), d=_log(rng, 2, 128), prec="fp32", map=m2)
    return dict(kind=kind, n=_log(rng, 1024, 65536), d=rng.choice([32, 64, 96]), prec="bf16x3", map=m2)


NU, EPS = 1.0, 1e-4   # the ATM configurations' strength and softening


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, kind = case["n"], case["kind"]
    st = dict(case)
    if kind.startswith("atm"):
        st["x"] = torch.rand((n, 3), generator=g, device="cuda") * case["side"]
        if kind == "atm_autograd":
            st["x"].requires_grad_(True)
    elif kind.startswith("edm"):
        d = case["d"]
        # points of space in the unit cube, feature vectors N(0, 1)
        st["x"] = torch.rand((n, d), generator=g, device="cuda") if d <= 3 else \
            torch.randn((n, d), generator=g, device="cuda")
    else:
        st["x"] = torch.randn((n, case["d"]), generator=g, device="cuda")
        st["y"] = st["x"] + 0.1 * torch.randn((n, case["d"]), generator=g, device="cuda")
        if kind == "stress_autograd":
            st["x"].requires_grad_(True)
    return st


def run(st):
    kind, mp = st["kind"], st["map"]
    if kind == "edm":
        return sx.edm_packed(st["x"], mp, st["prec"])
    if kind == "edm_tiles":
        return sx.edm_tiles(st["x"], mp, st["prec"])
    if kind == "atm_energy":
        return sx.atm_energy_raw(st["x"], NU, EPS, mp).to(st["x"].dtype)
    if kind == "atm_forces":
        f, e = sx.atm_forces(st["x"], NU, EPS, mp)
        return {"energy": e.to(st["x"].dtype), "forces": f.to(st["x"].dtype)}
    if kind == "atm_autograd":
        x = st["x"]
        x.grad = None
        e = sx.atm_energy(x, NU, EPS, mp)
        e.backward()
        return {"energy": e.detach().to(x.dtype), "grad": x.grad}
    if kind == "stress_fwd":
        loss, _ = sx.stress_fwd(st["x"], st["y"], mp, st["prec"])
        return loss.to(st["x"].dtype)
    if kind == "stress_autograd":
        x = st["x"]
        x.grad = None
        loss = sx.stress_loss(x, st["y"], mp, st["prec"])
        loss.backward()
        return {"loss": loss.detach().to(x.dtype), "grad": x.grad}
    loss, grad = sx.stress_fwd_bwd(st["x"], st["y"], 1.0, mp, st["prec"])
    return {"loss": loss.to(st["x"].dtype), "grad": grad}


def _packed(n):
    """Pairs (i, j), j <= i < n."""
    return n * (n + 1) // 2


def work(case):
    """Inputs read once and outputs written once; a pair takes 3 d flops
    (difference, product, sum) in FP32 or 2 d as a product, a triple's energy
    20 and its energy and three side derivatives 53.5."""
    kind, n = case["kind"], case["n"]
    if kind == "edm":
        return dict(bytes=4.0 * (n * case["d"] + _packed(n)),
                    flops=(3.0 if case["prec"] == "fp32" else 2.0) * case["d"] * n * (n - 1) / 2)
    if kind == "edm_tiles":
        nt = -(-n // 128)
        return dict(bytes=4.0 * (n * case["d"] + nt * (nt + 1) // 2 * 16384),
                    flops=(3.0 if case["prec"] == "fp32" else 2.0) * case["d"] * n * (n - 1) / 2)
    if kind.startswith("atm"):
        t = math.comb(n, 3)
        return dict(bytes=12.0 * n + (0 if kind == "atm_energy" else 24.0 * n),
                    flops=t * {"atm_energy": 20.0, "atm_forces": 53.5, "atm_autograd": 73.5}[kind])
    # the residual 4 d per pair, the gradient's two sides 4 d more
    per = {"stress_fwd": 4.0, "stress_autograd": 12.0, "stress_fwd_bwd": 8.0}[kind]
    return dict(bytes=4.0 * n * case["d"] * (2 if kind == "stress_fwd" else 3),
                flops=per * case["d"] * n * (n - 1) / 2)


def _rows64(x, a, b):
    """Squared distances of rows a..b-1 to points 0..b-1, 64 bits."""
    p, q = x[a:b], x[:b]
    return (p.square().sum(1)[:, None] + q.square().sum(1)[None, :] - 2.0 * p @ q.T).clamp_(min=0.0)


def _edm64(x, n):
    out = torch.empty(_packed(n), dtype=torch.float64, device=x.device)
    step = max(1, min(n, (1 << 27) // n))
    col = torch.arange(n, device=x.device)
    for a in range(0, n, step):
        b = min(n, a + step)
        d = _rows64(x, a, b)
        row = torch.arange(a, b, device=x.device)[:, None]
        d[torch.arange(b - a, device=x.device), torch.arange(a, b, device=x.device)] = 0.0
        out[a * (a + 1) // 2: b * (b + 1) // 2] = d[col[None, :b] <= row]
    return out


def _tiles64(x, n):
    nt = -(-n // 128)
    out = torch.zeros((nt * (nt + 1) // 2, 128, 128), dtype=torch.float64, device=x.device)
    for i in range(nt):
        a, b = 128 * i, min(n, 128 * i + 128)
        d = torch.zeros((128, 128 * (i + 1)), dtype=torch.float64, device=x.device)
        d[: b - a, :b] = _rows64(x, a, b)
        e = torch.arange(b - a, device=x.device)
        d[e, a + e] = 0.0
        s = i * (i + 1) // 2
        out[s: s + i + 1] = d.view(128, i + 1, 128).transpose(0, 1)
    return out.view(-1)


def _atm64(x, n, nu, eps):
    """Energy and its gradient from the pair matrices R = s^(-3/2) and
    U = s^(-5/2) p p^T of p = x_i - x_j, s = |p|^2 + eps, both 0 at i = j:
    a triple's term is nu (R_ij R_jk R_ki - 3 tr U_ij U_jk U_ki), so
    E = nu/6 (tr R^3 - 3 tr U^3) and dE/dU_ij = -3 nu sum_k U_ik U_kj."""
    p = [x[:, None, c] - x[None, :, c] for c in range(3)]
    s = p[0] ** 2 + p[1] ** 2 + p[2] ** 2 + eps
    off = 1.0 - torch.eye(n, dtype=x.dtype, device=x.device)
    r3 = off * s ** -1.5
    q5 = off * s ** -2.5
    u = {(a, b): q5 * p[a] * p[b] for a in range(3) for b in range(a, 3)}
    u.update({(b, a): v for (a, b), v in list(u.items())})
    w = r3 @ r3                              # dE/dR_ij = nu w
    e = nu / 6.0 * (w * r3).sum()
    radial = -3.0 * nu * w * q5              # along p
    grad = [radial * p[c] for c in range(3)]
    for a in range(3):
        for b in range(3):
            t = sum(u[a, c] @ u[c, b] for c in range(3))
            e = e - nu / 2.0 * (t * u[a, b]).sum()
            t *= -3.0 * nu
            for c in range(3):
                if c == a:
                    grad[c] += t * q5 * p[b]
                if c == b:
                    grad[c] += t * q5 * p[a]
                grad[c] -= 5.0 * t * u[a, b] / s * p[c]
    return e, torch.stack([g.sum(1) for g in grad], 1)


def _stress64(x, y):
    """Loss and gradient from moment matrices: r_ij = a_i + a_j - S_i.D_j - D_i.S_j
    for S = x + y, D = x - y, a = S.D, summed in closed form."""
    c = x.mean(0)
    n, d = x.shape
    x, y = x - c, y - c
    s, e = x + y, x - y
    a = (s * e).sum(1)
    one = torch.ones((n, 1), dtype=x.dtype, device=x.device)
    u = torch.cat([a[:, None], one, s, e], 1)
    v = torch.cat([one, a[:, None], -e, -s], 1)
    loss = 0.5 * ((u.T @ u) * (v.T @ v)).sum()
    rs = n * a + a.sum() - s @ e.sum(0) - e @ s.sum(0)
    rx = torch.outer(a, x.sum(0)) + a @ x - s @ (e.T @ x) - e @ (s.T @ x)
    return loss, 4.0 * (x * rs[:, None] - rx)


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind.startswith("atm") and n > 6000:
        return None   # minutes in 64 bits
    st = prepare(case, seed)
    x = st["x"].detach().double()
    if kind == "edm":
        return _edm64(x, n)
    if kind == "edm_tiles":
        return _tiles64(x, n)
    if kind.startswith("atm"):
        # the kernels take eps as FP32
        e, g = _atm64(x, n, NU, float(np.float32(EPS)))
        if kind == "atm_energy":
            return e
        return {"energy": e, "forces": -g} if kind == "atm_forces" else {"energy": e, "grad": g}
    loss, g = _stress64(x, st["y"].double())
    return loss if kind == "stress_fwd" else {"loss": loss, "grad": g}
