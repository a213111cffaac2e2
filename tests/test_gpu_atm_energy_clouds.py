"""ATM energy alone on the tensor cores (from 1280 points) where close pairs,
equal distances and tight clusters meet its half tables, masks and passes; the
same clouds through the forces call.  Energies within 1e-6 of the sum of the
terms' sizes in 64 bits, forces within 32 u kappa per atom."""
import numpy as np
import pytest
import torch

import synth
from helpers import to_gpu
from test_gpu_atm import E_TOL, KAPPA_C, U32, near_coincident

pytestmark = pytest.mark.gpu


def cloud(kind, n):
    if kind == "near":
        return near_coincident(n, 12.0, 50, 1e-3), 1e-4
    if kind == "lattice":   # every nearest neighbour is a tie
        g = np.stack(np.meshgrid(np.arange(12.0), 1.25 * np.arange(12.0), 1.5 * np.arange(12.0), indexing="ij"), -1)
        return g.reshape(-1, 3).astype(np.float32)[:n], 1e-4
    size = 5 if kind == "clusters5" else 8   # tight clusters: large triples without a nearest-neighbour pair
    c = synth.uniform_cube(-(-n // size), 3, 20.0, seed=1).astype(np.float64)
    x = np.repeat(c, size, axis=0)[:n] + 0.02 * synth.normal(n, 3, 2)
    return x.astype(np.float32), 1e-6


@pytest.mark.parametrize("mp,kind,n", [("lambda", "near", 1300), ("bbox", "lattice", 1400), ("linear", "clusters5", 1345),
                                       ("lambda", "clusters8", 1600)])
def test_energy_clouds(gpu, oracle, mp, kind, n):
    x, eps = cloud(kind, n)
    E, size = oracle.atm_energy(x, 1.0, eps), oracle.atm_abs_energy(x, 1.0, eps)
    F, e = gpu.atm_forces(to_gpu(x), 1.0, eps, mp)
    raw = gpu.atm_energy_raw(to_gpu(x), 1.0, eps, mp).item()
    print(kind, n, f"energy {abs(raw - E) / size:.1e}, with forces {abs(e.item() - E) / size:.1e} of the terms' sizes")
    assert abs(raw - E) <= E_TOL * size and abs(e.item() - E) <= E_TOL * size
    G, kappa = oracle.atm_grad(x, 1.0, eps), oracle.atm_grad_abs(x, 1.0, eps)
    assert (np.linalg.norm(F.cpu().numpy() + G, axis=1) <= KAPPA_C * U32 * kappa).all()


def test_energy_strips(gpu):
    """More than 24 super-blocks a side (the list in strips): against the
    sum over pair matrices in 64 bits."""
    n = 6400
    x = to_gpu(synth.uniform_cube(n, 3, 20.0, seed=3))
    xd = x.double()
    p = [xd[:, None, c] - xd[None, :, c] for c in range(3)]
    s = p[0] ** 2 + p[1] ** 2 + p[2] ** 2 + float(np.float32(1e-4))
    off = 1 - torch.eye(n, dtype=torch.float64, device="cuda")
    R, q = off * s ** -1.5, off * s ** -2.5
    E = (R @ R * R).sum() / 6
    for a in range(3):
        for b in range(3):
            t = sum((q * p[a] * p[c]) @ (q * p[c] * p[b]) for c in range(3))
            E -= 0.5 * (t * q * p[a] * p[b]).sum()
    assert gpu.atm_energy_raw(x).item() == pytest.approx(E.item(), rel=E_TOL)
    assert gpu.atm_forces(x)[1].item() == pytest.approx(E.item(), rel=E_TOL)
