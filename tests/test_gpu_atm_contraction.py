"""ATM energy and forces where they run as contractions on the tensor cores
(forces from 640 points, energy from 1280), at the edges of its tiles (128 rows,
256-row super-blocks, 64-point chunks) against the FP64 oracle, with the
tolerances of the FP32 path: energy 1e-6, forces 1e-4 per atom and, for clouds
of close pairs, 32 u kappa per atom."""
import numpy as np
import pytest
import torch

import synth
from helpers import grad_all_threads, to_gpu
from test_gpu_atm import E_TOL, F_TOL, KAPPA_C, U32, atom_err, near_coincident

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mp,n,eps", [("lambda", 640, 1e-4), ("bbox", 641, 1e-4), ("linear", 767, 0.0),
                                      ("lambda", 769, 1e-4), ("bbox", 1025, 1e-2), ("lambda", 1280, 1e-4), ("bbox", 1281, 1e-4),
                                      ("lambda", 1664, 1e-4),
                                      ("linear", 1793, 1e-4)])
def test_contraction_edges(gpu, oracle, mp, n, eps):
    """Smallest sizes of both calls, one row past a tile, a super-block and a
    chunk, a last super-block with one row block."""
    x = synth.uniform_cube(n, 3, n ** (1 / 3), seed=n)
    F, E = gpu.atm_forces(to_gpu(x), 1.5, eps, mp)
    e_ref, G = grad_all_threads(oracle, x, 1.5, eps)
    err = atom_err(F.cpu().numpy(), G)
    print(f"contraction {mp} n={n}: force max {err.max():.2e} median {np.median(err):.2e}, "
          f"energy {abs(E.item() / e_ref - 1):.2e}")
    assert err.max() <= F_TOL
    assert E.item() == pytest.approx(e_ref, rel=E_TOL)
    if n >= 1280:   # below, the energy alone keeps the FP32 loop
        assert gpu.atm_energy_raw(to_gpu(x), 1.5, eps, mp).item() == pytest.approx(e_ref, rel=E_TOL)
    gpu.simplex_device_errors()


@pytest.mark.parametrize("side,sep,eps", [(10.0, 1e-3, 1e-4), (10.0, 1e-3, 1e-8), (20.0, 1e-2, 1e-4)])
def test_contraction_near_pairs(gpu, oracle, side, sep, eps):
    x = near_coincident(700, side, 50, sep)
    F, E = gpu.atm_forces(to_gpu(x), 1.0, eps)
    G = oracle.atm_grad(x, 1.0, eps)
    kappa = oracle.atm_grad_abs(x, 1.0, eps)
    err = np.linalg.norm(F.cpu().numpy() + G, axis=1)
    assert (err <= KAPPA_C * U32 * kappa).all()
    assert E.item() == pytest.approx(oracle.atm_energy(x, 1.0, eps), rel=E_TOL)


def test_contraction_lattice_ties(gpu, oracle):
    """Equal distances everywhere: every point's nearest neighbour is a tie,
    and a triple can hold several near pairs.  A cubic lattice, slightly
    stretched along two axes."""
    g = np.stack(np.meshgrid(np.arange(9.0), 1.25 * np.arange(9.0), 1.5 * np.arange(9.0), indexing="ij"), -1)
    x = g.reshape(-1, 3).astype(np.float32)[:700]
    F, E = gpu.atm_forces(to_gpu(x), 1.0, 1e-4)
    e_ref, G = grad_all_threads(oracle, x)
    assert np.abs(F.cpu().numpy() + G).max() <= F_TOL * np.abs(G).max()
    assert E.item() == pytest.approx(e_ref, rel=E_TOL)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_contraction_not_finite(gpu, bad):
    """One coordinate that is not finite: every triple with it is not finite,
    as in the FP32 path (n = 600)."""
    for n in (600, 1700):
        x = synth.uniform_cube(n, 3, 10.0, seed=9)
        x[n // 2, 1] = bad
        F, E = gpu.atm_forces(to_gpu(x))
        assert torch.isnan(F).all() and torch.isnan(E)
        assert torch.isnan(gpu.atm_energy_raw(to_gpu(x)))
