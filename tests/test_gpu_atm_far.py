"""ATM energy and forces on the tensor cores: points so far apart that the
square of their distance overflows FP32."""
import numpy as np
import pytest
import torch

import synth
from helpers import grad_all_threads, to_gpu
from test_gpu_atm import E_TOL, F_TOL, atom_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("far", [1e15, 1e25])
def test_far_points(gpu, oracle, far):
    """Two points parked far away: their triples vanish, the others' do not
    change (as in the FP32 loop of the energy, which n = 600 takes)."""
    n = 1400
    x = synth.uniform_cube(n, 3, n ** (1 / 3), seed=n)
    x[n // 2], x[n - 1] = (far, 0, 0), (0, -far, 0)
    rest = np.delete(x, [n // 2, n - 1], axis=0)
    e_ref, G = grad_all_threads(oracle, rest, 1.0, 1e-4)
    assert gpu.atm_energy_raw(to_gpu(x), 1.0, 1e-4).item() == pytest.approx(e_ref, rel=E_TOL)
    F, E = gpu.atm_forces(to_gpu(x), 1.0, 1e-4)
    F = F.cpu().numpy()
    assert E.item() == pytest.approx(e_ref, rel=E_TOL)
    assert np.abs(F[[n // 2, n - 1]]).max() <= 1e-30
    assert atom_err(np.delete(F, [n // 2, n - 1], axis=0), G).max() <= F_TOL
    assert torch.isfinite(gpu.atm_energy_raw(to_gpu(np.delete(x, range(800), axis=0)), 1.0, 1e-4))
