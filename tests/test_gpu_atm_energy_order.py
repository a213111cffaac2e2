"""The ATM energy on the tensor cores is a sum in a fixed order: the same bits
from every call."""
import pytest
import torch

import synth
from helpers import to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [700, 1400, 5000])
def test_energy_repeats(gpu, n):
    x = to_gpu(synth.uniform_cube(n, 3, n ** (1 / 3), seed=n))
    assert len({gpu.atm_forces(x)[1].item() for _ in range(20)}) == 1
    assert len({gpu.atm_energy_raw(x).item() for _ in range(20)}) == 1
