"""Autotune remembers a choice per shape; with a solid mask the times depend on the mask,
so every masked lattice is timed, and what one chose is not another's."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_cases import gpu_lattice

pytestmark = pytest.mark.gpu


def test_every_masked_lattice_is_timed():
    for fill in (0.0, 0.1, 0.1):
        rng = np.random.default_rng(71)
        solid = (rng.uniform(size=(1, 30, 72)) < fill).astype(np.uint8)
        solid[0, 10:14, 20:24] = 1
        g = gpu_lattice(O.D2Q9, (1, 30, 72), O.P_TRT, 0.05, 0.25, storage="F32", solid=solid)
        g.init_equilibrium(torch.ones((1, 30, 72)), torch.zeros((2, 1, 30, 72)))
        before = g.launches
        g.autotune(reps=1, report=False)
        assert g.launches > before
