"""Autotune remembers a choice per shape; on an A/B lattice with a solid mask the times
depend on the mask, so each is timed, and what one chose is not another's. In
place, where a trial advances the lattice, the choice is remembered."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_cases import gpu_lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", ["AB", "AA"])
def test_masked_lattices_are_timed_where_that_is_free(layout):
    for k, fill in enumerate((0.0, 0.1, 0.1)):
        rng = np.random.default_rng(71)
        solid = (rng.uniform(size=(1, 30, 72)) < fill).astype(np.uint8)
        solid[0, 10:14, 20:24] = 1
        g = gpu_lattice(O.D2Q9, (1, 30, 72), O.P_TRT, 0.05, 0.25, storage="F32", solid=solid,
                        layout=layout)
        g.init_equilibrium(torch.ones((1, 30, 72)), torch.zeros((2, 1, 30, 72)))
        before, t = g.launches, g.t
        g.autotune(reps=1, report=False)
        if layout == "AB" or k == 0:
            assert g.launches > before
        else:
            assert g.launches == before and g.t == t
