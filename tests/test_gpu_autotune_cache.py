"""What autotune remembers for a shape is used again only where the same kernels run:
not after open boundaries (whose update ignores the variant), nor for a force where
there was none."""
import pytest
import torch

import oracle as O
from gpu_cases import gpu_lattice

pytestmark = pytest.mark.gpu


def _tune(g):
    """Whether an autotune of g timed anything (it counts its launches)."""
    g.init_equilibrium(torch.ones((1, 26, 88)), torch.zeros((2, 1, 26, 88)))
    before = g.launches
    g.autotune(reps=1, report=False)
    return g.launches > before


def test_autotune_is_not_shared_by_other_kernels():
    def lattice(force=(0.0, 0.0, 0.0)):
        return gpu_lattice(O.D2Q9, (1, 26, 88), O.P_TRT, 0.05, 0.25, storage="F64", force=force,
                           periodic=(0, 1, 1))
    g = lattice()
    g.set_open_boundaries(0.01, 1.0)
    assert _tune(g)
    assert _tune(lattice())  # closed: not the open lattice's choice
    assert not _tune(lattice())  # remembered
    assert _tune(lattice(force=(1e-6, 0.0, 0.0)))
    assert not _tune(lattice(force=(2e-6, 0.0, 0.0)))
