"""Which launches are chained depends on the number of blocks: on both sides of each
line of that rule many steps in a row give the register kernel's state."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_cases import gpu_lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny,storage,layout", [
    (228, "F64", "AB"), (229, "F64", "AB"),  # two launches of three blocks an SM fit, or not
    (152, "F64", "AA"), (153, "F64", "AA"),  # in place: one block an SM
    (600, "F32", "AB"),                      # with a capped number of blocks
])
def test_chained_and_plain_launches_give_one_state(ny, storage, layout):
    rng = np.random.default_rng(67)
    shape = (1, ny, 24)
    rho, u = W.random_macros(shape, 2, rng, umax=0.05)
    g = gpu_lattice(O.D2Q9, shape, O.TRT_RLB, 0.03, 0.25, storage=storage, layout=layout,
                    force=(1e-5, 0.0, 0.0), periodic=(1, 0, 1))
    names = g.variants()
    out = {}
    for n in ("nv1_b32x8", "tma_X256_s4", "tma_X256_s2", "tma_X256_s2_b2"):
        if n not in names:
            continue
        g.variant = names.index(n)
        g.init_equilibrium(rho, u)
        g.step(40)
        assert g.status()[0] == 0
        out[n] = g.populations().cpu().numpy()
    ref = out.pop("nv1_b32x8")
    assert out
    for n, f in out.items():
        assert np.array_equal(f, ref), n
