"""Which launches are chained depends on the number of blocks: on both sides of each
line of that rule many steps in a row give the register kernel's state."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_cases import gpu_lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,shape,storage,layout", [
    (O.D2Q9, (1, 228, 24), "F64", "AB"),    # two launches of three blocks an SM fit
    (O.D2Q9, (1, 229, 24), "F64", "AB"),    # or not
    (O.D2Q9, (1, 152, 24), "F64", "AA"),    # in place: one block an SM
    (O.D2Q9, (1, 153, 24), "F64", "AA"),
    (O.D2Q9, (1, 600, 24), "F32", "AB"),    # with a capped number of blocks
    (O.D3Q19, (12, 12, 24), "F16", "AA"),   # 144 rows
    (O.D3Q19, (12, 14, 24), "BF16", "AA"),  # 168
])
def test_chained_and_plain_launches_give_one_state(lat, shape, storage, layout):
    rng = np.random.default_rng(67)
    rho, u = W.random_macros(shape, O.D_OF[lat], rng, umax=0.05)
    g = gpu_lattice(lat, shape, O.TRT_RLB, 0.03, 0.25, storage=storage, layout=layout,
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
