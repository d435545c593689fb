"""The untuned choice of kernel of three-dimensional lattices with few short rows, on both
sides of its line, and the bits of another variant."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_cases import gpu_lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,shape,storage,name", [
    (O.D3Q27, (3, 4, 16), "F16", "tma_X256_s2_q"),
    (O.D3Q27, (19, 32, 16), "BF16", "tma_X256_s2_q"),  # 608 rows
    (O.D3Q27, (29, 21, 16), "F16", "nv1_b32x8"),       # 609
    (O.D3Q27, (24, 24, 24), "F32", "tma_X256_s2"),
    (O.D3Q27, (25, 25, 24), "F32", "nv1_b32x8"),
    (O.D3Q19, (16, 16, 64), "F16", "tma_X256_s2_q"),
    (O.D3Q19, (29, 21, 64), "F16", "nv1_b32x8"),
    (O.D3Q19, (16, 16, 64), "F32", "nv1_b32x8"),
])
def test_default_variant_of_few_rows(lat, shape, storage, name):
    rng = np.random.default_rng(59)
    rho, u = W.random_macros(shape, O.D_OF[lat], rng, umax=0.05)
    g = gpu_lattice(lat, shape, O.P_TRT, 0.03, 0.25, storage=storage)
    names = g.variants()
    assert names[g.variant] == name
    out = []
    for v in (g.variant, names.index("nv2_b32x8")):
        g.variant = v
        g.init_equilibrium(rho, u)
        g.step(5)
        assert g.status()[0] == 0
        out.append(g.populations().cpu().numpy())
    assert np.array_equal(out[0], out[1])
