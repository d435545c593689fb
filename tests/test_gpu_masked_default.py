"""The untuned choice of kernel on lattices with a solid mask, on both sides of each
line of its rule: the kernel it names, and the bits of another variant."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_cases import gpu_lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,shape,storage,name", [
    (O.D2Q9, (1, 6, 130), "F64", "tma_X128_s4"),
    (O.D2Q9, (1, 6, 131), "F64", "nv1_b64x4"),     # rows of no whole 16-byte words
    (O.D3Q19, (3, 4, 20), "F64", "tma_X128_s2"),
    (O.D3Q27, (3, 4, 20), "F64", "nv1_b64x4"),
    (O.D2Q9, (1, 256, 512), "F32", "nv1_b64x4"),   # 2^17 nodes
    (O.D2Q9, (1, 257, 512), "F32", "nv4_b64x4"),
    (O.D3Q19, (32, 32, 128), "F32", "nv1_b64x4"),
    (O.D3Q19, (33, 32, 128), "F32", "nv2_b64x4"),
    (O.D2Q9, (1, 529, 248), "F16", "nv1_b64x4"),   # short rows of a larger lattice
    (O.D2Q9, (1, 513, 256), "F16", "tma_X512_s4"),
    (O.D2Q9, (1, 512, 256), "F16", "nv1_b64x4"),
    (O.D3Q19, (33, 32, 128), "BF16", "nv4_b64x4"),
    (O.D3Q27, (33, 32, 128), "F32", "nv1_b64x4"),
])
def test_masked_default_variant(lat, shape, storage, name):
    rng = np.random.default_rng(53)
    solid = (rng.uniform(size=shape) < 0.1).astype(np.uint8)
    rho, u = W.random_macros(shape, O.D_OF[lat], rng, umax=0.05)
    g = gpu_lattice(lat, shape, O.P_TRT, 0.03, 0.25, storage=storage, solid=solid,
                    force=(1e-5, 0.0, 0.0))
    names = g.variants()
    assert names[g.variant] == name
    other = [v for v, n in enumerate(names) if n.startswith("nv") and v != g.variant][0]
    out = []
    for v in (g.variant, other):
        g.variant = v
        g.init_equilibrium(rho, u)
        g.step(3)
        assert g.status()[0] == 0
        out.append(g.populations().cpu().numpy()[:, solid == 0])
    assert np.array_equal(out[0], out[1])
