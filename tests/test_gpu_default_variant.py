"""The untuned choice of kernel on both sides of each line of its rule: the kernel
it names, and the same bits as another variant."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_cases import gpu_lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,shape,storage,layout,periodic,name", [
    (O.D2Q9, (1, 6, 256), "F32", "AB", (1, 1, 1), "tma2_X256_s3"),
    (O.D2Q9, (1, 6, 257), "F32", "AB", (1, 1, 1), "tma2_X512_s3"),
    (O.D2Q9, (1, 2048, 512), "F16", "AB", (1, 1, 1), "tma_X512_s2_q"),
    (O.D2Q9, (1, 2047, 512), "F16", "AB", (1, 1, 1), "tma2_X512_s3"),
    (O.D2Q9, (1, 6, 256), "F32", "AB", (1, 0, 1), "tma_X512_s4"),
    (O.D3Q19, (3, 4, 124), "F32", "AB", (1, 1, 1), "nv1_b32x8"),
    (O.D3Q19, (3, 4, 128), "F32", "AB", (1, 1, 1), "tma_X256_s2"),
    (O.D3Q19, (3, 4, 384), "F32", "AB", (1, 1, 1), "tma_X384_s2"),
    (O.D3Q19, (3, 4, 88), "F16", "AB", (1, 1, 1), "nv1_b32x8"),
    (O.D3Q19, (3, 4, 96), "F16", "AB", (1, 1, 1), "tma_X256_s2_q"),
    (O.D3Q19, (3, 4, 96), "F64", "AB", (1, 1, 1), "tma_X128_s2"),
    (O.D3Q19, (3, 4, 256), "F64", "AB", (1, 1, 1), "tma_X256_s2"),
    (O.D3Q19, (3, 4, 168), "F32", "AA", (1, 1, 1), "nv1_b32x8"),
    (O.D3Q19, (3, 4, 172), "F32", "AA", (1, 1, 1), "tma_X256_s2"),
    (O.D3Q27, (3, 4, 192), "F32", "AB", (1, 1, 1), "tma_X256_s2"),
])
def test_default_variant(lat, shape, storage, layout, periodic, name):
    rng = np.random.default_rng(43)
    rho, u = W.random_macros(shape, O.D_OF[lat], rng, umax=0.05)
    g = gpu_lattice(lat, shape, O.P_TRT, 0.03, 0.25, storage=storage, layout=layout,
                    periodic=periodic)
    names = g.variants()
    assert names[g.variant] == name
    out = []
    for v in (g.variant, [k for k, n in enumerate(names) if n.startswith("nv1")][1]):
        g.variant = v
        g.init_equilibrium(rho, u)
        g.step(5)
        assert g.status()[0] == 0
        out.append(g.populations().cpu().numpy())
    if storage == "F64":  # the two kernels may contract the force-free sums differently
        assert np.max(np.abs(out[0] - out[1])) < 5 * 64 * 2.0 ** -53
    else:
        assert np.array_equal(out[0], out[1])
