"""Rows that leave consumer warps of the pipelined 16-bit kernels without a node, at the edges
of a warp and of a tile: the same bits as the register kernel."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_cases import gpu_lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,shape,storage,layout", [
    (O.D2Q9, (1, 9, 16), "F16", "AB"),    # one warp of four nodes a thread has nodes
    (O.D2Q9, (1, 9, 128), "F16", "AB"),   # exactly one
    (O.D2Q9, (1, 9, 136), "BF16", "AB"),  # a few nodes of the second
    (O.D2Q9, (1, 9, 384), "F16", "AB"),   # a full 384-wide tile
    (O.D2Q9, (1, 9, 640), "F16", "AB"),   # a second tile with idle warps
    (O.D3Q19, (3, 5, 8 * 17), "F16", "AB"),
    (O.D3Q27, (3, 4, 128), "F16", "AB"),
    (O.D2Q9, (1, 9, 64), "F16", "AA"),    # one warp of two nodes a thread
    (O.D2Q9, (1, 9, 72), "BF16", "AA"),
    (O.D2Q9, (1, 9, 520), "F16", "AA"),
    (O.D3Q19, (3, 5, 136), "F16", "AA"),
])
def test_rows_with_idle_warps(lat, shape, storage, layout):
    rng = np.random.default_rng(61)
    rho, u = W.random_macros(shape, O.D_OF[lat], rng, umax=0.05)
    g = gpu_lattice(lat, shape, O.P_TRT, 0.03, 0.25, storage=storage, layout=layout,
                    force=(1e-5, 0.0, 0.0), periodic=(1, 0, 1))
    names = g.variants()
    out = {}
    for v, n in enumerate(names):
        if n.startswith("tma") or n == "nv1_b32x8":
            g.variant = v
            g.init_equilibrium(rho, u)
            g.step(5)
            assert g.status()[0] == 0
            out[n] = g.populations().cpu().numpy()
    ref = out.pop("nv1_b32x8")
    assert out
    for n, f in out.items():
        assert np.array_equal(f, ref), n
