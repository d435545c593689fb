"""The pipelined update on lattices with a solid mask, against the register
kernel of the same library: the same bits, wherever the solid nodes lie (row ends,
tile and warp edges, whole warps without one, beside walls)."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_cases import gpu_lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,shape,storage,periodic", [
    (O.D2Q9, (1, 9, 516), "F32", (1, 1, 1)),    # a second tile of four nodes
    (O.D2Q9, (1, 9, 1024), "F32", (0, 1, 1)),   # x walls
    (O.D2Q9, (1, 1, 8), "F32", (1, 1, 1)),      # smallest row: its own neighbour
    (O.D2Q9, (1, 7, 536), "F16", (1, 0, 1)),    # adjacent node pairs, y walls
    (O.D2Q9, (1, 6, 130), "F64", (1, 1, 1)),    # one node per thread
    (O.D3Q19, (4, 5, 260), "F32", (1, 1, 1)),
    (O.D3Q19, (3, 4, 64), "BF16", (0, 0, 0)),   # a closed box
    (O.D3Q27, (3, 4, 40), "F32", (1, 1, 0)),
])
def test_masked_pipeline_matches_register_kernel(lat, shape, storage, periodic):
    rng = np.random.default_rng(41)
    solid = (rng.uniform(size=shape) < 0.03).astype(np.uint8)
    solid[..., :1, 0] = 1
    solid[..., -1:, -1] = 1
    if shape[2] > 64:
        solid[..., 96:200] = 0  # warps with no solid node in reach
    rho, u = W.random_macros(shape, O.D_OF[lat], rng, umax=0.05)
    g = gpu_lattice(lat, shape, O.P_TRT, 0.03, 0.25, storage=storage, force=(1e-5, 0, 0),
                    periodic=periodic, solid=solid)
    names = g.variants()
    tma = [v for v, n in enumerate(names) if n.startswith("tma")]
    reg = [v for v, n in enumerate(names) if not n.startswith("tma")][0]
    assert tma
    out = {}
    for v in [reg] + tma:
        g.variant = v
        g.init_equilibrium(rho, u)
        g.step(6)
        assert g.status()[0] == 0
        out[v] = g.populations().cpu().numpy()[:, solid == 0]
    for v in tma:
        assert np.array_equal(out[v], out[reg]), names[v]
