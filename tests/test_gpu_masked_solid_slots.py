"""The stored slots of solid nodes: no kernel writes them, so a checkpoint of a
masked lattice does not depend on the kernel that made it."""
import numpy as np
import pytest
import torch

import oracle as O
import workloads as W
from gpu_cases import gpu_lattice

pytestmark = pytest.mark.gpu


def _raw(g, buf, storage):
    """The stored words [Q, nz, ny, nx] of a buffer, as integers."""
    es = {"F16": 2, "BF16": 2, "F32": 4, "F64": 8}[storage]
    t = buf.view({2: torch.int16, 4: torch.int32, 8: torch.int64}[es])
    pitch = -(-g.p.nx // (16 // es)) * (16 // es)
    t = t.view(g.Q, t.numel() // g.Q)[:, :pitch * g.p.ny * g.p.nz]
    return t.reshape(g.Q, g.p.nz, g.p.ny, pitch)[..., :g.p.nx].cpu().numpy()


@pytest.mark.parametrize("lat,shape,storage", [
    (O.D2Q9, (1, 9, 520), "F16"),   # adjacent pairs, a ragged second tile
    (O.D2Q9, (1, 6, 16), "BF16"),   # the smallest row
    (O.D3Q19, (3, 5, 256), "F16"),  # a full tile
    (O.D2Q9, (1, 9, 516), "F32"),
    (O.D2Q9, (1, 6, 130), "F64"),
])
def test_solid_slots_are_not_written(lat, shape, storage):
    rng = np.random.default_rng(47)
    solid = (rng.uniform(size=shape) < 0.2).astype(np.uint8)
    solid[..., 0, 2], solid[..., 0, 3] = 1, 0  # a pair whose even node is solid
    solid[..., 0, 4], solid[..., 0, 5] = 0, 1  # and one whose odd node is
    rho, u = W.random_macros(shape, O.D_OF[lat], rng, umax=0.05)
    g = gpu_lattice(lat, shape, O.P_TRT, 0.03, 0.25, storage=storage, solid=solid)
    for v, name in enumerate(g.variants()):
        g.variant = v
        g.pop_a.fill_(0x11)
        g.pop_b.fill_(0x11)
        before = _raw(g, g.pop_b, storage)[:, solid == 1]
        g.init_equilibrium(rho, u)
        after_init = _raw(g, g.pop_a, storage)[:, solid == 1]
        g.step(2)
        assert g.status()[0] == 0
        assert np.array_equal(_raw(g, g.pop_b, storage)[:, solid == 1], before), name
        assert np.array_equal(_raw(g, g.pop_a, storage)[:, solid == 1], after_init), name
