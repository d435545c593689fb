"""Conservation of momentum by the FP64 update over many steps."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from gpu_cases import gpu_lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lat,shape", [(O.D2Q9, (1, 64, 64)), (O.D3Q19, (16, 16, 16))])
@pytest.mark.parametrize("coll", [O.P_TRT, O.TRT])
def test_fp64_momentum_does_not_drift(lat, shape, coll):
    """The relaxation multiplies the momentum by cm + 36 wmd at every step; with
    both rounded to nearest that product is off by up to 1.7e-16 (1/tau- = 1.99) and
    2000 steps drift by 3e-13.  The bound is a sixth of that; what rounding of the
    populations leaves is random from node to node and averages out."""
    rng = np.random.default_rng(34)
    rho, u = W.random_macros(shape, O.D_OF[lat], rng, umax=0.01)
    u[0] += 0.05
    g = gpu_lattice(lat, shape, coll, 0.05, 0.15 * (1.0 / 1.99 - 0.5), storage="F64")
    g.init_equilibrium(rho, u)
    m0 = g.diagnostics()["momentum"][0]
    g.step(2000)
    m1 = g.diagnostics()["momentum"][0]
    assert abs(m1 - m0) < 5e-14 * abs(m0)
