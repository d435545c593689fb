"""The kernel that takes two time steps per launch (periodic D2Q9, 32- and 16-bit
storage, A/B layout), against the register kernel of the same library: both round
the state to the storage type after every step and run the same collision, so they agree bit for
bit.  Also the FP64 update's conservation of momentum over many steps."""
import numpy as np
import pytest
import torch

import oracle as O
import workloads as W
from gpu_cases import gpu_lattice

pytestmark = pytest.mark.gpu


def _variants(g, prefix):
    return [v for v, n in enumerate(g.variants()) if n.startswith(prefix)]


@pytest.mark.parametrize("nx,ny,storage,coll,force,steps", [
    (8, 1, "F32", O.P_TRT, (0.0, 0.0, 0.0), 4),       # smallest rows: both wraps in one window
    (12, 2, "F32", O.TRT, (1e-5, 2e-5, 0.0), 9),      # fewer rows than ring stages, one single step
    (60, 33, "F32", O.P_TRT, (0.0, 0.0, 0.0), 3),     # no pair fits: single steps only
    (256, 40, "F32", O.TRT_RLB, (0.0, 0.0, 0.0), 8),  # one full strip
    (260, 7, "F32", O.P_TRT, (1e-5, 0.0, 0.0), 6),    # two strips of 256-wide tiles, two steps left over
    (516, 331, "F32", O.P_TRT, (0.0, 0.0, 0.0), 12),  # ragged strips, many row chunks
    (1276, 90, "F32", O.TRT, (0.0, 0.0, 0.0), 5),     # strips of unequal width
    (9, 5, "F32", O.P_TRT, (0.0, 0.0, 0.0), 8),      # row ends within a 16-byte word: one node
    (1023, 61, "F32", O.P_TRT, (0.0, 0.0, 0.0), 8),  # three of four
    (4097, 6, "F32", O.P_TRT, (0.0, 0.0, 0.0), 4),   # a last strip of one node is avoided
    (17, 7, "F16", O.P_TRT, (0.0, 0.0, 0.0), 8),     # one of eight
    (522, 25, "F16", O.TRT, (0.0, 1e-5, 0.0), 8),  # two of eight, two strips
    (768, 31, "BF16", O.P_TRT, (1e-5, 0.0, 0.0), 8),
])
def test_two_steps_per_launch_match_single_steps(nx, ny, storage, coll, force, steps):
    rng = np.random.default_rng(31)
    rho, u = W.random_macros((1, ny, nx), 2, rng, umax=0.05)
    g = gpu_lattice(O.D2Q9, (1, ny, nx), coll, 0.03, 0.25, storage=storage, force=force)
    two = _variants(g, "tma2")
    one = [v for v, n in enumerate(g.variants()) if not n.startswith("tma")][0]
    assert two

    def run(v):
        g.variant = v
        g.init_equilibrium(rho, u)
        g.step(steps)
        assert g.status()[0] == 0 and g.t == steps
        return g.populations().cpu().numpy(), g.pop_a.clone(), g.pop_b.clone()

    ref, _, _ = run(one)
    for v in two:
        f, a, b = run(v)
        # up to the sign of zero: the force-free path skips adding zero forces
        assert np.array_equal(f, ref), g.variants()[v]
        # the state is in the buffer that the step count gives it, whatever ran
        ck, t = g.checkpoint()
        want = (b if steps % 2 else a).view(torch.uint8)
        assert t == steps and torch.equal(ck, want)


def test_two_step_divergence_is_the_first_bad_step():
    rng = np.random.default_rng(32)
    rho, u = W.random_macros((1, 40, 520), 2, rng, umax=0.05)
    u[0, 0, 17, 300] = 0.97  # |u| > 1 within a few steps
    g = gpu_lattice(O.D2Q9, (1, 40, 520), O.TRT, 1e-4, 0.25, storage="F32")
    got = []
    for v in [_variants(g, "nv")[0]] + _variants(g, "tma2"):
        g.variant = v
        g.init_equilibrium(rho, u)
        g.step(40)
        got.append(g.status())
    assert got[0][1] >= 0 and all(s == got[0] for s in got), got


def test_two_step_wait_runs_out_and_reports():
    """Bytes that never arrive: every warp gives up within the limit, none is left
    at the block barrier, the error word is set, and the context stays usable."""
    rng = np.random.default_rng(33)
    rho, u = W.random_macros((1, 64, 256), 2, rng, umax=0.05)
    g = gpu_lattice(O.D2Q9, (1, 64, 256), O.P_TRT, 0.03, 0.25, storage="F32")
    g.variant = _variants(g, "tma2")[0]
    g.init_equilibrium(rho, u)
    g.set_wait_limit(0.2, 64)
    g.step(4)
    from paper_2602_06686_gb300 import LBMError
    with pytest.raises(LBMError) as e:
        g.status()
    assert e.value.code == -4
    g.set_wait_limit(2.0, 0)
    g.init_equilibrium(rho, u)
    g.step(8)
    assert g.status()[0] == 0
