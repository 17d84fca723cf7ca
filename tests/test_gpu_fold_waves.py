"""Folded forward with many CTAs against the same volumes one by one (few CTAs:
blocks of 4 time samples with three steps in the ring): more CTAs than fit the
GPU twice (blocks of 8 with one step, at any depth count), and 65 to 80 depths
on three quarters of the places or more (blocks of 4 with two steps)."""
import pytest

import oracle
from paper_2603_28150_gb300 import Medium, Plan, synth
from tests.helpers import MED_50UM, cuda

pytestmark = pytest.mark.gpu


# depths: two CTAs an SM, one, all that are resident, and a second pass
@pytest.mark.parametrize("nz,nt,B", [(50, 7, 40), (84, 13, 40), (128, 8, 40), (132, 9, 40),
                                     (65, 9, 16), (80, 6, 16)])
def test_many_volumes_match_single_ones(nz, nt, B):
    n = 32
    g = oracle.Grid.square(n, nz, nt)
    plan = Plan(n, n, nz, nt, g.px, g.py, max_batch=B,
                medium=Medium(MED_50UM.c, MED_50UM.dx, MED_50UM.dy, MED_50UM.dz, MED_50UM.dt,
                              oracle.mz_for(nz, nt, MED_50UM), 1))
    info = plan.info()
    assert info["folded"] == 1 and info["table_rows"] // 32 * B >= (608 if B == 40 else 229)
    rho = cuda(synth.gaussian_field((B, nz, n, n), seed=nz))
    d = plan.forward(rho)
    for b in range(B):
        ref = plan.forward(rho[b:b + 1].contiguous())[0]
        # the same float32 products summed over depths in the same order; only
        # the split of the passes differs: rounding of one sum
        assert float((d[b] - ref).norm()) <= 1e-6 * float(ref.norm())
