"""Folded forward with more CTAs than fit the GPU twice (blocks of 8 time
samples with one step in the ring, at any depth count) against the same
volumes one by one (few CTAs: blocks of 4)."""
import pytest

import oracle
from paper_2603_28150_gb300 import Medium, Plan, synth
from tests.helpers import MED_50UM, cuda

pytestmark = pytest.mark.gpu


# depths: two CTAs an SM, one, all that are resident, and a second pass
@pytest.mark.parametrize("nz,nt", [(50, 7), (84, 13), (128, 8), (132, 9)])
def test_many_volumes_match_single_ones(nz, nt):
    n, B = 32, 40
    g = oracle.Grid.square(n, nz, nt)
    plan = Plan(n, n, nz, nt, g.px, g.py, max_batch=B,
                medium=Medium(MED_50UM.c, MED_50UM.dx, MED_50UM.dy, MED_50UM.dz, MED_50UM.dt,
                              oracle.mz_for(nz, nt, MED_50UM), 1))
    info = plan.info()
    assert info["folded"] == 1 and info["table_rows"] // 32 * B >= 608
    rho = cuda(synth.gaussian_field((B, nz, n, n), seed=nz))
    d = plan.forward(rho)
    for b in range(B):
        ref = plan.forward(rho[b:b + 1].contiguous())[0]
        # the same float32 products summed over depths in the same order; only
        # the split of the passes differs: rounding of one sum
        assert float((d[b] - ref).norm()) <= 1e-6 * float(ref.norm())
