"""Waits of the folded contraction's table rings: with a wait limit of 0 every
warp gives up at its first step with its whole ring in flight, waits for these
copies and leaves; pat_plan_check reports it once, and at the default limit the
same calls give the same bits as before."""
import pytest

import oracle
from paper_2603_28150_gb300 import Medium, PatError, Plan, pat, synth
from tests.helpers import MED_50UM, cuda

pytestmark = pytest.mark.gpu


def timed_out(plan):
    with pytest.raises(PatError) as e:
        plan.check()
    plan.check()  # the flag was cleared
    return e.value.code == pat.PAT_ERR_TIMEOUT


def medium(nz, nt):
    return Medium(MED_50UM.c, MED_50UM.dx, MED_50UM.dy, MED_50UM.dz, MED_50UM.dt,
                  oracle.mz_for(nz, nt, MED_50UM), 1)


# one instance of the kernels each: blocks of 8 samples with two steps and one
# step in the ring, of 4 with three, two passes over the depths; time samples
# split over eight, two and one warps (their partial sums reuse the rings'
# shared memory), one and two z-groups per warp
@pytest.mark.parametrize("n,nz,nt,B", [(16, 5, 13, 1), (100, 8, 20, 1), (100, 24, 9, 1),
                                       (100, 64, 20, 1), (100, 50, 9, 3), (16, 132, 10, 2)])
def test_ring_timeout_is_reported_and_recovers(n, nz, nt, B):
    import torch
    g = oracle.Grid.square(n, nz, nt)
    plan = Plan(n, n, nz, nt, g.px, g.py, medium=medium(nz, nt), max_batch=B)
    assert plan.info()["folded"] == 1
    rho = cuda(synth.gaussian_field((B, nz, n, n), seed=3))
    d = cuda(synth.gaussian_field((B, nt, n, n), seed=4))
    ref = plan.forward(rho), plan.adjoint(d), plan.fista(d, iters=2, L=1.0)[0]
    plan.check()
    plan.set_wait_limit(0)
    for call in (lambda: plan.forward(rho), lambda: plan.adjoint(d),
                 lambda: plan.fista(d, iters=2, L=1.0)):
        call()
        assert timed_out(plan)
    plan.set_wait_limit(-1)
    got = plan.forward(rho), plan.adjoint(d), plan.fista(d, iters=2, L=1.0)[0]
    plan.check()
    assert all(torch.equal(a, b) for a, b in zip(ref, got))


def test_ring_timeout_of_a_shard():
    import torch
    n, nz, nt = 16, 5, 7
    g = oracle.Grid.square(n, nz, nt)
    shard = Plan(n, n, nz, nt, g.px, g.py, medium=medium(nz, nt), shard=(0, 1))
    W = shard.shard_info()["slot_width"]
    X = shard.shard_spectrum(0, cuda(synth.gaussian_field((nz, n, n), seed=5))).reshape(nz, W)
    Y = torch.zeros((nt, W), dtype=torch.complex64, device="cuda")
    ref = shard.shard_contract(X, Y).clone()
    shard.set_wait_limit(0)
    shard.shard_contract(X, Y)
    assert timed_out(shard)
    shard.set_wait_limit(-1)
    assert torch.equal(ref, shard.shard_contract(X, Y.zero_()))
    shard.check()
