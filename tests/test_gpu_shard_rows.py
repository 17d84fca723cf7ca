"""Folded contraction on the exchange slots of a frequency shard: a
representative's four slots are stored with one 32-byte access per time
sample where they are aligned, else one by one. Ragged sample counts, and
output buffers that are not 32-byte aligned."""
import pytest

import oracle
from paper_2603_28150_gb300 import Medium, Plan, synth
from paper_2603_28150_gb300.shard import ShardedOperator
from tests.helpers import MED_50UM, cuda

pytestmark = pytest.mark.gpu


class OneRank:
    def all_to_all(self, send):
        return send

    def sum(self, value, device):
        return value


# nt off and on whole quads and blocks of eight; 132 depths take two passes
# over the resident spectra (the second adds to what the first stored)
@pytest.mark.parametrize("n,nz,nt", [(16, 3, 1), (16, 5, 7), (32, 16, 13), (32, 33, 64),
                                     (16, 132, 10)])
def test_shard_contraction_stores(n, nz, nt):
    import torch
    g = oracle.Grid.square(n, nz, nt)
    med = Medium(MED_50UM.c, MED_50UM.dx, MED_50UM.dy, MED_50UM.dz, MED_50UM.dt,
                 oracle.mz_for(nz, nt, MED_50UM), 1)
    full = Plan(n, n, nz, nt, g.px, g.py, medium=med)
    shard = Plan(n, n, nz, nt, g.px, g.py, medium=med, shard=(0, 1))
    rho = cuda(synth.gaussian_field((nz, n, n), seed=5))
    d = ShardedOperator(shard, OneRank()).forward(rho)
    ref = full.forward(rho)
    # the same float32 sums over depths in the same order but for the FFTs'
    # row pairing: rounding of the stages, as for the sharded operator
    assert float((d - ref).norm()) <= 1e-6 * float(ref.norm())

    W = shard.shard_info()["slot_width"]
    X = shard.shard_spectrum(0, rho).reshape(nz, W)
    a = torch.zeros((nt, W), dtype=torch.complex64, device="cuda")
    shard.shard_contract(X, a)
    store = torch.zeros(nt * W + 1, dtype=torch.complex64, device="cuda")
    b = store[1:].view(nt, W)  # 8-byte aligned: single stores
    shard.shard_contract(X, b)
    assert float(a.abs().max()) > 0 and torch.equal(a, b)


# the stage entry on rows of several volumes with ragged last groups: in rows,
# and (five volumes at 128^2: 133 MB) converted to groups and back, against
# single volumes in rows
@pytest.mark.parametrize("n,nz,nt,B", [(16, 5, 13, 3), (16, 1, 9, 2), (128, 5, 101, 5)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_stage_rows_of_several_volumes(n, nz, nt, B, adjoint):
    import torch
    med = Medium(MED_50UM.c, MED_50UM.dx, MED_50UM.dy, MED_50UM.dz, MED_50UM.dt,
                 oracle.mz_for(nz, nt, MED_50UM), 1)
    plan = Plan(n, n, nz, nt, 2 * n, 2 * n, medium=med, max_batch=B)
    assert plan.info()["folded"] == 1
    Kp = plan.info()["bins_padded"]
    nin, nout = (nt, nz) if adjoint else (nz, nt)
    gen = torch.Generator(device="cuda").manual_seed(7)
    X = torch.randn((B, nin, Kp), dtype=torch.complex64, device="cuda", generator=gen)
    K = plan.info()["bins"]
    Y = plan.stage_contract(X, torch.zeros((B, nout, Kp), dtype=torch.complex64, device="cuda"),
                            batch=B, adjoint=adjoint)[..., :K]
    for b in range(B):
        y = plan.stage_contract(X[b].contiguous(), torch.zeros((nout, Kp), dtype=torch.complex64,
                                                               device="cuda"), adjoint=adjoint)
        # sums of at most 101 float32 products, their order free: about
        # sqrt(101) * 2^-24 of the terms' size, 1.2e-5 if every error added up
        assert float((Y[b] - y[..., :K]).norm()) <= 1e-5 * float(y[..., :K].norm())
