"""Stage entry point of the contraction: what it leaves alone."""
import pytest

import oracle
from paper_2603_28150_gb300 import Medium, Plan
from tests.helpers import MED_50UM

pytestmark = pytest.mark.gpu


# rows are padded to 32 bins; P = 16 and 48 have such bins. Tensor batches and
# large spectra are converted on the way, small ones are not; ragged and whole
# groups of slices
@pytest.mark.parametrize("n,P,nz,nt,B,split", [(8, 16, 128, 128, 2, True), (24, 48, 5, 510, 8, False),
                                               (24, 48, 5, 510, 30, False), (8, 16, 9, 13, 1, False)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_padding_bins_of_the_output_are_left_alone(n, P, nz, nt, B, split, adjoint):
    import torch
    med = Medium(MED_50UM.c, MED_50UM.dx, MED_50UM.dy, MED_50UM.dz, MED_50UM.dt,
                 oracle.mz_for(nz, nt, MED_50UM), 1)
    plan = Plan(n, n, nz, nt, P, P, medium=med, max_batch=B, bf16_split=split)
    info = plan.info()
    K, Kp = info["bins"], info["bins_padded"]
    assert info["folded"] == 1 and K < Kp
    nin, nout = (nt, nz) if adjoint else (nz, nt)
    X = torch.ones((B, nin, Kp), dtype=torch.complex64, device="cuda")
    out = torch.full((B, nout, Kp), 3 - 4j, dtype=torch.complex64, device="cuda")
    plan.stage_contract(X, out, batch=B, adjoint=adjoint)
    assert bool((out[..., K:] == 3 - 4j).all())
    assert not bool((out[..., :K] == 3 - 4j).any())


def per_bin_adjoint(X, Y, D, Z):
    """Largest per-bin mismatch of sum_t Y conj(D) and sum_z X conj(Z), of the
    bound |Y||D| + |X||Z| (Cauchy-Schwarz)."""
    import torch
    X, Y, D, Z = (a.to(torch.complex128) for a in (X, Y, D, Z))
    lhs, rhs = (Y * D.conj()).sum(-2), (X * Z.conj()).sum(-2)
    size = Y.norm(dim=-2) * D.norm(dim=-2) + X.norm(dim=-2) * Z.norm(dim=-2)
    return float(((lhs - rhs).abs() / size.clamp_min(1e-30)).max())


# more CTAs than SMs: the forward on rows without rings, with two CTAs an SM and
# with one (more than 112 depths); the adjoint without rings from 64 depths on,
# in one and two z-chunks. float32 sums of at most 116 random products:
# about sqrt(116) * 2^-24 = 6.4e-7 of their size, the largest of 33024 bins some
# five times that
@pytest.mark.parametrize("n,nz,nt,B", [(128, 33, 9, 1), (128, 40, 7, 2), (128, 61, 37, 1),
                                       (128, 116, 6, 1)])
def test_rows_forward_is_the_adjoint_of_the_adjoint(n, nz, nt, B):
    import torch
    plan = Plan(n, n, nz, nt, 2 * n, 2 * n, max_batch=B,
                medium=Medium(MED_50UM.c, MED_50UM.dx, MED_50UM.dy, MED_50UM.dz, MED_50UM.dt,
                              oracle.mz_for(nz, nt, MED_50UM), 1))
    K, Kp = plan.info()["bins"], plan.info()["bins_padded"]
    gen = torch.Generator(device="cuda").manual_seed(11)
    X = torch.randn((B, nz, Kp), dtype=torch.complex64, device="cuda", generator=gen)
    D = torch.randn((B, nt, Kp), dtype=torch.complex64, device="cuda", generator=gen)
    Y = plan.stage_contract(X, torch.zeros_like(D), batch=B)
    Z = plan.stage_contract(D, torch.zeros_like(X), batch=B, adjoint=True)
    assert float(Y.abs().max()) > 0
    assert per_bin_adjoint(X[..., :K], Y[..., :K], D[..., :K], Z[..., :K]) < 1e-5


# the same on the slots of a shard: rings at few and at many depths, none between
@pytest.mark.parametrize("nz,nt", [(17, 6), (40, 7), (116, 5)])
def test_shard_forward_is_the_adjoint_of_the_adjoint(nz, nt):
    import torch
    n = 128
    shard = Plan(n, n, nz, nt, 2 * n, 2 * n, shard=(0, 1),
                 medium=Medium(MED_50UM.c, MED_50UM.dx, MED_50UM.dy, MED_50UM.dz, MED_50UM.dt,
                               oracle.mz_for(nz, nt, MED_50UM), 1))
    W = shard.shard_info()["slot_width"]
    gen = torch.Generator(device="cuda").manual_seed(12)
    X = torch.randn((nz, W), dtype=torch.complex64, device="cuda", generator=gen)
    D = torch.randn((nt, W), dtype=torch.complex64, device="cuda", generator=gen)
    Y = shard.shard_contract(X, torch.zeros_like(D))
    Z = shard.shard_contract(D, torch.zeros_like(X), adjoint=True)
    assert float(Y.abs().max()) > 0
    # slots of no bin stay zero on both sides
    assert per_bin_adjoint(X, Y, D, Z) < 1e-5
    store = torch.zeros(nt * W + 1, dtype=torch.complex64, device="cuda")
    b = shard.shard_contract(X, store[1:].view(nt, W))  # 8-byte aligned: single stores
    assert torch.equal(Y, b)


# rows of ragged groups converted in both directions (143 MB and past 32 depths)
def test_converted_rows_of_ragged_groups():
    import torch
    n, nz, nt = 256, 35, 101
    plan = Plan(n, n, nz, nt, 2 * n, 2 * n,
                medium=Medium(MED_50UM.c, MED_50UM.dx, MED_50UM.dy, MED_50UM.dz, MED_50UM.dt,
                              oracle.mz_for(nz, nt, MED_50UM), 1))
    K, Kp = plan.info()["bins"], plan.info()["bins_padded"]
    gen = torch.Generator(device="cuda").manual_seed(13)
    X = torch.randn((nz, Kp), dtype=torch.complex64, device="cuda", generator=gen)
    D = torch.randn((nt, Kp), dtype=torch.complex64, device="cuda", generator=gen)
    Y = plan.stage_contract(X, torch.zeros_like(D))
    Z = plan.stage_contract(D, torch.zeros_like(X), adjoint=True)
    assert float(Y.abs().max()) > 0 and float(Z.abs().max()) > 0
    # sums of at most 101 products: as above, over 131584 bins
    assert per_bin_adjoint(X[:, :K], Y[:, :K], D[:, :K], Z[:, :K]) < 1e-5
