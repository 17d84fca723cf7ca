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
