"""FP64 adjoint contraction at depth counts around its splits of the depth
groups over chunks and warps (real tables: two depths a group, complex: one)."""
import numpy as np
import pytest

import oracle
from paper_2603_28150_gb300 import Plan, synth
from tests.helpers import cuda, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("even", [True, False])
@pytest.mark.parametrize("nz", [16, 17, 33, 34, 48, 50, 65])
@pytest.mark.parametrize("B", [1, 3])
def test_fp64_adjoint_depth_groups(nz, B, even):
    g = oracle.Grid(nx=8, ny=7, nz=nz, nt=11, px=16, py=16)
    h = synth.random_kernels(nz, g.nt, 16, 16, seed=nz, d4=even)
    plan = Plan(g.nx, g.ny, nz, g.nt, 16, 16, table=h, fp64=True, max_batch=B)
    Hf = oracle.table_spectrum(h)
    ys = np.stack([synth.gaussian_field((g.nt, g.ny, g.nx), 15 + b) for b in range(B)])
    a = host(plan.adjoint(cuda(ys, fp64=True)))
    for b in range(B):
        # double precision against the FP64 oracle, as for every FP64 plan
        assert oracle.rel_l2(a[b], oracle.adjoint_fft(Hf, ys[b], g)) < 1e-12
