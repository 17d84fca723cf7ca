"""Unfolded forward at depth counts whose spectra of four (or two) volumes do
not fit a CTA's shared memory: the batch runs with fewer volumes per table pass."""
import numpy as np
import pytest

import oracle
from paper_2603_28150_gb300 import Plan, synth
from tests.helpers import cuda, host

pytestmark = pytest.mark.gpu


# 227 KB hold 113 depths of four volumes in FP64 (227 of two), twice that in
# complex FP32; below and past the first, at the second
@pytest.mark.parametrize("fp64,nz,B", [(True, 112, 4), (True, 114, 4), (True, 120, 5), (True, 227, 3),
                                       (False, 228, 4)])
def test_batches_of_many_depths_match_oracle(fp64, nz, B):
    P, n, nt = 16, 8, 3
    g = oracle.Grid.square(n, nz, nt, pad=P)
    h = synth.random_kernels(nz, nt, P, P, seed=nz)
    Hf = oracle.table_spectrum(h)
    plan = Plan(n, n, nz, nt, P, P, table=h, max_batch=B, fp64=fp64)
    assert plan.info()["folded"] == 0
    xs = np.stack([synth.gaussian_object(n, n, nz, 3 + b) for b in range(B)])
    d = host(plan.forward(cuda(xs, fp64)))
    for b in range(B):
        assert oracle.rel_l2(d[b], oracle.forward_fft(Hf, xs[b], g)) < (1e-12 if fp64 else 1e-5)
