"""||H x - y||^2 of the residual pass: the squares are widened exactly for
every kind of single-precision value. With x = 0 the residual is -y, so the
norm is the FP64 sum of y's squares whatever their size (FP64 sums of n terms:
n 2^-53 relative)."""
import numpy as np
import pytest

import oracle
from paper_2603_28150_gb300 import Plan, synth
from tests.helpers import host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P", [16, 48, 256, 512, 768])
@pytest.mark.parametrize("values", ["normal", "large", "small", "subnormal", "mixed", "zero", "inf",
                                    "nan"])
def test_residual_norm_of_any_value(P, values):
    import torch
    n, nz, nt = P // 2 - 1, 1, 3
    h = synth.random_kernels(nz, nt, P, P, seed=P, d4=True)
    plan = Plan(n, n, nz, nt, P, P, table=h)
    g = np.random.default_rng(P)
    y = g.normal(size=(nt, n, n))
    y = y * {"large": 1e30, "small": 1e-30, "subnormal": 1e-41, "zero": 0.0}.get(values, 1.0)
    if values == "mixed":
        y = y * 10.0 ** g.integers(-44, 20, size=y.shape)
    y = y.astype(np.float32)
    if values in ("inf", "nan"):
        y[1, 2, 3] = float(values)
    x = torch.zeros((nz, n, n), device="cuda")
    _, r2 = plan.gradient(x, torch.tensor(y, device="cuda"))
    ref = float(np.sum(y.astype(np.float64) ** 2))
    if np.isnan(ref):
        assert np.isnan(r2)
    elif np.isinf(ref) or ref == 0.0:
        assert r2 == ref
    else:
        assert abs(r2 - ref) <= y.size * 2.0 ** -53 * ref
