"""Folded CUDA-core contraction on spectra interleaved by eight slices: depth
and time counts around the tiles (groups and quads of slices, blocks of 4 / 8
samples, stages, rings, z-chunks, the second pass past 128 depths), every transform
length's thread layout, several volumes, and the plain layout of the stage
entry point, against the FP64 oracle (FP32 target: 1e-5 relative l2)."""
import numpy as np
import pytest

import oracle
from paper_2603_28150_gb300 import PatError, Plan, synth
from tests.helpers import cuda, host

pytestmark = pytest.mark.gpu

# (n, P, nz, nt, B): the smallest counts, one past and one short of a group,
# ragged time blocks, few and many z-groups, the largest depth count
SHAPES = [(8, 16, 1, 1, 1), (8, 16, 3, 2, 2), (12, 24, 4, 3, 1), (16, 32, 5, 5, 3),
          (24, 48, 17, 13, 1), (32, 64, 9, 65, 2), (48, 96, 33, 31, 1), (64, 128, 49, 40, 1),
          (64, 128, 12, 7, 4), (90, 192, 21, 18, 1), (8, 16, 66, 9, 1), (8, 16, 130, 34, 1),
          (8, 16, 224, 6, 2), (128, 256, 6, 9, 1), (150, 384, 2, 5, 1), (256, 512, 5, 3, 1),
          (300, 768, 1, 6, 1), (512, 1024, 1, 2, 1)]


@pytest.mark.parametrize("n,P,nz,nt,B", SHAPES, ids=[str(s) for s in SHAPES])
def test_folded_groups_match_oracle(n, P, nz, nt, B):
    import torch
    g = oracle.Grid(nx=n, ny=max(1, n - 3), nz=nz, nt=nt, px=P, py=P)
    h = synth.random_kernels(nz, nt, P, P, seed=n + nz, d4=True)
    plan = Plan(g.nx, g.ny, nz, nt, P, P, table=h, max_batch=B)
    assert plan.info()["folded"] == 1
    Hf = oracle.table_spectrum(h)
    xs = np.stack([synth.gaussian_object(g.nx, g.ny, nz, 5 + b) for b in range(B)])
    ys = np.stack([synth.gaussian_field((nt, g.ny, g.nx), 15 + b) for b in range(B)])
    d, a = host(plan.forward(cuda(xs))), host(plan.adjoint(cuda(ys)))
    gr, r2 = plan.gradient(cuda(xs), cuda(ys))
    gr = host(gr)
    r2_ref = 0.0
    for b in range(B):
        d_ref, a_ref = oracle.forward_fft(Hf, xs[b], g), oracle.adjoint_fft(Hf, ys[b], g)
        assert oracle.rel_l2(d[b], d_ref) < 1e-5
        assert oracle.rel_l2(a[b], a_ref) < 1e-5
        assert oracle.rel_l2(gr[b], oracle.adjoint_fft(Hf, d_ref - ys[b], g)) < 1e-5
        r2_ref += float(np.sum((d_ref - ys[b]) ** 2))
    assert abs(r2 - r2_ref) < 1e-5 * r2_ref
    # the stage entry point keeps one row of bins per slice
    K, Kp = plan.info()["bins"], plan.info()["bins_padded"]
    rng = np.random.default_rng(nz)
    Hk = np.moveaxis(Hf[:, :, :, :P // 2 + 1].real, 3, 2).reshape(nz, nt, K) / (P * P)
    for adj in (False, True):
        rin, rout = (nt, nz) if adj else (nz, nt)
        X = rng.normal(size=(rin, K)) + 1j * rng.normal(size=(rin, K))
        Xt = torch.zeros((rin, Kp), dtype=torch.complex64, device="cuda")
        Xt[:, :K] = torch.tensor(X, dtype=torch.complex64)
        out = torch.zeros((rout, Kp), dtype=torch.complex64, device="cuda")
        plan.stage_contract(Xt, out, adjoint=adj)
        got = out[:, :K].cpu().numpy().astype(np.complex128)
        ref = np.einsum("ztk,tk->zk" if adj else "ztk,zk->tk", Hk, X)
        assert np.linalg.norm(got - ref) < 1e-5 * np.linalg.norm(ref)


def test_more_depths_than_the_forward_holds_stay_refused():
    P, nz = 16, 225
    h = synth.random_kernels(nz, 2, P, P, seed=3, d4=True)
    plan = Plan(8, 8, nz, 2, P, P, table=h)
    assert plan.info()["folded"] == 1
    with pytest.raises(PatError):
        plan.forward(cuda(np.zeros((nz, 8, 8))))
