"""The fused projection stage of k_spectral.cu at N = 24, which FP32 plans do not take (their radial sum is in spectra) but
tensor-core plans of low rank and the allocation-free FP32 call do: ranks at the edges of the slot groups, per-node gamma and
b with both loss weights (the per-node loss table). And the FP32 VSS kernel at N = 32 against the FP64 oracle.

Tolerances of tests/test_gpu_parity.py, of the loss term: F16S 1e-3, BF16X3 1e-4, FP32 1e-5 (twice that for the JVP, which
has two); two results of one precision that each keep theirs differ by at most twice that.
"""
import numpy as np
import pytest
import torch

import oracle as O
from oracle import vss as V
from paper_1809_10186_gb300 import binding, workloads as W

pytestmark = pytest.mark.gpu

N, L = 24, 6.0
TOL = {"f16s": 1e-3, "bf16x3": 1e-4, "fp32": 1e-5}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1809_10186_gb300 import build
    build.build()


def _loss_norm(gamma, b, f):
    op = O.OraclePlan(N, L, gamma=gamma, b=b, M=6, Nrho=N, nyquist="sym")
    return np.linalg.norm(np.real(O.loss_Q(op, f, f)))


@pytest.mark.parametrize("prec", ["f16s", "bf16x3", "fp32"])
@pytest.mark.parametrize("rank", [1, 2, 7, 8, 17])
def test_ranks_against_fp64(prec, rank):
    kw = dict(N=N, L=L, gamma=0.4, M=6, N_rho=N, svd_rank=rank)
    f, v = (torch.from_numpy(W.two_maxwellian(2, N, L, s)[0].astype(np.float32)).cuda() for s in (1, 2))
    plan, p64 = binding.Plan(precision=prec, **kw), binding.Plan(precision="fp64", **kw)
    a, b = f[0].double().cpu().numpy(), v[0].double().cpu().numpy()
    loss = max(_loss_norm(0.4, None, a), _loss_norm(0.4, None, b))
    calls = [(plan.collide_noalloc(f), p64.collide(f.double()), 1)]
    if prec != "fp32":
        calls += [(plan.collide(f), p64.collide(f.double()), 1), (plan.collide2(f, v), p64.collide2(f.double(), v.double()), 1),
                  (plan.collide_jvp(f, v), p64.collide_jvp(f.double(), v.double()), 2)]
    for got, ref, scale in calls:
        assert (got.double() - ref).flatten(1).norm(dim=1).max().item() < TOL[prec] * scale * loss
    plan.stream_status()


@pytest.mark.parametrize("loss", ["paper", "conservative"])
@pytest.mark.parametrize("prec,rank", [("f16s", 1), ("f16s", 8), ("f16s", 17), ("bf16x3", 7)])
def test_per_node_kernel_equals_plans(prec, rank, loss):
    gam, b = [0.0, 0.52, 1.0], [0.05, 0.08, 0.11]
    F = W.two_maxwellian(3, N, L, 5)[0].astype(np.float32)
    f = torch.from_numpy(F).cuda()
    kw = dict(N=N, L=L, M=6, N_rho=N, precision=prec, svd_rank=rank, loss=loss)
    plan = binding.Plan(gamma=0.3, **kw)
    got = binding.collide_ragged([plan], [0, 0, 0], np.arange(3) * N ** 3, f.reshape(-1), node_gamma=gam, node_b=b)
    for i in range(3):
        ref = binding.Plan(gamma=gam[i], b=b[i], **kw).collide(f[i:i + 1].contiguous())
        scale = _loss_norm(gam[i], b[i], F[i].astype(np.float64))
        assert (got.reshape(3, N, N, N)[i].double() - ref[0].double()).norm().item() < 2 * TOL[prec] * scale


def test_vss_n32_one_node_against_the_oracle():
    n, half = 32, 7.0
    f = W.two_maxwellian(1, n, half, 3)[0].astype(np.float32)
    q = binding.Plan(N=n, L=half, gamma=0.4, M=6, N_rho=n, alpha=1.4, precision="fp32").collide(torch.from_numpy(f).cuda())
    op = V.VSSPlan(n, half, gamma=0.4, alpha=1.4, Nrho=n, nyquist="sym", M=6)
    a = f[0].astype(np.float64)
    loss = np.linalg.norm(a * np.real(op.idft3(op.Gloss * op.dft3(a))))
    assert np.linalg.norm(q[0].double().cpu().numpy() - V.fast_Q_vss(op, a)) < TOL["fp32"] * loss
