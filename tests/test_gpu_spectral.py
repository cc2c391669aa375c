"""The fused Fourier stage at N = 12 and 24 and its per-node loss table (k_spectral.cu): ranks at the edges of
the slot groups, one and two loss fields, per-node gamma and b with both loss weights.

Tolerance: 1e-5 of the loss term, the FP32 tolerance of tests/test_gpu_parity.py (against FP64 plans, which take
the separate kernels at N = 24, and against the oracle at N = 12); twice that between two FP32 results.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1809_10186_gb300 import binding, workloads as W

pytestmark = pytest.mark.gpu

L_OF = {8: 3.5, 12: 4.0, 16: 5.0, 24: 6.0, 32: 7.0}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1809_10186_gb300 import build
    build.build()


def _loss_norm(N, f, g):
    op = O.OraclePlan(N, L_OF[N], gamma=0.4, M=6, Nrho=N, nyquist="sym")
    return np.linalg.norm(np.real(O.loss_Q(op, f, g)))


@pytest.mark.parametrize("rank", [1, 2, 7, 8, 24])
@pytest.mark.parametrize("N", [12, 24])
def test_ranks_against_fp64(N, rank):
    rank = min(rank, N)
    kw = dict(N=N, L=L_OF[N], gamma=0.4, M=6, N_rho=N, svd_rank=rank)
    f, v = (torch.from_numpy(W.two_maxwellian(3, N, L_OF[N], s)[0].astype(np.float32)).cuda() for s in (1, 2))
    p32, p64 = binding.Plan(precision="fp32", **kw), binding.Plan(precision="fp64", **kw)
    for got, ref, scale in ((p32.collide(f), p64.collide(f.double()), 1), (p32.collide2(f, v), p64.collide2(f.double(), v.double()), 1),
                            (p32.collide_jvp(f, v), p64.collide_jvp(f.double(), v.double()), 2)):
        loss = _loss_norm(N, f[0].double().cpu().numpy(), v[0].double().cpu().numpy())
        assert (got.double() - ref).flatten(1).norm(dim=1).max().item() < 1e-5 * scale * loss


@pytest.mark.parametrize("loss", ["paper", "conservative"])
@pytest.mark.parametrize("prec,N", [("fp64", 8), ("fp64", 12), ("fp32", 12), ("fp32", 16), ("fp32", 24), ("f16x3", 24), ("fp32", 32)])
def test_per_node_kernel_equals_plans(prec, N, loss):
    """Nodes with a gamma and b of their own against one plan per node."""
    gam, b = [0.0, 0.52, 1.0], [0.05, 0.08, 0.11]
    F = W.two_maxwellian(3, N, L_OF[N], 5)[0].astype(np.float32).astype(np.float64)
    dt = torch.float64 if prec == "fp64" else torch.float32
    f = torch.from_numpy(F).to("cuda", dt)
    kw = dict(N=N, L=L_OF[N], M=6, N_rho=N, precision=prec, loss=loss)
    plan = binding.Plan(gamma=0.3, **kw)
    got = binding.collide_ragged([plan], [0, 0, 0], np.arange(3) * N ** 3, f.reshape(-1), node_gamma=gam, node_b=b)
    tol = 2e-10 if prec == "fp64" else 2e-5
    for i in range(3):
        ref = binding.Plan(gamma=gam[i], b=b[i], **kw).collide(f[i:i + 1].contiguous())
        op = O.OraclePlan(N, L_OF[N], gamma=gam[i], b=b[i], M=6, Nrho=N, nyquist="sym")
        scale = np.linalg.norm(np.real(O.loss_Q(op, F[i], F[i])))
        assert (got.reshape(3, N, N, N)[i].double() - ref[0].double()).norm().item() < tol * scale
