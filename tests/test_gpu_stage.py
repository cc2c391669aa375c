"""The Fourier stage in spectra (capi.cu stage_in_spectra, tc_stage_in_spectra; k_shift_sum.cu): ranks at the edges of
its rules against the stage by projection, and results that do not depend on the batch.

Tolerances: 1e-5 of the loss term, the FP32 tolerance of tests/test_gpu_parity.py; twice that between two FP32 results.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1809_10186_gb300 import binding, workloads as W

pytestmark = pytest.mark.gpu

L_OF = {12: 4.0, 16: 5.0, 24: 6.0, 32: 7.0}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1809_10186_gb300 import build
    build.build()


def _fields(N, B, seed):
    return torch.from_numpy(W.two_maxwellian(B, N, L_OF[N], seed)[0].astype(np.float32)).cuda()


def _loss_norm(N, f, g):
    op = O.OraclePlan(N, L_OF[N], gamma=0.4, M=6, Nrho=N, nyquist="sym")
    return np.linalg.norm(np.real(O.loss_Q(op, f.double().cpu().numpy(), g.double().cpu().numpy())))


@pytest.mark.parametrize("Nrho,rank", [(32, 15), (32, 16), (32, 24), (9, 5), (1, 1)])
def test_fp32_ranks_at_n32_against_fp64(Nrho, rank):
    """FP64 plans of up to three quarters of the full rank take the projection."""
    N = 32
    kw = dict(N=N, L=L_OF[N], gamma=0.4, M=6, N_rho=Nrho, svd_rank=rank)
    f, v = _fields(N, 2, 1), _fields(N, 2, 2)
    p32, p64 = binding.Plan(precision="fp32", **kw), binding.Plan(precision="fp64", **kw)
    for got, ref, scale in ((p32.collide(f), p64.collide(f.double()), 1), (p32.collide2(f, v), p64.collide2(f.double(), v.double()), 1),
                            (p32.collide_jvp(f, v), p64.collide_jvp(f.double(), v.double()), 2)):
        assert (got.double() - ref).flatten(1).norm(dim=1).max().item() < 1e-5 * scale * _loss_norm(N, f[0], v[0])


@pytest.mark.parametrize("N,projected,rank", [(24, 17, 18), (24, 17, 24), (32, 19, 20), (32, 19, 32)])
def test_tensor_core_stage_against_the_projection(N, projected, rank):
    """Ranks on both sides of the rule: the factors above `projected` carry less than 1e-7 of the kernel."""
    f, v = _fields(N, 3, 3), _fields(N, 3, 4)
    kw = dict(N=N, L=L_OF[N], gamma=0.4, M=6, N_rho=N, precision="f16s")
    a, b = binding.Plan(svd_rank=projected, **kw), binding.Plan(svd_rank=rank, **kw)
    loss = _loss_norm(N, f[0], v[0])
    for got, ref, scale in ((b.collide(f), a.collide(f), 1), (b.collide2(f, v), a.collide2(f, v), 1),
                            (b.collide_jvp(f, v), a.collide_jvp(f, v), 2)):
        assert (got.double() - ref.double()).flatten(1).norm(dim=1).max().item() < 2e-5 * scale * loss


@pytest.mark.parametrize("loss", ["paper", "conservative"])
@pytest.mark.parametrize("N", [24, 32])
def test_tensor_core_per_node_kernel_equals_plans(N, loss):
    gam, b = [0.0, 0.52, 1.0], [0.05, 0.08, 0.11]
    kw = dict(N=N, L=L_OF[N], M=6, N_rho=N, precision="f16s", loss=loss)
    f = _fields(N, 3, 5)
    got = binding.collide_ragged([binding.Plan(gamma=0.3, **kw)], [0, 0, 0], np.arange(3) * N ** 3, f.reshape(-1), node_gamma=gam, node_b=b)
    for i in range(3):
        ref = binding.Plan(gamma=gam[i], b=b[i], **kw).collide(f[i:i + 1].contiguous())
        op = O.OraclePlan(N, L_OF[N], gamma=gam[i], b=b[i], M=6, Nrho=N, nyquist="sym")
        F = f[i].double().cpu().numpy()
        scale = np.linalg.norm(np.real(O.loss_Q(op, F, F)))
        assert (got.reshape(3, N, N, N)[i].double() - ref[0].double()).norm().item() < 2e-5 * scale


@pytest.mark.parametrize("prec,N,B,kw", [("fp32", 12, 160, {}), ("fp32", 24, 60, {}), ("fp32", 24, 60, dict(N_rho=13)), ("fp32", 32, 45, {}),
                                         ("f16s", 32, 45, {}), ("f16s", 24, 60, {}), ("fp64", 16, 160, {}),
                                         ("fp32", 16, 60, dict(alpha=1.3)), ("fp64", 12, 20, dict(alpha=1.3))])
def test_a_node_does_not_depend_on_its_batch(prec, N, B, kw):
    """One node, many nodes (sums in one block per column), and one node at a time with a workspace of one node
    (sums over part of the radial points per launch) give the same bits."""
    plan = binding.Plan(**{**dict(N=N, L=L_OF[N], gamma=0.4, M=12, N_rho=N, precision=prec), **kw})
    small = binding.Plan(**{**dict(N=N, L=L_OF[N], gamma=0.4, M=12, N_rho=N, precision=prec, max_batch=1), **kw})
    f = _fields(N, B, 7).to(plan.dtype)
    q = plan.collide(f)
    for i in (0, B - 1):
        assert torch.equal(plan.collide(f[i:i + 1].contiguous())[0], q[i])
        assert torch.equal(small.collide(f[i:i + 1].contiguous())[0], q[i])
    assert torch.equal(small.collide(f[:3].contiguous()), q[:3])
