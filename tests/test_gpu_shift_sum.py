"""The VSS kernel and the adjoint on the shared translates (k_shift_sum.cu): rules that share shifts, that share none
and that have points on both sides of x = 0, odd product counts, the packed kz = 0 plane with rough inputs (Nyquist
content), few and many items, and a workspace that holds few radial points.

Tolerances: 1e-10 (FP64) and 1e-5 (FP32) of the loss term, those of tests/test_gpu_parity.py.
"""
import numpy as np
import pytest
import torch

import oracle as O
from oracle import vss as V
from paper_1809_10186_gb300 import binding, workloads as W

from test_gpu_shift import _oracle, _rule

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-10, "fp32": 1e-5}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1809_10186_gb300 import build
    build.build()


def _fields(B, N, prec):
    dt = torch.float64 if prec == "fp64" else torch.float32
    return [torch.from_numpy(W.rough(B, N, s)).to("cuda", dt) for s in (1, 2)]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("kind", ["generic", "planes", "no_x"])
@pytest.mark.parametrize("N,max_batch", [(8, 0), (12, 0), (12, 1)])
def test_vjp_rules_against_oracle(prec, kind, N, max_batch):
    rule, (f, u) = _rule(kind), _fields(3, N, prec)
    plan = binding.Plan(N=N, L=4.0, gamma=0.4, sphere=rule, N_rho=N, precision=prec, max_batch=max_batch)
    op = _oracle(N, 4.0, rule)
    got = plan.collide_vjp(f, u).double().cpu().numpy()
    plan.stream_status()
    for i in range(3):
        a, b = f[i].double().cpu().numpy(), u[i].double().cpu().numpy()
        scale = np.linalg.norm(b * O.collision._apply_multiplier(op, op.Gloss, a))
        assert np.linalg.norm(got[i] - O.vjp(op, a, b)) < TOL[prec] * scale


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("M,kind", [(6, None), (12, None), (26, None), (0, "generic"), (0, "planes"), (0, "no_x")])
@pytest.mark.parametrize("N,max_batch", [(8, 0), (12, 1)])
def test_vss_rules_against_oracle(prec, M, kind, N, max_batch):
    L, gamma, alpha = 4.0, 0.4, 1.5
    f, g = _fields(2, N, prec)
    if kind:
        rule = _rule(kind)
        kw = dict(sphere=rule)
        okw = dict(sphere=(np.concatenate([rule[:, :3], -rule[:, :3]]), np.concatenate([rule[:, 3], rule[:, 3]])))
    else:
        kw, okw = dict(M=M), dict(M=M)
    plan = binding.Plan(N=N, L=L, gamma=gamma, alpha=alpha, N_rho=N, precision=prec, max_batch=max_batch, **kw)
    vplan = V.VSSPlan(N, L, gamma=gamma, alpha=alpha, Nrho=N, nyquist="sym", **okw)
    q, q2 = plan.collide(f).double().cpu().numpy(), plan.collide2(f, g).double().cpu().numpy()
    j = plan.collide_jvp(f, g).double().cpu().numpy()
    plan.stream_status()
    for i in range(2):
        a, b = f[i].double().cpu().numpy(), g[i].double().cpu().numpy()
        loss = np.linalg.norm(a * np.real(vplan.idft3(vplan.Gloss * vplan.dft3(b))))
        qab, qba = V.fast_Q_vss(vplan, a, b), V.fast_Q_vss(vplan, b, a)
        assert np.linalg.norm(q[i] - V.fast_Q_vss(vplan, a)) < TOL[prec] * loss
        assert np.linalg.norm(q2[i] - qab) < TOL[prec] * loss
        assert np.linalg.norm(j[i] - (qab + qba)) < 2 * TOL[prec] * loss


@pytest.mark.parametrize("N,M", [(16, 12), (24, 26), (32, 38)])
@pytest.mark.parametrize("B", [1, 40])
def test_wide_and_narrow_launches_agree_with_fp64(N, M, B):
    """FP32 at the larger grids against FP64 plans (VSS at N = 32, which FP64 does not take: against one node at a time)."""
    L = {16: 5.0, 24: 6.0, 32: 7.0}[N]
    f = torch.from_numpy(W.two_maxwellian(B, N, L, 3)[0]).cuda()
    u = torch.from_numpy(W.directions(B, N, 4)).cuda()
    f32, u32 = f.float(), u.float()
    scale = lambda a, b: float(b.norm()) * float(a.abs().sum()) * (2 * L / N) ** 3   # ||u|| n bounds both loss terms
    kw = dict(N=N, L=L, gamma=0.4, M=M, N_rho=N)
    got = binding.Plan(precision="fp32", **kw).collide_vjp(f32, u32)
    p64 = binding.Plan(precision="fp64", **kw)
    for i in {0, B // 2, B - 1}:
        ref = p64.collide_vjp(f32[i:i + 1].double(), u32[i:i + 1].double())
        assert (got[i].double() - ref[0]).norm().item() < 1e-5 * scale(f[i], u[i])
    vss = binding.Plan(precision="fp32", alpha=1.4, **kw)
    q = vss.collide(f32)
    one = binding.Plan(precision="fp64", alpha=1.4, **kw) if N < 32 else vss
    for i in {0, B // 2, B - 1}:
        ref = one.collide(f32[i:i + 1].to(torch.float64 if N < 32 else torch.float32))
        assert (q[i].double() - ref[0].double()).norm().item() < 1e-5 * scale(f[i], f[i])
