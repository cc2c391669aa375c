"""The shared-shift translate products of FP32/FP64 plans (k_shift.cu) against the FP64 oracle and the
dense circulant kernel: rules whose points share x and (x, y) shifts, rules that share none, points in the
coordinate planes, both CTA widths (few and many (node, radial point) items), several batches, and a
workspace that holds only a few radial points of one node.

Tolerances: 1e-10 (FP64) and 1e-5 (FP32) of the loss term, those of tests/test_gpu_parity.py; two FP32
evaluations that each keep theirs differ by at most 2e-5.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1809_10186_gb300 import binding, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1809_10186_gb300 import build
    build.build()


def _rule(kind):
    """[P, 4] pair representatives and weights (sum of weights 2 pi)."""
    if kind == "generic":       # no two points share a component
        s = W.rng(5).normal(size=(7, 3))
    elif kind == "planes":      # zero components on every axis, shared and opposite ones, x < 0 leads
        s = np.array([[0, 0, 1.0], [0, 1, 0], [-1, 0, 0], [0, 0.6, -0.8], [0, 0.6, 0.8], [-0.6, 0.8, 0], [-0.6, -0.8, 0],
                      [0.6, 0, 0.8], [0.6, 0, -0.8]])
    else:                       # no x shift at all
        s = np.array([[0, 0, 1.0], [0, 1, 0], [0, 0.8, 0.6]])
    s = s / np.linalg.norm(s, axis=1, keepdims=True)
    w = W.rng(6).uniform(0.5, 1.5, size=len(s))
    return np.concatenate([s, (2 * np.pi * w / w.sum())[:, None]], axis=1)


def _oracle(N, L, rule):
    sphere = (np.concatenate([rule[:, :3], -rule[:, :3]]), np.concatenate([rule[:, 3], rule[:, 3]]))
    return O.OraclePlan(N, L, gamma=0.4, Nrho=N, sphere=sphere, nyquist="sym")


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("fp32", 1e-5)])
@pytest.mark.parametrize("kind", ["generic", "planes", "no_x"])
@pytest.mark.parametrize("N,max_batch", [(8, 0), (12, 0), (12, 1)])
def test_rules_against_oracle(prec, tol, kind, N, max_batch):
    L, rule = 4.0, _rule(kind)
    dt = torch.float64 if prec == "fp64" else torch.float32
    f, g = (torch.from_numpy(W.rough(3, N, seed)).to("cuda", dt) for seed in (1, 2))
    plan = binding.Plan(N=N, L=L, gamma=0.4, sphere=rule, N_rho=N, precision=prec, max_batch=max_batch)
    op = _oracle(N, L, rule)
    q, q2 = plan.collide(f).double().cpu().numpy(), plan.collide2(f, g).double().cpu().numpy()
    for i in range(3):
        a, b = f[i].double().cpu().numpy(), g[i].double().cpu().numpy()
        for got, x in ((q[i], a), (q2[i], b)):
            loss = np.linalg.norm(np.real(O.loss_Q(op, a, x)))
            assert np.linalg.norm(got - O.fast_Q(op, a, x)) < tol * loss


@pytest.mark.parametrize("N,M", [(8, 26), (12, 12), (16, 6), (24, 12), (32, 38)])
@pytest.mark.parametrize("items", [1, 700])
def test_widths_against_dense_kernel(N, M, items):
    """One node (two planes per CTA) and enough nodes for the wide CTAs, in batches of one and many."""
    L = {8: 3.5, 12: 4.0, 16: 5.0, 24: 6.0, 32: 7.0}[N]
    plan = binding.Plan(N=N, L=L, gamma=0.4, M=M, N_rho=N, precision="fp32", max_batch=300)
    B = max(1, items // N)
    f = torch.from_numpy(W.two_maxwellian(B, N, L, 3)[0]).to("cuda", torch.float32)
    q = plan.collide(f)
    if N == 12:   # the dense kernel does not take N = 12: an FP64 plan, whose products the oracle checks above
        plan64 = binding.Plan(N=N, L=L, gamma=0.4, M=M, N_rho=N, precision="fp64")
        ref = torch.cat([plan64.collide(x.contiguous()) for x in f.double().split(3)])
    else:
        ref = torch.cat([plan.collide_noalloc(x.contiguous()) for x in f.split(3)])
    fh = np.fft.fftn(f[0].double().cpu().numpy())
    loss = float(f[0].double().norm()) * float(abs(fh[0, 0, 0])) * (2 * L / N) ** 3   # ||f|| n: below 4 pi b R^gamma n ||f||
    plan.stream_status()
    err = (q.double() - ref.double()).flatten(1).norm(dim=1).max().item()
    assert err < 2e-5 * loss, (err, loss)
    one = plan.collide(f[-1:].contiguous())
    assert (one.double() - q[-1:].double()).norm().item() < 2e-5 * loss
