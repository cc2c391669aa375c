"""Which kernels an F16X3 plan's calls take: the FP32 translates (the bits of an FP32 plan) where the sphere points share
shifts, the split-data tensor-core kernel (the bits of the allocation-free call, which always takes it) where it is the
more exact or the faster one."""
import numpy as np
import pytest
import torch

from paper_1809_10186_gb300 import binding, workloads as W

pytestmark = pytest.mark.gpu

L_OF = {16: 5.0, 24: 6.0, 32: 7.0}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1809_10186_gb300 import build
    build.build()


def _generic(P):
    """P pairs without a common component."""
    s = W.rng(5).normal(size=(P, 3))
    s /= np.linalg.norm(s, axis=1, keepdims=True)
    return np.concatenate([s, np.full((P, 1), 2 * np.pi / P)], axis=1)


@pytest.mark.parametrize("N,rule,split", [(16, 6, True), (32, 6, True), (32, "generic", True), (24, 6, False), (16, 12, False),
                                          (32, 26, False), (32, 38, False), (24, 38, False), (16, "generic", False),
                                          (24, "generic", False)])
def test_engine(N, rule, split):
    kw = dict(N=N, L=L_OF[N], gamma=0.4, N_rho=N, **(dict(sphere=_generic(17)) if rule == "generic" else dict(M=rule)))
    f = torch.from_numpy(W.two_maxwellian(2, N, L_OF[N], 3)[0]).cuda().float()
    plan = binding.Plan(precision="f16x3", **kw)
    ref = plan.collide_noalloc(f) if split else binding.Plan(precision="fp32", **kw).collide(f)
    assert torch.equal(plan.collide(f), ref)
    plan.stream_status()


@pytest.mark.parametrize("N", [16, 32])
def test_six_point_error(N):
    """Q of the six-point rule: no further from FP64 than 1.1 times the split-data kernel's own error."""
    kw = dict(N=N, L=L_OF[N], gamma=0.4, N_rho=N, M=6)
    f = torch.from_numpy(W.two_maxwellian(4, N, L_OF[N], 4)[0]).cuda().float()
    plan = binding.Plan(precision="f16x3", **kw)
    ref = binding.Plan(precision="fp64", **kw).collide(f.double())
    err = lambda q: (q.double() - ref).norm().item()
    assert err(plan.collide(f)) <= 1.1 * err(plan.collide_noalloc(f))


@pytest.mark.parametrize("rule,candidates", [(12, 3), (6, 15)])
def test_autotune_times_radial_points_only_where_they_count(rule, candidates):
    """Three chunk sizes; five choices of radial points per item where Q(f, f) runs the kernel that reads them, else the
    batch-size rule stays in force (per calls of this batch: two CTAs an item, 16 items per SM)."""
    N, B = 32, 40
    plan = binding.Plan(N=N, L=7.0, gamma=0.4, N_rho=N, M=rule, precision="f16x3", max_batch=B)
    f = torch.from_numpy(W.two_maxwellian(B, N, 7.0, 5)[0]).cuda().float()
    plan.set_tuning(8, 0)
    rep = plan.autotune(f)
    assert rep["cached"] == 0 and rep["candidates"] == candidates
    if rule == 12:
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        want = next((c for c in (4, 2) if 2 * (N // c) * rep["chunk_nodes"] >= 16 * sms), 1)
        assert rep["rpc"] == want
    again = binding.Plan(N=N, L=7.0, gamma=0.4, N_rho=N, M=rule, precision="f16x3", max_batch=B).autotune(f)
    assert again["cached"] == 1 and again["rpc"] == rep["rpc"]
