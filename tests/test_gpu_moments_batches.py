"""Moments of small and large batches: a node's bits do not depend on the batch, and a large batch of small grids costs no
more per point than one of large grids, up to the per-node work."""
import pytest
import torch

from paper_1809_10186_gb300 import binding, workloads as W

pytestmark = pytest.mark.gpu

L_OF = {8: 3.5, 12: 4.0, 16: 5.0, 24: 6.0, 32: 7.0}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1809_10186_gb300 import build
    build.build()


@pytest.mark.parametrize("N,batches", [(8, (1, 40, 1300)), (12, (1, 500, 700, 1300)), (16, (1, 40, 400, 700, 1300)),
                                       (24, (1, 160, 310, 610)), (32, (1, 160, 310))])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_bits_do_not_depend_on_the_batch(prec, N, batches):
    plan = binding.Plan(N=N, L=L_OF[N], gamma=0.4, M=6, N_rho=8, precision=prec, max_batch=1)
    f = torch.from_numpy(W.two_maxwellian(3, N, L_OF[N], 3)[0]).to("cuda", plan.dtype)
    ref = torch.cat([plan.moments(f[i:i + 1].contiguous()) for i in range(3)])
    n = (f.double().sum((1, 2, 3)) * (2 * L_OF[N] / N) ** 3)
    assert torch.allclose(ref[:, 0], n, rtol=1e-13)      # a sum of up to 32768 terms in FP64
    for B in batches:
        idx = torch.arange(B, device="cuda") % 3
        assert torch.equal(plan.moments(f[idx].contiguous()), ref[idx])


def test_small_grids_cost_no_more_per_point():
    """2 Mi points as 4096 nodes of N = 8 and as 64 of N = 32: at most 3 times the time (a 512-point node has one reduction
    for every 2 points of a thread, a 32768-point node one for 16 and more; measured 1.5 with one CTA per small node)."""
    def best(N, B):
        plan = binding.Plan(N=N, L=L_OF[N], gamma=0.4, M=6, N_rho=8, precision="fp32", max_batch=1)
        f = torch.from_numpy(W.two_maxwellian(2, N, L_OF[N], 3)[0]).cuda().float().repeat(B // 2, 1, 1, 1)
        times = []
        for _ in range(6):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(4):
                plan.moments(f)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)
    assert best(8, 4096) < 3.0 * best(32, 64)
