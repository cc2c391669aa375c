"""FP32 errors against FP64 plans on the same inputs, relative to ||Q|| over a batch of two-Maxwellian nodes, for every
grid and built-in sphere rule.

Limits: the errors that a transform of its own for every sphere pair gives on these inputs (measured, LIMIT, in units of
1e-8), times 1.1, about what they differ by between batches of this size. The shared translates must not be less exact.
"""
import pytest
import torch

from paper_1809_10186_gb300 import binding, workloads as W

pytestmark = pytest.mark.gpu

L_OF = {8: 3.5, 12: 4.0, 16: 5.0, 24: 6.0, 32: 7.0}
RULES = (6, 12, 26, 38)
LIMIT = {
    (8, "collide"): (264.2, 250.6, 215.2, 220.9),
    (8, "collide2"): (48.6, 46.7, 41.7, 42.5),
    (8, "jvp"): (167.1, 167.6, 145.7, 148.2),
    (8, "vjp"): (24.8, 36.3, 40.7, 41.1),
    (8, "vss collide"): (274.2, 225.5, 230.0, 191.9),
    (8, "vss jvp"): (180.9, 143.5, 166.0, 133.5),
    (12, "collide"): (350.9, 270.8, 272.2, 255.3),
    (12, "collide2"): (63.7, 52.2, 52.6, 50.6),
    (12, "jvp"): (222.3, 182.4, 181.8, 174.4),
    (12, "vjp"): (27.5, 32.1, 35.0, 32.8),
    (12, "vss collide"): (357.2, 269.3, 284.7, 309.5),
    (12, "vss jvp"): (216.0, 169.7, 195.7, 210.2),
    (16, "collide"): (369.5, 373.4, 404.7, 391.6),
    (16, "collide2"): (68.6, 70.6, 79.1, 75.9),
    (16, "jvp"): (242.4, 248.0, 278.1, 265.5),
    (16, "vjp"): (23.9, 27.0, 30.5, 28.4),
    (16, "vss collide"): (377.5, 383.6, 470.8, 369.0),
    (16, "vss jvp"): (251.3, 265.6, 340.1, 259.6),
    (24, "collide"): (383.2, 315.1, 305.6, 306.9),
    (24, "collide2"): (70.6, 64.9, 63.2, 64.2),
    (24, "jvp"): (236.7, 220.7, 210.8, 216.6),
    (24, "vjp"): (20.7, 21.4, 22.9, 23.2),
    (24, "vss collide"): (378.4, 272.0, 266.7, 280.8),
    (24, "vss jvp"): (232.7, 185.6, 180.4, 184.9),
    (32, "collide"): (828.8, 755.5, 728.1, 787.3),
    (32, "collide2"): (149.7, 144.0, 143.7, 154.3),
    (32, "jvp"): (544.2, 528.3, 527.8, 566.7),
    (32, "vjp"): (27.8, 26.6, 24.9, 25.3),
}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1809_10186_gb300 import build
    build.build()


def errors(N, op):
    """Relative error of one call for every rule."""
    f, g = (torch.from_numpy(W.two_maxwellian(32, N, L_OF[N], seed)[0]).cuda().float() for seed in (11, 12))
    call = {"collide": lambda p, a, b: p.collide(a), "collide2": lambda p, a, b: p.collide2(a, b),
            "jvp": lambda p, a, b: p.collide_jvp(a, b), "vjp": lambda p, a, b: p.collide_vjp(a, b)}[op.split()[-1]]
    out = []
    for M in RULES:
        kw = dict(N=N, L=L_OF[N], gamma=0.38, M=M, N_rho=N, alpha=1.4 if op.startswith("vss") else 0.0)
        p32, p64 = binding.Plan(precision="fp32", **kw), binding.Plan(precision="fp64", **kw)
        ref = call(p64, f.double(), g.double())
        out.append(((call(p32, f, g).double() - ref).norm() / ref.norm()).item())
        p32.close()
        p64.close()
    return out


@pytest.mark.parametrize("N,op", sorted(LIMIT))
def test_error_is_no_larger_than_with_a_transform_per_pair(N, op):
    got = errors(N, op)
    print(N, op, ["%.1f" % (1e8 * e) for e in got])
    for M, e, limit in zip(RULES, got, LIMIT[N, op]):
        assert e < 1.1e-8 * limit, (M, e)


@pytest.mark.parametrize("prec", ["fp32", "f16x3"])
@pytest.mark.parametrize("N,N_rho", [(8, 33), (16, 40), (24, 33), (32, 40)])
def test_more_radial_points_than_the_fused_stage_takes(prec, N, N_rho):
    """Ranks above 32 (N = 8, 16: the separate projection kernels): 1e-5 of the loss term, the FP32 tolerance."""
    if prec == "f16x3" and N == 8:
        pytest.skip("tensor-core precisions start at N = 16")
    kw = dict(N=N, L=L_OF[N], gamma=0.38, M=26, N_rho=N_rho)
    f, g = (torch.from_numpy(W.two_maxwellian(3, N, L_OF[N], seed)[0]).cuda().float() for seed in (11, 12))
    p32, p64 = binding.Plan(precision=prec, **kw), binding.Plan(precision="fp64", **kw)
    bound = 1e-5 * (f.double() * f.double().sum((1, 2, 3), keepdim=True) * (2 * L_OF[N] / N) ** 3).norm()   # b n f bounds the loss
    assert (p32.collide(f).double() - p64.collide(f.double())).norm() < bound
    assert (p32.collide2(f, g).double() - p64.collide2(f.double(), g.double())).norm() < bound
    plan = binding.Plan(precision=prec, **dict(kw, N_rho=N_rho, gamma=0.5))
    packed = binding.collide_ragged([plan], [0, 0, 0], [i * N ** 3 for i in range(3)], f.reshape(-1), node_gamma=[0.38] * 3,
                                    node_b=[p64.info["b"]] * 3)
    assert (packed.reshape(f.shape).double() - p64.collide(f.double())).norm() < bound


@pytest.mark.parametrize("rank", [1, 2, 3, 5])
@pytest.mark.parametrize("N", [8, 16, 32])
def test_low_ranks(N, rank):
    """A radial kernel of a few factors, which passes zero at some radial points: 1e-5 of the loss term."""
    kw = dict(N=N, L=L_OF[N], gamma=0.38, M=12, N_rho=N, svd_rank=rank)
    f, g = (torch.from_numpy(W.two_maxwellian(3, N, L_OF[N], seed)[0]).cuda().float() for seed in (11, 12))
    p32, p64 = binding.Plan(precision="fp32", **kw), binding.Plan(precision="fp64", **kw)
    bound = 1e-5 * (f.double() * f.double().sum((1, 2, 3), keepdim=True) * (2 * L_OF[N] / N) ** 3).norm()   # b n f bounds the loss
    assert (p32.collide(f).double() - p64.collide(f.double())).norm() < bound
    assert (p32.collide2(f, g).double() - p64.collide2(f.double(), g.double())).norm() < 1.5 * bound   # norms of f and g differ
