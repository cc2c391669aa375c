"""The split-data tensor-core kernel in fp16 (F16X3: the allocation-free call, dQ/dgamma and SSP-RK), with and without pairs
that share their x and z filters, against FP64 plans.

Tolerances: 1e-5 of the loss term, the F16X3 tolerance of tests/test_gpu_parity.py; times max |ln c_r| for dQ/dgamma, whose
radial terms carry that factor; for a step, dt times that of each of its three evaluations and four FP32 roundings of f.
"""
import numpy as np
import pytest
import torch

from paper_1809_10186_gb300 import binding, workloads as W

pytestmark = pytest.mark.gpu

L_OF = {16: 5.0, 24: 6.0, 32: 7.0}
GAMMA = 0.4
# a single pair; a group of two (equal s_x, s_z); two groups and a pair between them
RULES = {"one": [(0.36, 0.48, 0.8)], "group": [(0.36, 0.48, 0.8), (0.36, -0.48, 0.8)],
         "mixed": [(0.36, 0.48, 0.8), (0.36, -0.48, 0.8), (0.8, 0.0, 0.6), (0.6, 0.64, 0.48), (0.6, -0.64, 0.48)]}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1809_10186_gb300 import build
    build.build()


def _kw(N, rule):
    kw = dict(N=N, L=L_OF[N], gamma=GAMMA, N_rho=N)
    if isinstance(rule, int):
        return dict(kw, M=rule)
    s = np.asarray(RULES[rule])
    return dict(kw, sphere=np.concatenate([s, np.full((len(s), 1), 2 * np.pi / len(s))], axis=1))


def _loss(N, b, f):
    """The loss term f K_L f in FP64, and max |ln c_r|."""
    c, w = binding.host_quadrature(N=N, L=L_OF[N], M=6, N_rho=N)[:2]
    k = np.fft.fftfreq(N, 1.0 / N)
    kabs = np.sqrt(k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None] ** 2)
    G = sum(4 * np.pi * wr * 4 * np.pi * b * cr ** (GAMMA + 2) * np.sinc(cr * kabs / L_OF[N]) for cr, wr in zip(c, w))
    f = f.double().cpu().numpy()
    return np.linalg.norm(f * np.fft.ifftn(G * np.fft.fftn(f, axes=(1, 2, 3)), axes=(1, 2, 3)).real), np.abs(np.log(c)).max()


@pytest.mark.parametrize("N,rule", [(16, 38), (16, "mixed"), (24, 6), (24, 26), (24, 38), (24, "one"), (24, "group"), (32, 6),
                                    (32, 26), (32, 38), (32, "one"), (32, "group"), (32, "mixed")])
def test_against_fp64(N, rule):
    kw = _kw(N, rule)
    f = torch.from_numpy(W.two_maxwellian(3, N, L_OF[N], 21)[0]).cuda().float()
    plan, ref = binding.Plan(precision="f16x3", **kw), binding.Plan(precision="fp64", **kw)
    loss, ln = _loss(N, ref.info["b"], f)
    assert (plan.collide_noalloc(f).double() - ref.collide(f.double())).norm().item() < 1e-5 * loss
    assert (plan.collide_dgamma(f).double() - ref.collide_dgamma(f.double())).norm().item() < 1e-5 * ln * loss
    dt = 0.02
    got, want = plan.ssprk(f.clone(), dt, 1, order=3), ref.ssprk(f.double(), dt, 1, order=3)
    plan.stream_status()
    assert (got.double() - want).norm().item() < 3 * dt * 1e-5 * loss + 4 * 2.0 ** -24 * f.norm().item()


@pytest.mark.parametrize("N,rule", [(16, 26), (24, 38), (24, "mixed"), (32, 38), (32, "group"), (32, "one")])
def test_radial_points_per_item_do_not_change_bits(N, rule):
    f = torch.from_numpy(W.two_maxwellian(3, N, L_OF[N], 22)[0]).cuda().float()
    plan = binding.Plan(precision="f16x3", **_kw(N, rule))
    out = []
    for rpc in (1, 2, 4):
        plan.set_tuning(rpc, 0)
        out.append((plan.collide_dgamma(f), plan.collide_noalloc(f), plan.ssprk(f.clone(), 0.02, 1, order=2)))
    plan.stream_status()
    for o in out[1:]:
        assert all(torch.equal(a, b) for a, b in zip(o, out[0]))
