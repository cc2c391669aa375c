"""VSS calls of a few nodes, whose products are spread over more blocks: the bits of the same node in a large batch, for odd
and even numbers of products."""
import numpy as np
import pytest
import torch

from paper_1809_10186_gb300 import binding, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1809_10186_gb300 import build
    build.build()


def _pairs(P):
    s = W.rng(5).normal(size=(P, 3))
    s /= np.linalg.norm(s, axis=1, keepdims=True)
    return np.concatenate([s, np.full((P, 1), 2 * np.pi / P)], axis=1)


@pytest.mark.parametrize("prec,N,rule", [("fp64", 8, 26), ("fp64", 12, 6), ("fp64", 16, "odd"), ("fp32", 8, "one"), ("fp32", 16, 38),
                                         ("fp32", 24, 12), ("fp32", 32, 26)])
def test_one_node_equals_its_bits_in_a_batch(prec, N, rule):
    kw = dict(sphere=_pairs({"odd": 7, "one": 1}[rule])) if isinstance(rule, str) else dict(M=rule)
    plan = binding.Plan(N=N, L=5.0, gamma=0.4, alpha=1.4, N_rho=N, precision=prec, **kw)
    B = {8: 300, 12: 120, 16: 80, 24: 40, 32: 40}[N]
    f, g = (torch.from_numpy(W.two_maxwellian(B, N, 5.0, s)[0]).to("cuda", plan.dtype) for s in (3, 4))
    Q, J = plan.collide(f), plan.collide_jvp(f, g)
    for n in (1, 3):
        assert torch.equal(plan.collide(f[:n].contiguous()), Q[:n])
        assert torch.equal(plan.collide_jvp(f[:n].contiguous(), g[:n].contiguous()), J[:n])
