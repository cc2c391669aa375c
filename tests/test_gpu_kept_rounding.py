"""dgfs_ssprk and dgfs_collide_dgamma of FP32 plans keep their rounding: checksums of the results' bits on fields made with
+, *, / alone (the same on every machine). A compiler that contracts other products in one of the kernels shows here."""
import zlib

import numpy as np
import pytest
import torch

from paper_1809_10186_gb300 import binding

pytestmark = pytest.mark.gpu

CRC = {(8, 6): (971597702, 1506348899), (12, 12): (3829420774, 3124352094),
       (16, 26): (2426323868, 214965850), (24, 12): (3506494628, 710126396),
       (32, 38): (559352672, 2353050415)}


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1809_10186_gb300 import build
    build.build()


def results(N, M):
    x = (np.arange(N) + 0.5) / N * 8.0 - 4.0
    u = np.array([0.25, -0.5, 1.0])[:, None]
    e = 1.0 / ((1.0 + (x - u) ** 2) * (1.0 + (x - u) ** 2) * (1.0 + 0.25 * x * x))
    f = torch.from_numpy((e[:, :, None, None] * e[:, None, :, None] * e[:, None, None, :]).astype(np.float32)).cuda()
    plan = binding.Plan(N=N, L=4.0, gamma=0.5, b=0.125, M=M, N_rho=8, precision="fp32")
    dq = plan.collide_dgamma(f)
    stepped = plan.ssprk(f.clone(), 2.0 ** -6, 2, order=3)
    return tuple(zlib.crc32(t.cpu().numpy().tobytes()) for t in (dq, stepped))


@pytest.mark.parametrize("N,M", sorted(CRC))
def test_bits(N, M):
    assert results(N, M) == CRC[N, M]
