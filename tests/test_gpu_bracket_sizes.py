"""The q->0 bracket over lattices and meshes whose lines and segments differ (GB300
only): skewed cells (lines that pass the origin off their middle), uneven meshes, a
mesh of one point, lines shorter and longer than one segment, a sphere that holds
nothing but the origin.

Tolerance: the sum holds up to ~10^7 terms and is subtracted from an integral of
order 10, so ~1e-16 * 10 * sqrt(10^7) ~ 3e-12 absolute; 5e-11 is taken.
"""
import math

import numpy as np
import pytest

from paper_1003_0524_gb300 import hfx
from paper_1003_0524_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


def reference(lattice, mesh, beta):
    q0 = math.sqrt(-math.log(beta) / beta)
    fine = S.reciprocal(lattice) / np.asarray(mesh, dtype=float)[:, None]
    n = [int(math.ceil(q0 * np.linalg.norm(lattice[i]) * mesh[i] / (2 * math.pi))) + 1 for i in range(3)]
    y, z = np.meshgrid(np.arange(-n[1], n[1] + 1), np.arange(-n[2], n[2] + 1), indexing="ij")
    yz = y.reshape(-1, 1) * fine[1] + z.reshape(-1, 1) * fine[2]
    tot = 0.0
    for x in range(-n[0], n[0] + 1):
        q2 = ((x * fine[0] + yz) ** 2).sum(1)
        q2 = q2[(q2 > 1e-18) & (q2 <= q0 * q0)]
        tot += (np.exp(-beta * q2) / q2).sum()
    om = abs(np.linalg.det(lattice))
    return math.erf(math.sqrt(beta) * q0) / math.sqrt(math.pi * beta) - 4 * math.pi / (np.prod(mesh) * om) * tot


SKEW = np.array([[7.0, 0.3, -0.2], [3.1, 6.0, 0.4], [-2.2, 2.9, 8.0]])


@pytest.mark.parametrize("lattice,mesh,beta", [
    (np.eye(3) * 8.0, (1, 1, 1), 0.005),
    (np.eye(3) * 10.3, (4, 4, 4), 0.005),
    (SKEW, (1, 1, 1), 0.005),
    (SKEW, (3, 1, 2), 0.005),
    (SKEW[[1, 2, 0]], (1, 2, 5), 0.02),
    (np.diag([2.0, 14.0, 3.0]), (2, 1, 1), 0.01),
    (np.diag([9.0, 3.0, 17.0]), (1, 1, 6), 0.05),
    (np.eye(3) * 4.0, (2, 2, 2), 0.9),
    (np.asarray(S.CONFIGS[4]["lattice"]), (2, 3, 1), 0.005),
])
def test_bracket_matches_the_direct_sum(lattice, mesh, beta):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1003_0524_gb300 import build
    build.build()
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    hfx.hfx_q0_bracket_noalloc(lattice, mesh, beta, out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert abs(float(out.cpu()[0]) - reference(lattice, mesh, beta)) <= 5e-11
