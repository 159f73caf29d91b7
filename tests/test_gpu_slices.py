"""The slicing of the projections from the interstitial kernel's plane against the
slicing of projections kept in FP64 (GB300 only): a build that keeps its products goes
through the transposed copy and the column-wise kernel, one that does not through the
fused kernel.  Both cut the same numbers, so V^x is the same to the last bit: column
counts that are no multiple of the 8-column blocks, one plane wave, no mu = 0 rows,
several band windows, a chunk boundary inside the muffin-tin rows."""
import numpy as np
import pytest

from paper_1003_0524_gb300 import hfx
from paper_1003_0524_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg,mesh,nb,no,aux,sparse,P", [
    (0, (2, 1, 1), 1, 1, (1, 1), "auto", 2),
    (0, (2, 2, 1), 7, 3, (20, 33), "off", 2),
    (0, (1, 1, 1), 9, 9, (64, 64), "auto", 1),
    (1, (2, 1, 1), 11, 5, (120, 140), "auto", 3),
    (2, (2, 2, 1), ("U", 3, 13), ("U", 1, 3), (90, 130), "auto", 3),
    (4, (1, 1, 2), 5, 3, (300, 301), "auto", 2),
])
def test_both_slicing_paths_give_the_same_bits(cfg, mesh, nb, no, aux, sparse, P):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1003_0524_gb300 import build
    build.build()
    s = S.make_system(dict(S.CONFIGS[cfg], P=P, sparse=sparse != "off"), mesh=mesh, nb=nb, no=no, aux=("count", *aux), seed=77)
    with hfx.Context(s, sparse=sparse) as c:
        c.load_system()
        c.build_all(keep_products=True)
        want = [c.exchange(ik) for ik in range(s.n_k)]
        for _ in range(3):   # direct, captured, replayed
            c.build_all()
            for ik in range(s.n_k):
                assert np.array_equal(c.exchange(ik), want[ik])
