"""The FP64 contraction and LAPW transform at the edges of their tiles (GB300 only):
band counts on both sides of the tile edges 16, 24, 32 and 40, one band and one
occupied band (a split with empty parts), a dense v (no mu = 0 rows), channels with
one, two and four functions, and the Hermitian mirror of V_GG' across tiles.

Tolerances are those of the FP64 build against the oracle (1e-10 relative).
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1003_0524_gb300 import hfx
from paper_1003_0524_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1003_0524_gb300 import build
    build.build()
    hfx.load()


@pytest.mark.parametrize("cfg,mesh,nb,no,P,sparse", [
    (0, (2, 1, 1), 1, 1, 2, "auto"),
    (0, (2, 2, 1), 17, 3, 2, "off"),
    (0, (1, 1, 2), 33, 33, 2, "auto"),
    (1, (2, 1, 1), 24, 5, 1, "auto"),
    (1, (2, 1, 1), 25, 2, 4, "on"),
    (1, (1, 1, 1), 41, 7, 3, "on"),
    (1, (1, 1, 1), 41, 7, 3, "off"),
])
def test_fp64_build_at_tile_edges(cfg, mesh, nb, no, P, sparse):
    s = S.make_system(dict(S.CONFIGS[cfg], P=P, sparse=sparse == "on" or cfg == 1), mesh=mesh, nb=nb, no=no,
                      aux=("count", 61, 83), seed=40 + nb)
    ref = O.Oracle(s)
    with hfx.Context(s, precision="fp64", sparse=sparse) as c:
        c.load_system()
        c.build_all()
        for ik in range(s.n_k):
            want = ref.vx(ik)
            assert np.abs(c.exchange(ik) - want).max() <= 1e-10 * np.abs(want).max()


@pytest.mark.parametrize("nb", [3, 40])
def test_lapw_transform_is_hermitian_and_matches(nb):
    s = S.make_system(0, mesh=(2, 1, 1), nb=nb, no=3, seed=9)
    with hfx.Context(s, precision="fp64") as c:
        c.load_system()
        c.build_all()
        for ik in range(s.n_k):
            hfx.hfx_set_overlap(c.ctx, ik, S.overlap(s, ik))
        hfx.hfx_lapw_transform_all(c.ctx)
        for ik in range(s.n_k):
            got = hfx.hfx_get_lapw_exchange(c.ctx, ik, s.Gk[ik].shape[0])
            want = O.lapw_trafo(S.overlap(s, ik), s.c[ik], c.exchange(ik))
            assert np.abs(got - want).max() <= 1e-10 * np.abs(want).max()
