"""The interstitial kernel's cover of the plane-wave spheres (lines of 4 points or patches
of 2 by 2) against the oracle's projections (GB300 only): one plane wave, odd and even
numbers of lines, the full spheres, a box that is not a cube, several k per row tile and a
single one, band counts around the band blocks (chunks of 4 and of 8 segments) and
different for every k.  Tolerance: the 1e-8 of the largest projection that the sliced
operands are held to elsewhere; a point missed or taken twice shows at 1e-3."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1003_0524_gb300 import hfx
from paper_1003_0524_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg,gmax,mesh,nb,no,tile", [
    (1, 0.45, (2, 1, 1), 3, 1, 0),
    (1, 0.95, (2, 2, 1), 9, 2, 8),
    (1, 1.4, (1, 1, 1), 33, 3, 40),
    (1, 3.0, (2, 1, 2), 41, 5, 48),
    (2, 2.3, (2, 2, 2), ("U", 5, 23), ("U", 1, 4), 16),
    (3, 3.0, (1, 2, 1), 57, 2, 56),
    (4, 2.6, (2, 1, 1), 65, 3, 64),
])
def test_interstitial_projections(cfg, gmax, mesh, nb, no, tile):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1003_0524_gb300 import build
    build.build()
    s = S.make_system(dict(S.CONFIGS[cfg], gmax=gmax, lmax=1, Lmax=1), mesh=mesh, nb=nb, no=no, aux=("count", 51, 90), seed=17)
    o = O.Oracle(s)
    with hfx.Context(s, tile_nb_zipw=tile) as c:
        c.load_system()
        c.build_all(keep_products=True)
        for ik in range(s.n_k):
            for iq in range(s.n_k):
                ikp, _ = o.fold(ik, iq)
                z, want = c.products(ik, iq, ikp)[s.n_mt:], o.zipw(ik, iq)
                assert np.abs(z - want).max() <= 1e-8 * np.abs(want).max()
