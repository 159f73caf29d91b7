"""The muffin-tin contraction at the edges of its sizes, against the oracle's
projections (GB300 only): angular cutoffs that differ, the largest one (coefficients in
several chunks), one radial function, band counts around the 32-band groups and
different for every k, the untransformed (dense) order.  Tolerance: FP64 sums of up to a
few hundred terms, 1e-12 of the largest projection."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1003_0524_gb300 import hfx
from paper_1003_0524_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lmax,Lmax,P,nb,sparse", [
    (0, 0, 1, 3, "off"),
    (1, 2, 2, 31, "auto"),
    (2, 5, 3, 33, "auto"),
    (6, 2, 5, ("U", 2, 9), "off"),
    (8, 3, 4, 4, "auto"),
    (8, 8, 2, 2, "off"),
])
def test_mt_projections(lmax, Lmax, P, nb, sparse):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1003_0524_gb300 import build
    build.build()
    s = S.make_system(dict(S.CONFIGS[1], lmax=lmax, Lmax=Lmax, P=P, sparse=sparse != "off"), mesh=(2, 1, 1), nb=nb, no=2,
                      aux=("count", 5, 9), seed=3 * lmax + P)
    o = O.Oracle(s)
    with hfx.Context(s, precision="fp64", sparse=sparse) as c:
        c.load_system()
        c.build_all(keep_products=True)
        for ik in range(2):
            for iq in range(2):
                ikp, _ = o.fold(ik, iq)
                z, want = c.products(ik, iq, ikp)[:s.n_mt], o.zmt(ik, iq)
                assert np.abs(z - want).max() <= 1e-12 * np.abs(want).max()
