"""The functions M_aLP of the radial basis are orthonormal to the rounding of their sums
(GB300 only), also where the wanted eigenvalues of the overlap matrix spread over five
orders of magnitude: the eigenvectors alone leave overlaps of 4e-13 to 4e-12 there.

Tolerance: a sum over n points of products whose absolute values add up to at most one
carries at most n eps; the library's sums and the test's are taken, 2 n eps."""
import numpy as np
import pytest

from paper_1003_0524_gb300 import hfx
from paper_1003_0524_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lmax,Lmax,P,n_r,seed", [(8, 8, 4, 400, 0), (8, 8, 4, 400, 1), (8, 8, 4, 400, 3), (4, 4, 3, 600, 2),
                                                   (0, 0, 1, 40, 0)])
def test_functions_are_orthonormal(lmax, Lmax, P, n_r, seed):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1003_0524_gb300 import build
    build.build()
    r, w, u = S.radial_functions(lmax, 2.2, n_r, seed)
    ctx = hfx.hfx_create(np.eye(3) * 10.0, np.zeros((1, 3)), np.array([2.2]), lmax, Lmax, P, (1, 1, 1))
    try:
        hfx.hfx_set_radial_functions(ctx, 0, r, w, u, 1e-4)
        M = hfx.hfx_get_radial_basis(ctx, 0, n_r, lmax, Lmax, P)["M"].reshape(Lmax + 1, P, n_r)
    finally:
        hfx.hfx_destroy(ctx)
    for m in M:
        assert np.abs((m * w * r * r) @ m.T - np.eye(P)).max() <= 2 * n_r * np.finfo(float).eps


def test_large_working_memory_is_given_back():
    """8192 points of lmax 8 need 40 MB; after the next build they are free again, up to
    the 2 MB granules of an allocation."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    s = S.make_system(dict(S.CONFIGS[0], lmax=8), mesh=(1, 1, 1), nb=2, no=1)
    r, w, u = S.radial_functions(s.lmax, float(s.rmt[0]), 8192, 3)
    with hfx.Context(s, sparse="off") as c:
        c.load_system()
        c.build_all()
        free = torch.cuda.mem_get_info()[0]
        hfx.hfx_set_radial_functions(c.ctx, 0, r, w, u, 1e-4)
        c.build_all()
        assert free - torch.cuda.mem_get_info()[0] <= 8 << 20
