"""The device-side checks of hfx_set_coulomb (GB300 only): a single bad element
anywhere in a matrix whose size is no multiple of the 32 x 32 tiles, deviations on
both sides of the tolerance, values in the row padding (ignored), and a refused
matrix leaving the accepted one in place."""
import numpy as np
import pytest

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


def _code(c, v, **kw):
    try:
        hfx.hfx_set_coulomb(c.ctx, 0, kw.pop("G"), v, **kw)
        return hfx.HFX_OK
    except hfx.HfxError as e:
        return e.code


@pytest.mark.parametrize("nipw", [0, 13, 14, 15, 47])
def test_bad_elements_are_found_and_refused(nipw):
    s = S.make_system(0, mesh=(1, 1, 1), nb=3, no=2, aux=("count", max(nipw, 1), max(nipw, 1)))
    n = s.n_mt + nipw
    v, G = np.ascontiguousarray(s.v[0][:n, :n]), s.Gaux[0][:nipw]
    with hfx.Context(s, precision="fp64") as c:
        c.load_system(coulomb=False)
        assert _code(c, v, G=G) == hfx.HFX_OK
        c.build_all()
        want = c.exchange(0)
        mx = max(np.abs(v.real).max(), np.abs(v.imag).max())
        for i, j in ((0, 0), (n - 1, 0), (0, n - 1), (n - 1, n - 1), (31, 32), (33, 2)):
            for bad in (np.nan, np.inf, -np.inf, 1j * np.inf):
                w = v.copy()
                w[i, j] = bad
                assert _code(c, w, G=G) == hfx.HFX_ENONFINITE
            w = v.copy()
            w[i, j] += 3e-10j * mx      # the tolerance is 1e-10 of the largest component
            assert _code(c, w, G=G) == hfx.HFX_ENOTHERM
        w = v.copy()
        w[n - 1, 3] += 0.5e-10 * mx     # within the tolerance
        assert _code(c, w, G=G) == hfx.HFX_OK
        pad = np.full((n, n + 3), np.nan + 0j)
        pad[:, :n] = v
        assert _code(c, pad, G=G, ld=n + 3) == hfx.HFX_OK
        w = v.copy()
        w[n - 1, n - 1] = np.nan
        assert _code(c, w, G=G) == hfx.HFX_ENONFINITE
        c.build_all()                   # the accepted matrix is still there
        assert np.array_equal(c.exchange(0), want)


def test_imaginary_parts_with_inversion():
    s = S.make_system(0, mesh=(1, 1, 1), nb=3, no=2, inversion=True)
    v = s.v[0]
    mx = np.abs(v.real).max()
    with hfx.Context(s) as c:
        c.load_system()
        for eps, code in ((0.4e-10, hfx.HFX_OK), (1.6e-10, hfx.HFX_EINVAL)):
            w = v.copy()
            w[3, 40] += 1j * eps * mx
            w[40, 3] -= 1j * eps * mx
            assert _code(c, w, G=s.Gaux[0]) == code
        c.build_all()
        assert np.abs(c.exchange(0).imag).max() == 0.0
