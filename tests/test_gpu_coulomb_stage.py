"""hfx_set_coulomb above and below the size where its checks move to the device, and the
memory it takes (GB300 only): matrices on both sides of 144 functions and of the 32 x 32
tiles, a first v, one that replaces it before and after a build (checked in a build buffer,
in the place of the slices of U, or in memory of its own), one of another size; what is refused leaves the old one in place.  A
call keeps no device memory besides v itself, up to the 2 MB granules of an allocation."""
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


def _code(c, G, v, **kw):
    try:
        hfx.hfx_set_coulomb(c.ctx, 0, G, v, **kw)
        return hfx.HFX_OK
    except hfx.HfxError as e:
        return e.code


@pytest.mark.parametrize("n,nb,precision", [(144, 2, "fp64"), (145, 2, "fp64"), (160, 2, "sliced"), (161, 100, "fp64"),
                                            (257, 2, "sliced")])
def test_refused_and_replaced(n, nb, precision):
    s = S.make_system(0, mesh=(1, 1, 1), nb=nb, no=min(nb, 4), aux=("count", n, n))
    N, m = s.n_mt, n - s.n_mt
    G, v = s.Gaux[0][:m], np.ascontiguousarray(s.v[0][:n, :n])
    w = np.ascontiguousarray(1.5 * s.v[0][:n, :n])

    def result(v, G):
        with hfx.Context(s, precision=precision) as c:
            c.load_system(coulomb=False)
            assert _code(c, G, v) == hfx.HFX_OK
            c.build_all()
            return c.exchange(0)

    want_v, want_w = result(v, G), result(w, G)
    mx = max(np.abs(v.real).max(), np.abs(v.imag).max())
    with hfx.Context(s, precision=precision) as c:
        c.load_system(coulomb=False)

        def refuse():
            for i, j in ((0, 0), (n - 1, 0), (0, n - 1), (n - 1, n - 1), (31, 32), (n - 1, n - 2)):
                for bad, code in ((np.nan, hfx.HFX_ENONFINITE), (-1j * np.inf, hfx.HFX_ENONFINITE),
                                  (v[i, j] + 3e-10j * mx, hfx.HFX_ENOTHERM)):
                    x = v.copy()
                    x[i, j] = bad
                    assert _code(c, G, x) == code

        refuse()                                   # a first v that is refused
        with pytest.raises(hfx.HfxError) as e:
            c.build_all()
        assert e.value.code == hfx.HFX_EMISSING
        pad = np.full((n, n + 5), np.nan + 0j)
        pad[:, :n] = w
        assert _code(c, G, pad, ld=n + 5) == hfx.HFX_OK
        refuse()
        assert _code(c, G, v) == hfx.HFX_OK        # replaced before the build
        c.build_all()
        assert np.array_equal(c.exchange(0), want_v)
        refuse()
        c.build_all()
        assert np.array_equal(c.exchange(0), want_v)
        assert _code(c, G, pad, ld=n + 5) == hfx.HFX_OK
        c.build_all()
        assert np.array_equal(c.exchange(0), want_w)
        k = N + 1 if n > 144 else n + 40           # another size, across the limit
        x = np.ascontiguousarray(s.v[0][:k, :k])
        assert _code(c, s.Gaux[0][:k - N], x) == hfx.HFX_OK
        c.build_all()
        assert np.array_equal(c.exchange(0), result(x, s.Gaux[0][:k - N]))


def test_no_memory_is_kept():
    import torch
    s = S.make_system(dict(S.CONFIGS[1], P=1, sparse=False), mesh=(1, 1, 1), nb=2, no=1, aux=("count", 9, 9))
    n = 1800
    G, _ = S._g_count(S.kpoint_frac(s.mesh, 0), s.lattice, n - s.n_mt)
    v = np.diag(1.0 + np.arange(n)).astype(np.complex128)
    free = lambda: torch.cuda.mem_get_info()[0]  # noqa: E731
    with hfx.Context(s, sparse="off", precision="fp64") as c:
        c.load_system(coulomb=False)
        f0 = free()
        hfx.hfx_set_coulomb(c.ctx, 0, G, v)
        assert f0 - free() <= v.nbytes + (8 << 20)
        c.build_all()
        f1 = free()
        hfx.hfx_set_coulomb(c.ctx, 0, G, v)        # two columns: no build buffer holds a v
        c.build_all()
        assert f1 - free() <= 8 << 20
