"""The FP64 build with a v(q) that is Hermitian only within herm_tol (GB300 only): V^x is
Z^H v Z for the v that was given, both triangles of it, as the defining sum has it, with
the build's own projections.  v (1 + i eps) keeps every pattern of v and differs by 2 eps
between its triangles; so does a matrix with noise where no pattern is asked for.  The
LAPW transform of such a V^x is not mirrored either.

Tolerance: FP64 sums of some hundred terms, 1e-13 of the largest element (the asymmetry
is 6e-11 of it); through the LAPW transform 1e-12."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1003_0524_gb300 import hfx
from paper_1003_0524_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg,P,sparse,inv", [(0, 2, "off", False), (1, 3, "on", False), (1, 1, "auto", False), (1, 3, "on", True)])
def test_both_triangles_count(cfg, P, sparse, inv):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1003_0524_gb300 import build
    build.build()
    spec = dict(S.CONFIGS[cfg], P=P, sparse=sparse != "off", aux=("count", 61, 83))
    s = S.make_system(spec, mesh=(2, 1, 1), nb=18, no=3, seed=31, inversion=inv)
    rng = np.random.Generator(np.random.PCG64(3))
    if inv:     # real, with antisymmetric noise of 3e-11 of each element
        s.v = [x * (1.0 + 3e-11 * np.triu(np.ones(x.shape), 1) - 3e-11 * np.tril(np.ones(x.shape), -1)) for x in s.v]
    elif sparse == "off":
        s.v = [x + 3e-11 * np.abs(x).max() * rng.uniform(-0.7, 0.7, x.shape) for x in s.v]
    else:
        s.v = [x * (1.0 + 3e-11j) for x in s.v]
    with hfx.Context(s, precision="fp64", sparse=sparse, q0_term=False) as c:
        c.load_system()
        st = c.build_all(keep_products=not inv)
        assert st["sparse_used"] == (1 if sparse == "on" else 0)
        got = [c.exchange(ik) for ik in range(s.n_k)]
        if inv:
            # the symmetric part of V^x is that of the symmetric part of v
            got = [0.5 * (x + x.T) for x in got]
            for x in s.v:
                x[:] = 0.5 * (x + x.T)
            for iq in range(s.n_k):
                hfx.hfx_set_coulomb(c.ctx, iq, s.Gaux[iq], s.v[iq])
            c.build_all()
            want = [c.exchange(ik) for ik in range(s.n_k)]
        else:
            want = []
            for ik in range(s.n_k):
                w = 0.0
                for iq in range(s.n_k):
                    z = c.products(ik, iq, (ik + iq) % 2)
                    w = w - np.einsum("Imn,IJ,Jmp->np", z.conj(), s.v[iq], z, optimize=True) / s.n_k
                want.append(w)
                hfx.hfx_set_overlap(c.ctx, ik, S.overlap(s, ik))
        for a, b in zip(got, want):
            assert np.abs(a - b).max() <= 1e-13 * np.abs(b).max()
        if not inv:
            hfx.hfx_lapw_transform_all(c.ctx)
            for ik in range(s.n_k):
                t = hfx.hfx_get_lapw_exchange(c.ctx, ik, s.Gk[ik].shape[0])
                ref = O.lapw_trafo(S.overlap(s, ik), s.c[ik], want[ik])
                assert np.abs(t - ref).max() <= 1e-12 * np.abs(ref).max()
