"""A caller's projections in the sliced builds (GB300 only), where the interstitial rows
are sliced from Z instead of the interstitial kernel's plane: on the digit and on the
residue apply, for every pair of a batch when one of them is given.

Projections handed back as they were computed change nothing: without a multipole
transform (P = 1) they are the same numbers, and the digits the same to the last bit.  The
residues take a column's norm from sums in another order, so that its power of two may
differ by one, i.e. the operands' last bit, 2^-31 of a column's largest element: 1e-9.
Given random ones, the sliced build is within 5e-9 of the FP64 build, as with its own."""
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


def _ikp(s, ik, iq):
    m = np.array(s.mesh)
    j = lambda i: np.array([i // (m[1] * m[2]), (i // m[2]) % m[1], i % m[2]])  # noqa: E731
    return S.kpoint_index(s.mesh, (j(ik) - j(iq)) % m)


@pytest.mark.parametrize("cfg,mesh,nb,no,aux", [
    (0, (1, 1, 1), 1, 1, (1, 1)),
    (0, (2, 1, 1), 7, 3, (39, 64)),
    (1, (2, 2, 1), 11, 5, (120, 143)),
    (3, (2, 1, 1), 7, 3, (1560, 1590)),      # 125 muffin-tin functions: residues
    (3, (1, 1, 1), 13, 20, (1667, 1667)),
])
def test_own_projections_change_nothing(cfg, mesh, nb, no, aux):
    s = S.make_system(dict(S.CONFIGS[cfg], P=1, sparse=False), mesh=mesh, nb=nb, no=no, aux=("count", *aux), seed=21)
    with hfx.Context(s, sparse="off") as c:
        c.load_system()
        c.build_all(keep_products=True)
        want = [c.exchange(ik) for ik in range(s.n_k)]
        iq = s.n_k - 1
        c.set_products(0, iq, c.products(0, iq, _ikp(s, 0, iq)))
        for _ in range(3):   # direct, captured, replayed
            c.build_all()
            for ik in range(s.n_k):
                got = c.exchange(ik)
                if cfg == 3:
                    assert np.abs(got - want[ik]).max() <= 1e-9 * np.abs(want[ik]).max()
                else:
                    assert np.array_equal(got, want[ik])


@pytest.mark.parametrize("cfg,mesh,nb,no,aux,P", [
    (1, (2, 1, 1), 9, 4, (130, 150), 3),
    (3, (2, 1, 1), 6, 3, (1560, 1600), 3),
    (3, (1, 1, 2), 33, 2, (1611, 1611), 2),
])
def test_given_projections_match_fp64(cfg, mesh, nb, no, aux, P):
    s = S.make_system(dict(S.CONFIGS[cfg], P=P), mesh=mesh, nb=nb, no=no, aux=("count", *aux), seed=22)
    rng = np.random.Generator(np.random.PCG64(5))
    given = {}
    for ik, iq in ((0, 1), (1, 1), (1, 0)):
        shape = (s.n_aux(iq), int(s.n_occ[_ikp(s, ik, iq)]), int(s.n_bands[ik]))
        given[ik, iq] = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    out = []
    for precision in ("fp64", "sliced"):
        with hfx.Context(s, precision=precision, q0_term=False) as c:
            c.load_system()
            for (ik, iq), z in given.items():
                c.set_products(ik, iq, z)
            c.build_all()
            out.append([c.exchange(ik) for ik in range(s.n_k)])
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= 5e-9 * np.abs(a).max()
