"""The Coulomb apply on residues (dense blocks of 1280 functions and more), against the
FP64 build (GB300 only): dense blocks at the edges of the 256-row tiles, the 128- and
64-value K chunks and the rule itself, one column, column counts that leave a tile or a
32-column store ragged, q of different size in one batch, several batches, no mu = 0
rows (dense mode), columns whose muffin-tin part is hundreds of times the interstitial
one, and small and large magnitudes.

Tolerance: operands are rounded to 0.3 units where their components have ~2^29 units,
and V^x is further limited by the FP32 pairs of Z^H Y, about 1e-9 relative at these
sizes; 5e-9 of the largest element is taken.  Builds that keep their projections slice
them from Z instead of the interstitial plane: the same bits.
"""
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


def _compare(s, sparse="auto", work_bytes=0, batches=None):
    with hfx.Context(s, precision="fp64", sparse=sparse) as c:
        c.load_system()
        c.build_all()
        want = [c.exchange(ik) for ik in range(s.n_k)]
    with hfx.Context(s, sparse=sparse, work_bytes=work_bytes) as c:
        c.load_system()
        st = c.build_all()
        if batches:
            assert st["n_batches"] >= batches
        got = [c.exchange(ik) for ik in range(s.n_k)]
        c.build_all(keep_products=True)
        kept = [c.exchange(ik) for ik in range(s.n_k)]
        for _ in range(2):   # captured, replayed
            c.build_all()
        again = [c.exchange(ik) for ik in range(s.n_k)]
    for a, b, k, r in zip(got, want, kept, again):
        assert np.abs(a - b).max() <= 5e-9 * np.abs(b).max()
        assert np.array_equal(a, k) and np.array_equal(a, r)


# 5 atoms, L <= 4: 125 channels, so the dense block has 125 + aux functions
@pytest.mark.parametrize("aux,mesh,nb,no", [
    ((1155, 1155), (1, 1, 1), 1, 1),       # 1280: the first size; one column
    ((1156, 1156), (1, 1, 1), 33, 1),      # 1281: a row tile of one function
    ((1218, 1220), (1, 1, 2), 7, 5),       # 1343 to 1345 around 1344 = 21 x 64
    ((1283, 1283), (1, 1, 1), 13, 20),     # 1408 = 11 x 128, 260 columns
    ((1411, 1411), (1, 1, 1), 9, 3),       # 1536 = 6 x 256
    ((1000, 1412), (2, 1, 2), 5, 3),       # very different q in one batch
])
def test_residue_apply_matches_fp64(aux, mesh, nb, no):
    _compare(S.make_system(dict(S.CONFIGS[3], aux=("count", *aux)), mesh=mesh, nb=nb, no=no, seed=60 + nb))


def test_residue_apply_dense_mode():
    s = S.make_system(dict(S.CONFIGS[3], P=1, sparse=False), mesh=(1, 1, 1), nb=6, no=4, aux=("count", 1200, 1200), seed=8)
    _compare(s, sparse="off")


def test_residue_apply_in_several_batches():
    s = S.make_system(dict(S.CONFIGS[3]), mesh=(2, 1, 2), nb=10, no=6, aux=("count", 1160, 1200), seed=9)
    _compare(s, work_bytes=90 << 20, batches=2)


@pytest.mark.parametrize("a_scale,fac", [(1.0, 1.0), (0.17, 1e-5), (0.17, 1e4)])
def test_residue_apply_over_magnitudes(a_scale, fac):
    s = S.make_system(dict(S.CONFIGS[3], a_scale=a_scale), mesh=(1, 1, 1), nb=8, no=5, aux=("count", 1180, 1180), seed=10)
    s.c = [x * fac for x in s.c]
    s.A = [x * fac for x in s.A]
    with hfx.Context(s, precision="fp64", q0_term=False) as c:
        c.load_system()
        c.build_all()
        want = c.exchange(0)
    with hfx.Context(s, q0_term=False) as c:
        c.load_system()
        c.build_all()
        got = c.exchange(0)
    assert np.abs(got - want).max() <= 5e-9 * np.abs(want).max()
