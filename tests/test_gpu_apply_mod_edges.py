"""The Coulomb apply on residues where it takes over from the digits (1664 dense functions,
GB300 only), against the FP64 build: dense blocks at the edges of the 256-row tiles and of
the 128- and 64-value K chunks, one column, columns that leave a tile or a 32-column store
ragged, q of very different size in one batch, several batches, no mu = 0 rows, small and
large magnitudes.  Replays and builds that keep their projections give the same bits.

Tolerance: the operands are exact to 2^-31 of a line's largest element and V^x is limited
by the digits and FP32 pairs of Z^H Y, about 1e-9 relative: 5e-9 of the largest element."""
import numpy as np
import pytest

from paper_1003_0524_gb300 import hfx
from paper_1003_0524_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


# 5 atoms, L <= 4: 125 channels, so the dense block has 125 + aux functions
@pytest.mark.parametrize("aux,mesh,nb,no,kw", [
    ((1539, 1539), (1, 1, 1), 1, 1, {}),          # 1664: the first size; one column
    ((1540, 1540), (1, 1, 1), 33, 1, {}),         # 1665: a row tile with one K chunk more
    ((1602, 1604), (1, 1, 2), 7, 5, {}),          # 1727 to 1729 around 1728 = 27 x 64
    ((1667, 1667), (1, 1, 1), 13, 20, {}),        # 1792 = 7 x 256, 260 columns
    ((1668, 1668), (1, 1, 1), 9, 3, {}),          # 1793: a row tile of one function
    ((1100, 1800), (2, 1, 2), 5, 3, {}),          # q of very different size in one batch
    ((1560, 1600), (2, 1, 2), 10, 6, {"work_bytes": 100 << 20}),
    ((1560, 1560), (1, 1, 1), 6, 4, {"P": 1, "sparse": "off"}),
    ((1560, 1560), (1, 1, 1), 8, 5, {"fac": 1e-5}),
    ((1560, 1560), (1, 1, 1), 8, 5, {"fac": 1e4}),
])
def test_residue_apply_matches_fp64(aux, mesh, nb, no, kw):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1003_0524_gb300 import build
    build.build()
    sparse, P = kw.get("sparse", "auto"), kw.get("P", 3)
    s = S.make_system(dict(S.CONFIGS[3], aux=("count", *aux), P=P, sparse=sparse != "off"), mesh=mesh, nb=nb, no=no, seed=60 + nb)
    s.c, s.A = [x * kw.get("fac", 1.0) for x in s.c], [x * kw.get("fac", 1.0) for x in s.A]
    with hfx.Context(s, precision="fp64", sparse=sparse, q0_term=False) as c:
        c.load_system()
        c.build_all()
        want = [c.exchange(ik) for ik in range(s.n_k)]
    with hfx.Context(s, sparse=sparse, q0_term=False, work_bytes=kw.get("work_bytes", 0)) as c:
        c.load_system()
        st = c.build_all()
        assert st["n_batches"] >= (2 if "work_bytes" in kw else 1)
        got = [c.exchange(ik) for ik in range(s.n_k)]
        for keep in (True, False, False):   # kept, captured, replayed
            c.build_all(keep_products=keep)
            for ik in range(s.n_k):
                assert np.array_equal(c.exchange(ik), got[ik])
    for a, b in zip(got, want):
        assert np.abs(a - b).max() <= 5e-9 * np.abs(b).max()
