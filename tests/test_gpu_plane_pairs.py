"""The interstitial plane as pairs of FP32 numbers in units of a column's power of two
(GB300 only).  The operands carry the exponents apart from the digits, so orbitals times
2^s give projections times 2^(2 s) to the last bit at any s, and, inside the FP32 range of
the Z^H Y sums, V^x times 2^(4 s) (off the diagonal, which has a term that does not depend
on the orbitals), on the digit and on the residue apply: odd band counts put pairs of
columns off the 32-byte boundary of a store, one k has far smaller orbitals than the
others."""
import copy

import numpy as np
import pytest

from paper_1003_0524_gb300 import hfx
from paper_1003_0524_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg,aux,nb,no", [
    (1, (90, 131), 7, 3),
    (2, (33, 64), ("U", 3, 13), ("U", 1, 3)),
    (3, (1180, 1200), 5, 3),
])
def test_powers_of_two_go_through(cfg, aux, nb, no):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1003_0524_gb300 import build
    build.build()
    s = S.make_system(dict(S.CONFIGS[cfg], aux=("count", *aux)), mesh=(2, 1, 1), nb=nb, no=no, seed=5)
    s.c[1], s.A[1] = s.c[1] * 2.0 ** -9, s.A[1] * 2.0 ** -9

    def build_v(shift):
        u = copy.copy(s)
        u.c, u.A = [x * 2.0 ** shift for x in s.c], [x * 2.0 ** shift for x in s.A]
        with hfx.Context(u) as c:
            c.load_system()
            c.build_all()
            v = [c.exchange(ik) for ik in range(s.n_k)]
            c.build_all(keep_products=True)
            return v, [c.products(0, 0, 0), c.products(1, 1, 0)]

    want, wz = build_v(0)
    with hfx.Context(s, precision="fp64") as c:
        c.load_system()
        c.build_all()
        for ik in range(s.n_k):
            v = c.exchange(ik)
            assert np.abs(want[ik] - v).max() <= 5e-9 * np.abs(v).max()
    for shift in (-60, -8, 20, 47):
        v, z = build_v(shift)
        for a, b in zip(z, wz):
            assert np.array_equal(a, b * 2.0 ** (2 * shift))
        for a, b in zip(v, want):
            off = ~np.eye(len(a), dtype=bool)
            if abs(shift) <= 20:
                assert np.array_equal(a[off], b[off] * 2.0 ** (4 * shift))
