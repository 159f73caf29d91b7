"""Digits and residues cut from the interstitial plane at extreme column exponents (GB300
only).  Orbitals times 2^s and v times 2^(-4 s) leave V^x as it is: the operands carry their
exponents apart from the digits and the sums of Z^H Y stay at the same scale, so V^x is the
same to the last bit.  (P = 1: the channel blocks of mu = 0 functions work in FP32 pairs,
whose range is smaller.)"""
import copy

import numpy as np
import pytest

from paper_1003_0524_gb300 import hfx
from paper_1003_0524_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg,aux,nb,no", [(0, (90, 131), 7, 3), (3, (1560, 1600), 5, 3)])
def test_exchange_at_extreme_exponents(cfg, aux, nb, no):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1003_0524_gb300 import build
    build.build()
    s = S.make_system(dict(S.CONFIGS[cfg], P=1, sparse=False), mesh=(2, 1, 1), nb=nb, no=no, aux=("count", *aux), seed=6)
    want = None
    for shift in (0, -60, 47):
        u = copy.copy(s)
        u.c, u.A = [x * 2.0 ** shift for x in s.c], [x * 2.0 ** shift for x in s.A]
        u.v = [x * 2.0 ** (-4 * shift) for x in s.v]
        with hfx.Context(u, sparse="off", q0_term=False) as c:
            c.load_system()
            c.build_all()
            got = [c.exchange(ik) for ik in range(s.n_k)]
        if want is None:
            want = got
        for a, b in zip(got, want):
            assert np.array_equal(a, b)
