"""The Coulomb apply at lines whose elements are all of one size, through a caller's
projections (GB300 only).  One band is a column z of such elements, the others are unit
vectors of the first functions, so that V^x holds single elements of U z (U the upper
triangle): no sum of Z^H Y hides the error of the apply.  Both sides of the limits between
digits and residues (1664 and 6144 dense functions), against the sums in FP64.

Tolerance on the root mean square over 128 components: the operands of the residue apply
are rounded to units of at most 2^-38.39 of their line's norm, a sqrt(2 D) for D elements
a (+-1 +- i); the 4 D independent errors of a component add up to the standard deviation
2 D 2^-38.39 a b / sqrt 6 (both operands).  Those of the digits are smaller at D = 1663.
The digits of U z that Z^H Y reads have units of 2^(e-32), e the column's exponent.  The
mean square of 128 samples scatters by 6 % (one standard deviation, root): 1.4 is six.
"""
import math

import numpy as np
import pytest

from paper_1003_0524_gb300 import hfx
from paper_1003_0524_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [1663, 1664, 2660, 6144, 6145])
def test_lines_of_equal_magnitude(D):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1003_0524_gb300 import build
    build.build()
    nb = 65
    s = S.make_system(dict(S.CONFIGS[0], P=1, sparse=False), mesh=(1, 1, 1), nb=nb, no=1, aux=("count", 9, 9), seed=3)
    G, _ = S._g_count(S.kpoint_frac(s.mesh, 0), s.lattice, D - s.n_mt)
    rng = np.random.Generator(np.random.PCG64(D))

    def signs(*shape):
        return rng.integers(0, 2, shape) * 2.0 - 1.0 + 1j * (rng.integers(0, 2, shape) * 2.0 - 1.0)

    a, b = 0.249, 0.497
    v = np.triu(signs(D, D), 1) * a
    z = b * signs(D)
    uz = v @ z + 0.5 * a * z
    v += v.conj().T
    v[np.diag_indices(D)] = a
    Z = np.zeros((D, 1, nb), np.complex128)
    Z[np.arange(nb - 1), 0, np.arange(nb - 1)] = 1.0
    Z[:, 0, nb - 1] = z
    with hfx.Context(s, sparse="off", q0_term=False) as c:
        c.load_system(coulomb=False)
        hfx.hfx_set_coulomb(c.ctx, 0, G, v)
        c.set_products(0, 0, Z)
        st = c.build_all()
        got = -c.exchange(0)[:nb - 1, nb - 1]
    assert st["apply_products"] == (18 if 1664 <= D <= 6144 else 40)
    err = got - (v[:nb - 1] @ z)
    unit = 2.0 ** (math.frexp(max(np.abs(uz.real).max(), np.abs(uz.imag).max()))[1] - 32)
    apply = 2.0 * D * 2.0 ** -38.39 * a * b / math.sqrt(6.0)
    rms = math.sqrt(0.5 * np.mean(np.abs(err) ** 2))
    assert rms <= 1.4 * math.sqrt(apply ** 2 + unit ** 2 / 12.0)
