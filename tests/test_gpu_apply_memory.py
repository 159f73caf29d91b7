"""The residue apply needs more memory than the digits (GB300 only): where a pair fits only
with the digits, the build takes those instead of failing.  The card is filled step by step
until a build no longer fits: the last one that does runs on digits, the first on residues,
and both give the same V^x within the tolerance of either (5e-9 of the largest element)."""
import numpy as np
import pytest

from paper_1003_0524_gb300 import hfx
from paper_1003_0524_gb300 import synthetic as S

pytestmark = pytest.mark.gpu


def test_digits_where_residues_do_not_fit():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1003_0524_gb300 import build
    build.build()
    s = S.make_system(dict(S.CONFIGS[3], P=1, sparse=False, aux=("count", 9, 9)), mesh=(1, 1, 1), nb=100, no=40, seed=4)
    n = 1700
    G, _ = S._g_count(S.kpoint_frac(s.mesh, 0), s.lattice, n - s.n_mt)
    rng = np.random.Generator(np.random.PCG64(2))
    v = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    v = v + v.conj().T + 200.0 * np.eye(n)
    torch.cuda.empty_cache()
    runs = []
    for left in np.arange(3.6, 1.2, -0.06):
        fill = torch.empty(torch.cuda.mem_get_info()[0] - int(left * 2 ** 30), dtype=torch.uint8, device="cuda:0")
        try:
            with hfx.Context(s, sparse="off") as c:
                c.load_system(coulomb=False)
                hfx.hfx_set_coulomb(c.ctx, 0, G, v)
                st = c.build_all()
                runs.append((st["apply_products"], c.exchange(0)))
        except hfx.HfxError as e:
            assert e.code == hfx.HFX_ENOMEM
            break
        finally:
            del fill
            torch.cuda.empty_cache()
    assert runs[0][0] == 18 and runs[-1][0] == 40
    assert np.abs(runs[0][1] - runs[-1][1]).max() <= 5e-9 * np.abs(runs[0][1]).max()
