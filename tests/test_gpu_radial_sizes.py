"""The radial-basis kernels at the edges of their sizes, against numpy (GB300 only):
one product per L, tiles of the overlap kernel one over and one under 16, the largest
angular cutoff (114 products), the most functions per channel (P = 16), grids below
one block and above one chunk per thread, and duplicated products (a rank-deficient
overlap matrix with a multiple zero eigenvalue).

Tolerance: the wanted eigenvalues lie above 1e-4 of a matrix of norm <= 114, so an
eigenpair carries at most ~114 * 1e-16 / 1e-4 ~ 1e-10 relative error; 1e-9 of the
largest value is taken (the functions are of order 1 to 10).
"""
import math

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


def reference(r, w, u, lmax, Lmax, P):
    nlp, wr = 2 * (lmax + 1), w * r * r
    out = {"M": np.zeros(((Lmax + 1) * P, r.size)), "mu": np.zeros((Lmax + 1) * P),
           "R": np.zeros(((Lmax + 1) * P, nlp, nlp)), "C": np.zeros((Lmax + 1, P, P))}
    for L in range(Lmax + 1):
        f = [u[a] * u[b] for a in range(nlp) for b in range(a, nlp) if abs(a // 2 - b // 2) <= L <= a // 2 + b // 2]
        f = np.array([x / math.sqrt(wr @ (x * x)) for x in f if wr @ (x * x) > 0])
        got = []
        if L == 0:
            got.append(np.full(r.size, 1.0 / math.sqrt(wr.sum())))
            f = f - np.outer(f @ (wr * got[0]), got[0])
        ev, vec = np.linalg.eigh((f * wr) @ f.T)
        for k in np.argsort(-ev)[:P - len(got)]:
            assert ev[k] > 1e-4
            x = vec[:, k] * (1.0 if vec[np.argmax(np.abs(vec[:, k])), k] >= 0 else -1.0)
            got.append(x @ f / math.sqrt(ev[k]))
        got = np.array(got)
        rl, rg = np.minimum(r[:, None], r[None, :]), np.maximum(r[:, None], r[None, :])
        s = slice(L * P, (L + 1) * P)
        out["M"][s], out["mu"][s] = got, got @ (w * r ** (L + 2))
        out["R"][s] = np.einsum("pi,ai,bi->pab", got * wr, u, u, optimize=True)
        out["C"][L] = 4.0 * math.pi / (2 * L + 1) * (got * wr) @ (rl ** L / rg ** (L + 1)) @ (got * wr).T
    return out


def _u(lmax, n_r, seed, wild=False):
    """wild: oscillating functions, so that many eigenvalues lie above the threshold."""
    r, w, u = S.radial_functions(lmax, 2.0, n_r, seed)
    if wild:
        k = np.arange(u.shape[0])[:, None] + 1.0
        u = np.cos(3.1 * k * r[None, :] + k)
    return r, w, u


@pytest.mark.parametrize("lmax,Lmax,P,n_r,wild", [
    (0, 0, 1, 40, False),     # L = 0 holds the constant alone
    (0, 0, 3, 40, True),      # three products, two wanted after the constant
    (1, 2, 2, 33, False),     # the last L has one product pair
    (3, 3, 3, 100, False),
    (4, 4, 3, 31, False),     # fewer points than a warp
    (4, 2, 16, 400, True),    # the most functions per channel
    (8, 8, 4, 257, False),    # 114 products: the largest shared memory
    (2, 2, 2, 8192, False),   # the longest grid
])
def test_radial_basis_at_its_edges(lmax, Lmax, P, n_r, wild):
    r, w, u = _u(lmax, n_r, 11 + lmax, wild)
    ref = reference(r, w, u, lmax, Lmax, P)
    ctx = hfx.hfx_create(np.eye(3) * 9.0, np.zeros((1, 3)), np.array([2.0]), lmax, Lmax, P, (1, 1, 1))
    try:
        for _ in range(2):   # the second call reuses the context's buffer
            hfx.hfx_set_radial_functions(ctx, 0, r, w, u, 1e-4)
            got = hfx.hfx_get_radial_basis(ctx, 0, n_r, lmax, Lmax, P)
            for key in ref:
                assert np.abs(got[key] - ref[key]).max() <= 1e-9 * max(1.0, np.abs(ref[key]).max()), key
    finally:
        hfx.hfx_destroy(ctx)


def test_duplicated_products_leave_the_span():
    """u-dot equal to u: every product occurs three or four times.  The basis is then
    that of the distinct products up to the weights; it stays orthonormal."""
    r, w, u = _u(4, 200, 3)
    u[1::2] = u[0::2]
    ctx = hfx.hfx_create(np.eye(3) * 9.0, np.zeros((1, 3)), np.array([2.0]), 4, 4, 2, (1, 1, 1))
    try:
        hfx.hfx_set_radial_functions(ctx, 0, r, w, u, 1e-4)
        M = hfx.hfx_get_radial_basis(ctx, 0, 200, 4, 4, 2)["M"]
    finally:
        hfx.hfx_destroy(ctx)
    ref = reference(r, w, u, 4, 4, 2)["M"]
    for L in range(5):
        m = M[2 * L:2 * L + 2]
        assert np.abs((m * w * r * r) @ m.T - np.eye(2)).max() <= 1e-9
        # equal components of a duplicated product leave its sign open
        assert np.abs(np.abs(m) - np.abs(ref[2 * L:2 * L + 2])).max() <= 1e-9 * np.abs(ref).max()


@pytest.mark.parametrize("scale", [1e200, 0.0])
def test_overflowing_or_vanishing_products_are_rejected(scale):
    r, w, u = _u(2, 50, 5)
    ctx = hfx.hfx_create(np.eye(3) * 9.0, np.zeros((1, 3)), np.array([2.0]), 2, 2, 2, (1, 1, 1))
    try:
        with pytest.raises(hfx.HfxError) as e:
            hfx.hfx_set_radial_functions(ctx, 0, r, w, u * scale, 1e-4)
        assert e.value.code == hfx.HFX_EINVAL
    finally:
        hfx.hfx_destroy(ctx)
