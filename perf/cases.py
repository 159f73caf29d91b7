"""Performance cases of the exchange-matrix library: what a user's program has it do.

A case is one pass through the Python entry points (paper_1003_0524_gb300.hfx) on
seeded inputs: the V^x build of a whole k mesh or of one k, an SCF step that first
uploads new wave functions, the start of an SCF cycle with new Coulomb matrices,
the LAPW transform of V^x, the muffin-tin product basis of one atom, and the q->0
bracket.  Cells, plane-wave cutoffs, band windows and basis sizes are those of the
workload table in paper_1003_0524_gb300/synthetic.py; meshes are cut to what one
pass can hold.  `exact` evaluates the defining sums with plain FP64 torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1003_0524_gb300 import hfx
from paper_1003_0524_gb300 import synthetic as S

DEV = "cuda:0"
WORK_BYTES = 24 << 30   # device budget of one batch: three contexts share the card

# Cells of the workload table, by their index there.
CELLS = {"1atom": 0, "2atom": 1, "5atom": 3, "10atom": 4}


def _build(name, cell, mesh, nb, no, aux, call="build", precision="sliced", inversion=False, P=None):
    c = {"kind": "build", "cell": cell, "mesh0": mesh[0], "mesh1": mesh[1], "mesh2": mesh[2],
         "nb_lo": nb[0], "nb_hi": nb[1], "no_lo": no[0], "no_hi": no[1], "aux_lo": aux[0], "aux_hi": aux[1],
         "P": S.CONFIGS[CELLS[cell]]["P"] if P is None else P,
         "call": call, "precision": precision, "inversion": inversion}
    return c if name is None else {"name": name, **c}


def listed():
    return [
        # the finite-size correction alone, as a caller without a context asks for it
        {"name": "q0_bracket_444", "kind": "bracket", "cell": "2atom", "mesh0": 4, "mesh1": 4, "mesh2": 4},
        # product basis of one atom from its radial functions, at the start of an SCF run
        {"name": "radial_basis", "kind": "radial", "lmax": 4, "Lmax": 4, "P": 3, "n_r": 600},
        # the smallest SCF step: new wave functions up, V^x and the energy back
        _build("scf_1atom_222", "1atom", (2, 2, 2), (8, 8), (4, 4), (130, 140), call="scf"),
        # a semiconductor on a converged mesh: many small pairs
        _build("build_2atom_444", "2atom", (4, 4, 4), (40, 40), (8, 8), (507, 507)),
        # the same with band windows and aux sets that differ from k to k, as an SCF step
        _build("scf_2atom_444_uneven", "2atom", (4, 4, 4), (32, 48), (6, 10), (520, 680), call="scf"),
        # an oxide with 120 bands on a coarse mesh
        _build("build_5atom_222", "5atom", (2, 2, 2), (120, 120), (20, 20), (1100, 1100)),
        # start of an SCF cycle: every v(q) is new, transformed and sliced before the build
        _build("coulomb_5atom_222", "5atom", (2, 2, 1), (40, 40), (8, 8), (1100, 1100), call="coulomb"),
        # the largest cell: V^x of a single k (a band-structure point)
        _build("kpoint_10atom_222", "10atom", (2, 2, 2), (250, 250), (48, 48), (2300, 2300), call="kpoint"),
        # the largest cell, whole mesh
        _build("build_10atom_222", "10atom", (2, 2, 2), (250, 250), (48, 48), (2300, 2300)),
        # the same with inversion symmetry: the real-valued path
        _build("build_10atom_inversion", "10atom", (2, 2, 2), (250, 250), (48, 48), (2300, 2300), inversion=True),
        # every step in FP64, for users who want no slicing
        _build("fp64_2atom_222", "2atom", (2, 2, 2), (40, 40), (8, 8), (507, 507), precision="fp64"),
        # V^x into the LAPW basis of every k, the step that follows a build
        _build("lapw_10atom_222", "10atom", (2, 2, 2), (250, 250), (4, 4), (60, 60), call="lapw"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["bracket", "radial", "scf", "build", "build", "build", "kpoint", "coulomb", "inversion", "fp64",
                       "lapw"])
    if kind == "bracket":
        return {"kind": "bracket", "cell": rng.choice(list(CELLS)), "mesh0": rng.randint(1, 6),
                "mesh1": rng.randint(1, 6), "mesh2": rng.randint(1, 6)}
    if kind == "radial":
        lmax = rng.randint(3, 6)
        return {"kind": "radial", "lmax": lmax, "Lmax": rng.randint(2, lmax), "P": rng.randint(2, 3),
                "n_r": _log(rng, 100, 900)}
    if kind == "fp64":
        nb = _log(rng, 8, 48)
        no = rng.randint(2, min(8, nb))
        return _build(None, rng.choice(["1atom", "2atom"]), (2, 2, rng.randint(1, 2)), (nb, nb), (no, no),
                      (60, _log(rng, 100, 507)), precision="fp64")
    if kind == "lapw":
        nb = _log(rng, 12, 250)
        return _build(None, rng.choice(["2atom", "10atom"]), (2, rng.randint(1, 2), 2), (nb, nb), (3, 3), (40, 70),
                      call="lapw")
    cell = rng.choice(["1atom", "2atom", "2atom", "5atom", "10atom"])
    mesh = {"1atom": (2, 2, 2), "2atom": (rng.randint(2, 4), rng.randint(2, 4), rng.randint(2, 4)),
            "5atom": (2, rng.randint(1, 2), rng.randint(1, 3)), "10atom": (2, rng.randint(1, 2), rng.randint(1, 2))}[cell]
    nbmax = {"1atom": 24, "2atom": 64, "5atom": 120, "10atom": 250}[cell]
    nomax = {"1atom": 6, "2atom": 10, "5atom": 20, "10atom": 48}[cell]
    auxmax = {"1atom": 140, "2atom": 680, "5atom": 1100, "10atom": 2300}[cell]
    nb_hi = _log(rng, 8, nbmax)
    nb_lo = rng.randint(max(4, nb_hi * 2 // 3), nb_hi)
    no_hi = min(rng.randint(2, nomax), nb_lo)
    no_lo = rng.randint(1, no_hi)
    aux_hi = rng.randint(auxmax // 3, auxmax)
    aux_lo = rng.randint(aux_hi * 3 // 4, aux_hi)
    P = 2 if cell == "10atom" else rng.randint(2, 3)
    return _build(None, cell, mesh, (nb_lo, nb_hi), (no_lo, no_hi), (aux_lo, aux_hi), P=P, inversion=kind == "inversion",
                  call=kind if kind in ("scf", "kpoint", "coulomb") else "build")


# ------------------------------------------------------------------ inputs
def _spec(case):
    return S.CONFIGS[CELLS[case["cell"]]]


def _mesh(case):
    return (case["mesh0"], case["mesh1"], case["mesh2"])


def _g_sorted(kf, lattice, radius):
    """Integer G with |k + G| <= radius, ascending in the norm (ties in lattice order)."""
    B = S.reciprocal(lattice)
    r = [np.arange(-b, b + 1) for b in
         (int(math.ceil(radius * np.linalg.norm(lattice[i]) / (2 * math.pi))) + 2 for i in range(3))]
    g = np.stack(np.meshgrid(*r, indexing="ij"), axis=-1).reshape(-1, 3)
    nrm = np.linalg.norm((kf[None, :] + g) @ B, axis=1)
    g, nrm = g[nrm <= radius + 1e-12], nrm[nrm <= radius + 1e-12]
    order = np.lexsort((g[:, 2], g[:, 1], g[:, 0], np.round(nrm, 12)))
    return np.ascontiguousarray(g[order].astype(np.int32)), nrm[order]


def _cn(gen, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=gen, device=DEV, dtype=torch.float64)) / math.sqrt(2.0)


def _mixed(gen, d, real):
    """U diag(d) U^H with U a product of Fourier (real: Hartley) transforms and random phases (signs):
    a dense Hermitian matrix with the eigenvalues d whose elements are all of one size."""
    n = d.shape[0]
    m = torch.diag(d).to(torch.float64 if real else torch.complex128)

    def rows(x):   # x -> F D x along dim 0
        if real:
            f = torch.fft.fft(x, dim=0, norm="ortho")
            return f.real - f.imag
        return torch.fft.fft(x, dim=0, norm="ortho")

    for _ in range(3):
        if real:
            p = torch.randint(0, 2, (n,), generator=gen, device=DEV).to(torch.float64) * 2 - 1
        else:
            p = torch.exp(2j * math.pi * torch.rand(n, generator=gen, device=DEV, dtype=torch.float64))
        m = rows(p[:, None] * m)
        m = rows(p[:, None] * m.mH).mH
    return 0.5 * (m + m.mH)


def _system(case, seed):
    """The inputs of a build as a synthetic.System (numpy arrays, as a host program holds them)."""
    spec, mesh, inv = _spec(case), _mesh(case), bool(case["inversion"])
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    rng = np.random.Generator(np.random.PCG64(seed))
    lattice = np.asarray(spec["lattice"], dtype=np.float64)
    pos = np.asarray(spec.get("pos_inv", spec["pos"]) if inv else spec["pos"], dtype=np.float64)
    rmt = np.asarray(spec["rmt"], dtype=np.float64)
    n_at, n_k = pos.shape[0], int(np.prod(mesh))
    lmax, Lmax, P = spec["lmax"], spec["Lmax"], int(case["P"])
    n_lp, nlm, nLM = 2 * (lmax + 1), (lmax + 1) ** 2, (Lmax + 1) ** 2
    partner = S.inversion_partners(pos, rmt) if inv else np.arange(n_at)
    # the counts of every k and q belong to the case, the values to the seed
    crng = np.random.Generator(np.random.PCG64(n_k))
    n_bands = crng.integers(case["nb_lo"], case["nb_hi"] + 1, size=n_k).astype(np.int32)
    n_occ = np.minimum(crng.integers(case["no_lo"], case["no_hi"] + 1, size=n_k), n_bands).astype(np.int32)
    n_ipw = crng.integers(case["aux_lo"], case["aux_hi"] + 1, size=n_k)

    Gk, c, A = [], [], []
    for ik in range(n_k):
        kf = S.kpoint_frac(mesh, ik)
        g, _ = _g_sorted(kf, lattice, spec["gmax"])
        nb = int(n_bands[ik])
        ck = _cn(gen, nb, g.shape[0]) / math.sqrt(g.shape[0])
        Ak = (_cn(gen, nb, n_at, 2 * nlm) * spec["a_scale"]).cpu().numpy()
        if inv:
            ck = (ck.real * math.sqrt(2.0)).to(torch.complex128)
            full = np.zeros_like(Ak)
            for a in range(n_at):
                b = int(partner[a])
                if b < a:
                    continue
                T = kf @ (pos[a] + pos[b])
                for l in range(lmax + 1):
                    sg = np.array([(-1.0) ** (l + m) for m in range(-l, l + 1)])
                    lo = 2 * l * l
                    blk = Ak[:, a, lo:lo + 2 * (2 * l + 1)].reshape(nb, 2 * l + 1, 2).copy()
                    mirror = np.exp(2j * math.pi * T) * (np.conj(blk) * sg[None, :, None])[:, ::-1]
                    if b == a:   # m > 0 and m < 0 belong together, m = 0 is fixed up to a real factor
                        blk[:, :l] = mirror[:, :l]
                        x = blk[:, l].real
                        blk[:, l] = np.exp(1j * math.pi * T) * (x if l % 2 == 0 else 1j * x)
                    else:
                        full[:, b, lo:lo + 2 * (2 * l + 1)] = mirror.reshape(nb, -1)
                    full[:, a, lo:lo + 2 * (2 * l + 1)] = blk.reshape(nb, -1)
            Ak = full
        Gk.append(g)
        c.append(ck.cpu().numpy())
        A.append(np.ascontiguousarray(Ak))

    R = rng.standard_normal((n_at, (Lmax + 1) * P, n_lp, n_lp)) * 0.1
    R = np.triu(R) + np.swapaxes(np.triu(R, 1), -1, -2)
    mu = rng.standard_normal((n_at, (Lmax + 1) * P))
    for a in range(n_at):
        if partner[a] < a:
            R[a], mu[a] = R[partner[a]], mu[partner[a]]

    # per channel an orthogonal frame whose first row is mu/|mu| (a Householder reflection)
    frames = np.zeros((n_at, Lmax + 1, P, P))
    for a in range(n_at):
        for L in range(Lmax + 1):
            x = mu[a, L * P:(L + 1) * P] / np.linalg.norm(mu[a, L * P:(L + 1) * P])
            w = x.copy()
            w[0] += 1.0 if x[0] >= 0 else -1.0
            frames[a, L] = (np.eye(P) - 2.0 * np.outer(w, w) / (w @ w)) * (-1.0 if x[0] >= 0 else 1.0)
    Ls = np.array([math.isqrt(i) for i in range(nLM)])
    F = torch.from_numpy(frames[:, Ls].reshape(n_at * nLM, P, P)).to(DEV)
    # channel whose blocks each channel shares (its partner's with inversion symmetry)
    src = np.arange(n_at * nLM)
    for a in range(n_at):
        for lm in range(nLM):
            L = int(Ls[lm])
            M = lm - L * L - L
            if inv and (partner[a] < a or (partner[a] == a and M > 0)):
                src[a * nLM + lm] = partner[a] * nLM + L * L + L - M
    src = torch.from_numpy(src).to(DEV)

    n_mt, nch = n_at * nLM * P, n_at * nLM
    scale = 4.0 * math.pi * spec["scale"]
    # |q + G| <= this holds at least the wanted count for every q
    rad = (1.3 * (int(n_ipw.max()) * abs(np.linalg.det(S.reciprocal(lattice))) * 3.0 / (4.0 * math.pi)) ** (1.0 / 3.0) + 1.0)
    Gaux, v = [], []
    for iq in range(n_k):
        g, nrm = _g_sorted(S.kpoint_frac(mesh, iq), lattice, rad)
        g, nrm = np.ascontiguousarray(g[:n_ipw[iq]]), nrm[:n_ipw[iq]]
        Gaux.append(g)
        gmax = float(nrm.max())
        kap = torch.rand(nch, generator=gen, device=DEV, dtype=torch.float64) * gmax
        gg = torch.cat([kap, torch.from_numpy(nrm).to(DEV)])
        d = scale / (gg * gg + 0.05)
        dense = _mixed(gen, d, inv)
        n_aux = n_mt + g.shape[0]
        vt = torch.zeros(n_aux, n_aux, device=DEV, dtype=torch.complex128)
        idx = torch.cat([torch.arange(nch, device=DEV) * P, n_mt + torch.arange(g.shape[0], device=DEV)])
        vt[idx[:, None], idx[None, :]] = dense.to(torch.complex128)
        if P > 1:   # multipole-free functions: a (P-1) x (P-1) block per channel and its weak coupling
            k2 = torch.rand(nch, generator=gen, device=DEV, dtype=torch.float64) * gmax
            w, cc = _cn(gen, nch, P - 1, P - 1), _cn(gen, nch, P - 1)
            if inv:
                w, cc = w.real.to(torch.complex128), cc.real.to(torch.complex128)
            eye = torch.eye(P - 1, device=DEV, dtype=torch.complex128)
            bc = (scale / (k2 * k2 + 0.05))[:, None, None] * 0.5 * (eye + w @ w.mH / (P - 1))
            bc = 0.5 * (bc + bc.mH)
            q = (cc.conj() * torch.linalg.solve(bc, cc[:, :, None])[:, :, 0]).sum(1).real
            cc = (cc * torch.sqrt(0.25 * float(d.min()) / q)[:, None])[src]
            bc = bc[src]
            o = (torch.arange(nch, device=DEV) * P)[:, None] + torch.arange(1, P, device=DEV)
            vt[o[:, :, None], o[:, None, :]] = bc
            vt[o, (torch.arange(nch, device=DEV) * P)[:, None]] = cc
            vt[(torch.arange(nch, device=DEV) * P)[:, None], o] = cc.conj()
        # back to the product-basis order: v = F^T v_t F block by block
        Fc = F.to(torch.complex128)
        vt[:n_mt] = torch.bmm(Fc.mT, vt[:n_mt].reshape(nch, P, n_aux)).reshape(n_mt, n_aux)
        right = vt[:, :n_mt].reshape(n_aux, nch, P).transpose(0, 1)
        vt[:, :n_mt] = torch.bmm(right, Fc).transpose(0, 1).reshape(n_aux, n_mt)
        v.append((0.5 * (vt + vt.mH)).cpu().numpy())
    return S.System(name=case["cell"], lattice=lattice, pos_frac=pos, rmt=rmt, lmax=lmax, Lmax=Lmax, P=P, mesh=mesh,
                    gmax=float(spec["gmax"]), n_bands=n_bands, n_occ=n_occ, Gk=Gk, c=c, A=A, R=R, mu=mu, Gaux=Gaux, v=v,
                    sparse=True, scale=float(spec["scale"]), seed=seed, inversion=inv)


def _overlaps(s, seed):
    """S_GG'(k) of the LAPW functions: the unit matrix and a positive part."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed + 7)
    out = []
    for g in s.Gk:
        w = _cn(gen, g.shape[0], g.shape[0])
        m = torch.eye(g.shape[0], device=DEV, dtype=torch.complex128) + 0.1 * (w @ w.mH) / g.shape[0]
        out.append((0.5 * (m + m.mH)).cpu().numpy())
    return out


def prepare(case, seed):
    if case["kind"] == "bracket":
        rng = np.random.Generator(np.random.PCG64(seed))
        return {"case": case, "lattice": np.asarray(_spec(case)["lattice"]) * rng.uniform(0.95, 1.05),
                "beta": rng.uniform(0.004, 0.006), "out": torch.zeros(1, device=DEV, dtype=torch.float64),
                "stream": torch.cuda.current_stream().cuda_stream}
    if case["kind"] == "radial":
        r, w, u = S.radial_functions(case["lmax"], 2.2, case["n_r"], seed)
        ctx = hfx.hfx_create(np.eye(3) * 10.0, np.zeros((1, 3)), np.array([2.2]), case["lmax"], case["Lmax"], case["P"],
                             (1, 1, 1))
        return {"case": case, "ctx": _Handle(ctx), "r": r, "w": w, "u": u}
    s = _system(case, seed)
    ctx = hfx.Context(s, precision=case["precision"], work_bytes=WORK_BYTES)
    ctx.load_system()
    state = {"case": case, "sys": s, "ctx": ctx}
    if case["call"] == "lapw":
        ctx.build_all()
        for ik, m in enumerate(_overlaps(s, seed)):
            hfx.hfx_set_overlap(ctx.ctx, ik, m)
    return state


class _Handle:
    def __init__(self, ctx):
        self.ctx = ctx

    def __del__(self):
        hfx.hfx_destroy(self.ctx)


def run(state):
    case = state["case"]
    if case["kind"] == "bracket":
        hfx.hfx_q0_bracket_noalloc(state["lattice"], _mesh(case), state["beta"], state["out"].data_ptr(), state["stream"])
        return state["out"]
    if case["kind"] == "radial":
        h = state["ctx"].ctx
        hfx.hfx_set_radial_functions(h, 0, state["r"], state["w"], state["u"], 1e-4)
        return hfx.hfx_get_radial_basis(h, 0, case["n_r"], case["lmax"], case["Lmax"], case["P"])
    s, ctx = state["sys"], state["ctx"]
    if case["call"] == "lapw":
        hfx.hfx_lapw_transform_all(ctx.ctx)
        return [hfx.hfx_get_lapw_exchange(ctx.ctx, ik, s.Gk[ik].shape[0]) for ik in range(s.n_k)]
    if case["call"] == "kpoint":
        return ctx.build_exchange(s.n_k - 1)
    if case["call"] == "scf":
        ctx.set_kpoints()
    if case["call"] == "coulomb":
        for iq in range(s.n_k):
            hfx.hfx_set_coulomb(ctx.ctx, iq, s.Gaux[iq], s.v[iq])
    ctx.build_all()
    return {"vx": np.concatenate([ctx.exchange(ik).ravel() for ik in range(s.n_k)]), "energy": ctx.energy()}


# ------------------------------------------------------------------ work
def _mean(case, key):
    return 0.5 * (case[key + "_lo"] + case[key + "_hi"])


def _sizes(case):
    spec = _spec(case)
    n_at, P = len(spec["pos"]), case["P"]
    vol = abs(np.linalg.det(np.asarray(spec["lattice"], dtype=np.float64)))
    npw = vol * spec["gmax"] ** 3 / (6.0 * math.pi ** 2)
    nch = n_at * (spec["Lmax"] + 1) ** 2
    return {"nk": int(np.prod(_mesh(case))), "nb": _mean(case, "nb"), "no": _mean(case, "no"), "nipw": _mean(case, "aux"),
            "npw": npw, "nch": nch, "nmt": nch * P, "P": P, "nat": n_at, "nlmp": 2 * (spec["lmax"] + 1) ** 2}


def work(case):
    if case["kind"] == "bracket":
        # one exponential per G of the sphere |q + G| <= q0, over every q
        lat = np.asarray(_spec(case)["lattice"], dtype=np.float64)
        q0 = math.sqrt(-math.log(0.005) / 0.005)
        n = q0 ** 3 * abs(np.linalg.det(lat)) / (6.0 * math.pi ** 2) * int(np.prod(_mesh(case)))
        return {"bytes": 8.0, "flops": 30.0 * n}
    if case["kind"] == "radial":
        nlp, n_r, P, nL = 2 * (case["lmax"] + 1), case["n_r"], case["P"], case["Lmax"] + 1
        nc = nlp * (nlp + 1) / 2
        # overlaps, a symmetric eigenproblem, the functions and their integrals, per L
        fl = nL * (nc * nc * n_r + 9.0 * nc ** 3 + 2.0 * P * nc * n_r + 2.0 * P * nc * n_r + 4.0 * P * P * n_r)
        by = 8.0 * (n_r * (2 + nlp) + nL * P * (n_r + 1 + nlp * nlp + P))
        return {"bytes": by, "flops": fl}
    z = _sizes(case)
    nk, m, n, naux = z["nk"], z["no"], z["nb"], z["nmt"] + z["nipw"]
    if case["call"] == "lapw":
        return {"bytes": 16.0 * nk * (2 * z["npw"] ** 2 + n * z["npw"] + n * n),
                "flops": 8.0 * nk * (n * z["npw"] ** 2 + n * n * z["npw"] + z["npw"] ** 2 * n)}
    D = z["nch"] + z["nipw"]
    nnz = D * D + z["nch"] * (z["P"] ** 2 - 1)
    pairs = nk * (1 if case["call"] == "kpoint" else nk)
    f = 2.0 if case["inversion"] else 8.0
    per = f * m * n * (nnz + naux * n) + f * m * n * (z["nlmp"] * z["nmt"] + z["nipw"] * z["npw"])
    by = 16.0 * nk * (n * (z["npw"] + z["nat"] * z["nlmp"]) + naux * naux + n * n)
    return {"bytes": by, "flops": pairs * per}


# ------------------------------------------------------------------ exact values
EXACT_MAX_FLOPS = 9e12   # about ten seconds of FP64 on the device


def _legendre_norm(lmax, x):
    """Normalised associated Legendre functions N_lm P_lm(x), m >= 0, with the Condon-Shortley phase."""
    p = np.zeros((lmax + 1, lmax + 1, x.size))
    s = np.sqrt(1.0 - x * x)
    p[0, 0] = math.sqrt(1.0 / (4.0 * math.pi))
    for m in range(1, lmax + 1):
        p[m, m] = -math.sqrt((2 * m + 1) / (2.0 * m)) * s * p[m - 1, m - 1]
    for m in range(lmax + 1):
        for l in range(m + 1, lmax + 1):
            a = math.sqrt((4.0 * l * l - 1.0) / (l * l - m * m))
            b = math.sqrt(((l - 1.0) ** 2 - m * m) / (4.0 * (l - 1.0) ** 2 - 1.0)) if l - 1 > m else 0.0
            p[l, m] = a * (x * p[l - 1, m] - (b * p[l - 2, m] if l - 1 > m else 0.0))
    return p


def _ylm(lmax, x, phi):
    p = _legendre_norm(lmax, x)
    y = np.zeros(((lmax + 1) ** 2, x.size, phi.size), dtype=np.complex128)
    for l in range(lmax + 1):
        for m in range(l + 1):
            v = p[l, m][:, None] * np.exp(1j * m * phi)[None, :]
            y[l * l + l + m] = v
            y[l * l + l - m] = (-1.0) ** m * np.conj(v)
    return y


def _gaunt(Lmax, lmax):
    """G[LM, lm, l'm'] = int Y*_LM Y*_lm Y_l'm' by a quadrature that is exact for these degrees."""
    x, w = np.polynomial.legendre.leggauss(Lmax + 2 * lmax + 2)
    nphi = 2 * (Lmax + 2 * lmax) + 3
    phi = 2.0 * math.pi * np.arange(nphi) / nphi
    Y, y = _ylm(Lmax, x, phi), _ylm(lmax, x, phi)
    wt = (w[:, None] * (2.0 * math.pi / nphi) * np.ones(nphi)[None, :]).ravel()
    Y, y = Y.reshape(Y.shape[0], -1), y.reshape(y.shape[0], -1)
    g = np.einsum("Ai,abi->Aab", np.conj(Y) * wt, np.conj(y)[:, None, :] * y[None, :, :], optimize=True).real
    g[np.abs(g) < 1e-13] = 0.0
    return g


def _bracket(lattice, mesh, beta):
    omega, nk = abs(np.linalg.det(lattice)), int(np.prod(mesh))
    q0 = math.sqrt(-math.log(beta) / beta)
    B = torch.from_numpy(S.reciprocal(lattice)).to(DEV)
    bound = [int(math.ceil(q0 * np.linalg.norm(lattice[i]) / (2 * math.pi))) + 2 for i in range(3)]
    g = torch.cartesian_prod(*[torch.arange(-b, b + 1, device=DEV, dtype=torch.float64) for b in bound])
    tot = 0.0
    for iq in range(nk):
        x = (g + torch.from_numpy(S.kpoint_frac(mesh, iq)).to(DEV)) @ B
        n2 = (x * x).sum(1)
        n2 = n2[(n2 > 1e-20) & (n2 <= q0 * q0)]
        tot += float((torch.exp(-beta * n2) / n2).sum())
    return math.erf(math.sqrt(beta) * q0) / math.sqrt(math.pi * beta) - 4.0 * math.pi / (nk * omega) * tot


def _exact_vx(s, ks):
    """V^x(k) of the listed k by the defining sums, and the energy where every k is listed."""
    nk, n_at, P, Lmax, lmax = s.n_k, s.n_atoms, s.P, s.Lmax, s.lmax
    nLM, nlm, omega = (Lmax + 1) ** 2, (lmax + 1) ** 2, abs(np.linalg.det(s.lattice))
    c128 = torch.complex128
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
    Bm = t(S.reciprocal(s.lattice))
    pos, mesh = s.pos_frac, s.mesh
    # W[LM P, lmp, l'm'p'] of one atom: Gaunt times radial integral
    g = t(_gaunt(Lmax, lmax))
    Ls = torch.tensor([math.isqrt(i) for i in range(nLM)], device=DEV)
    ls = torch.tensor([math.isqrt(i) for i in range(nlm)], device=DEV)
    W = []
    for a in range(n_at):
        R = t(s.R[a]).reshape(Lmax + 1, P, lmax + 1, 2, lmax + 1, 2)
        R = R[Ls][:, :, ls][:, :, :, :, ls]                      # [LM, P, lm, p, l'm', p']
        W.append((R * g[:, None, :, None, :, None]).reshape(nLM * P, 2 * nlm, 2 * nlm).to(c128))
    # the box of K = G + G1 - G0 and T_n(K) = sum_G2 Theta_{K - G2} c_G2
    lo = np.min([x.min(0) for x in s.Gk], 0) + np.min([x.min(0) for x in s.Gaux], 0)
    hi = np.max([x.max(0) for x in s.Gk], 0) + np.max([x.max(0) for x in s.Gaux], 0) + 1
    dim = hi - lo + 1
    K = torch.cartesian_prod(*[torch.arange(int(a), int(b) + 1, device=DEV) for a, b in zip(lo, hi)])

    def theta(d):   # d [..., 3] integer
        kc = d.to(torch.float64) @ Bm
        kn = kc.norm(dim=-1)
        out = (kn < 1e-12).to(c128)
        for a in range(n_at):
            x = kn * float(s.rmt[a])
            j1 = torch.where(x < 1e-8, torch.full_like(x, 1.0 / 3.0), (torch.sin(x) - x * torch.cos(x)) / x.clamp_min(1e-8) ** 3)
            ph = torch.exp(-2j * math.pi * (d.to(torch.float64) @ t(pos[a])))
            out -= (4.0 * math.pi * float(s.rmt[a]) ** 3 / omega) * j1 * ph
        return out

    partner = S.inversion_partners(pos, s.rmt) if s.inversion else None
    vg = {}
    out, ex = [], 0.0
    q0b = _bracket(s.lattice, mesh, 0.005)
    for ik in ks:
        n = int(s.n_bands[ik])
        A = t(s.A[ik])
        Bk = torch.stack([torch.einsum("Iab,nb->Ian", W[a], A[:, a]) for a in range(n_at)])   # [at, I, lmp, n]
        ck, T = t(s.c[ik]), torch.empty(K.shape[0], n, device=DEV, dtype=c128)
        for i0 in range(0, K.shape[0], 8192):
            T[i0:i0 + 8192] = theta(K[i0:i0 + 8192, None, :] - t(s.Gk[ik]).long()[None]) @ ck.T
        V = torch.zeros(n, n, device=DEV, dtype=c128)
        jk = np.array([ik // (mesh[1] * mesh[2]), (ik // mesh[2]) % mesh[1], ik % mesh[2]])
        for iq in range(nk):
            jq = np.array([iq // (mesh[1] * mesh[2]), (iq // mesh[2]) % mesh[1], iq % mesh[2]])
            jp = (jk - jq) % np.array(mesh)
            g0 = (jk - jq - jp) // np.array(mesh)
            ikp = S.kpoint_index(mesh, jp)
            m = int(s.n_occ[ikp])
            if m == 0:
                continue
            G, G1 = t(s.Gaux[iq]).long(), t(s.Gk[ikp]).long()
            naux = s.n_aux(iq)
            Z = torch.empty(naux, m, n, device=DEV, dtype=c128)
            Am = t(s.A[ikp][:m]).conj()
            ph = np.exp(-2j * math.pi * (pos @ S.kpoint_frac(mesh, iq)))
            for a in range(n_at):
                Z[a * nLM * P:(a + 1) * nLM * P] = complex(ph[a]) * torch.einsum("ml,Iln->Imn", Am[:, a], Bk[a])
            cm = t(s.c[ikp][:m]).conj() / math.sqrt(omega)
            base = G - torch.from_numpy(g0 + lo).to(DEV)
            st = max(1, int(2e8 / (G1.shape[0] * n * 16)) * 2)
            for i0 in range(0, G.shape[0], st):
                x = base[i0:i0 + st, None, :] + G1[None]
                idx = (x[..., 0] * int(dim[1]) + x[..., 1]) * int(dim[2]) + x[..., 2]
                Z[s.n_mt + i0:s.n_mt + i0 + x.shape[0]] = torch.matmul(cm, T[idx])
            if s.inversion:   # <M'| of the symmetrized functions
                r = math.sqrt(0.5)
                for a in range(n_at):
                    b = int(partner[a])
                    for L in range(Lmax + 1):
                        for M in range(-L, L + 1):
                            i = (a * nLM + L * L + L + M) * P
                            j = (b * nLM + L * L + L - M) * P
                            if a == b and M == 0:
                                Z[i:i + P] *= 1.0 if L % 2 == 0 else -1j
                            elif a < b or (a == b and M < 0):
                                u, w = Z[i:i + P].clone(), (-1.0) ** (L + M) * Z[j:j + P]
                                Z[i:i + P], Z[j:j + P] = r * (u + w), -1j * r * (u - w)
            if iq not in vg:
                vg[iq] = t(s.v[iq])
            for m0 in range(0, m, 16):
                z = Z[:, m0:m0 + 16]
                y = (vg[iq] @ z.reshape(naux, -1)).reshape(z.shape)
                V += torch.einsum("Imn,Imp->np", z.conj(), y)
            del Z
        V /= -float(nk)
        occ = torch.arange(n, device=DEV) < int(s.n_occ[ik])
        V -= torch.diag(occ.to(c128) * q0b)
        ex += 0.5 / nk * float(V.diagonal().real[occ].sum())
        out.append(V)
    return out, ex


def _exact_radial(case, seed):
    r, w, u = S.radial_functions(case["lmax"], 2.2, case["n_r"], seed)
    nlp, P, nL, n_r = 2 * (case["lmax"] + 1), case["P"], case["Lmax"] + 1, r.size
    wr = w * r * r
    M, mu = np.zeros((nL * P, n_r)), np.zeros(nL * P)
    R, C = np.zeros((nL * P, nlp, nlp)), np.zeros((nL, P, P))
    for L in range(nL):
        f = []
        for a in range(nlp):
            for b in range(a, nlp):
                if abs(a // 2 - b // 2) <= L <= a // 2 + b // 2:
                    x = u[a] * u[b]
                    f.append(x / math.sqrt(wr @ (x * x)))
        f = np.array(f)
        got = []
        if L == 0:
            got.append(np.full(n_r, 1.0 / math.sqrt(wr.sum())))
            f = f - np.outer(f @ (wr * got[0]), got[0])
        ev, vec = np.linalg.eigh((f * wr) @ f.T)
        for k in np.argsort(-ev)[:P - len(got)]:
            x = vec[:, k] * (1.0 if vec[np.argmax(np.abs(vec[:, k])), k] >= 0 else -1.0)
            got.append(x @ f / math.sqrt(ev[k]))
        got = np.array(got)
        rl, rg = np.minimum(r[:, None], r[None, :]), np.maximum(r[:, None], r[None, :])
        M[L * P:(L + 1) * P] = got
        mu[L * P:(L + 1) * P] = got @ (w * r ** (L + 2))
        R[L * P:(L + 1) * P] = np.einsum("pi,ai,bi->pab", got * wr, u, u, optimize=True)
        C[L] = 4.0 * math.pi / (2 * L + 1) * (got * wr) @ (rl ** L / rg ** (L + 1)) @ (got * wr).T
    return {"M": M, "mu": mu, "R": R, "C": C}


def exact(case, seed):
    if case["kind"] == "bracket":
        s = prepare(case, seed)
        return torch.tensor([_bracket(s["lattice"], _mesh(case), s["beta"])], device=DEV, dtype=torch.float64)
    if case["kind"] == "radial":
        return _exact_radial(case, seed)
    if case["call"] != "lapw":
        complex_work = work({**case, "inversion": False})["flops"]
        if complex_work > EXACT_MAX_FLOPS:
            return None
    s = _system(case, seed)
    if case["call"] == "kpoint":
        return _exact_vx(s, [s.n_k - 1])[0][0].cpu().numpy()
    vx, ex = _exact_vx(s, range(s.n_k))
    if case["call"] == "lapw":
        out = []
        for ik, m in enumerate(_overlaps(s, seed)):
            sc = torch.from_numpy(m).to(DEV) @ torch.from_numpy(s.c[ik]).to(DEV).T
            out.append((sc @ vx[ik] @ sc.mH).cpu().numpy())
        return out
    return {"vx": np.concatenate([x.cpu().numpy().ravel() for x in vx]), "energy": ex}
