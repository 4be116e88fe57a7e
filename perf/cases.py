"""Timed cases of the JK build: what a user's program calls, over the range of sizes, precisions and options.

The workloads are the shapes the library's benchmark and tests use: 6-31G*-shaped molecules of 3 to 60 atoms (one at a
time and in batches), water-like clusters, uncontracted s p d f shells in Cartesian and real solid harmonic form, and the
training gradient of the precision router. A case is one SCF iteration's build (or one router gradient) on a handle that
the program keeps; every input is drawn from the seed.
"""
import itertools
import math

import numpy as np
import torch

from paper_2507_09772_gb300 import jk, synth

CUTOFF = 1e-13
ROUTER_N = 5313
SPDF = (("s", 0, 3), ("p", 1, 1), ("d", 2, 1), ("f", 3, 1))   # shells of an atom of the high angular momentum cases


# ------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest call: one iteration on a three-atom molecule, captured in a graph, nothing waited for
        dict(name="tiny_fp64", kind="mol", natm=3, heavy=True, precision="fp64", ndm=1, out="jk", omega=0.0, graph=True),
        # a small organic molecule with every option at its default (eager launches, checked results)
        dict(name="mol20_fp64", kind="mol", natm=20, precision="fp64", ndm=1, out="jk", omega=0.0, graph=False),
        # an open-shell molecule of odd size: two densities, mixed precision, default options
        dict(name="mol33_uhf_mixed", kind="mol", natm=33, precision="mixed", ndm=2, out="jk", omega=0.0, graph=False),
        # exchange of a range-separated hybrid functional: K only, short-range operator
        dict(name="mol14_erfc_k", kind="mol", natm=14, precision="fp64", ndm=1, out="k", omega=-0.3, graph=False),
        # a late iteration of a pure functional: J of a small density change, screened on the change
        dict(name="mol41_incremental_j", kind="mol", natm=41, precision="fp64", ndm=1, out="j", omega=0.0, graph=True,
             delta=1e-5),
        # high-throughput screening: independent molecules in one handle, plain FP64 and mixed precision
        dict(name="batch8_fp64", kind="batch", nmol=8, lo=10, hi=60, precision="fp64", ndm=1, out="jk", omega=0.0,
             graph=True),
        dict(name="batch24_mixed", kind="batch", nmol=24, lo=10, hi=60, precision="mixed", ndm=1, out="jk", omega=0.0,
             graph=True),
        # one large system: 120 atoms of a water-like cluster
        dict(name="cluster40_mixed", kind="cluster", units=40, precision="mixed", ndm=1, out="jk", omega=0.0, graph=True),
        # high angular momentum in both forms of the functions
        dict(name="spdf6_sph_fp64", kind="spdf", natm=6, spherical=True, precision="fp64", ndm=1, out="jk", omega=0.0,
             graph=True),
        dict(name="spdf9_cart_mixed", kind="spdf", natm=9, spherical=False, precision="mixed", ndm=1, out="jk", omega=0.0,
             graph=False),
        # the learned precision router inside a mixed build, and the gradient its training takes
        dict(name="mol45_routed", kind="mol", natm=45, precision="routed", ndm=1, out="jk", omega=0.0, graph=True),
        dict(name="router_gradient", kind="router", rows=50000, noalloc=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["mol", "mol", "mol", "batch", "cluster", "spdf", "router"])
    if kind == "router":
        rows = _log_int(rng, 500, 200000)
        return dict(kind="router", rows=rows, noalloc=rows <= jk_noalloc_rows() and rng.random() < 0.5)
    c = dict(kind=kind, precision=rng.choice(["fp64", "mixed"]), ndm=1, out="jk", omega=0.0, graph=rng.random() < 0.5)
    if kind == "mol":
        form = rng.choice(["plain", "plain", "uhf", "erfc_k", "incremental_j", "routed"])
        if form == "plain":
            c.update(natm=_log_int(rng, 4, 60))
        elif form == "uhf":
            c.update(natm=_log_int(rng, 4, 40), ndm=2)
        elif form == "erfc_k":
            c.update(natm=_log_int(rng, 4, 30), precision="fp64", out="k", omega=-round(rng.uniform(0.1, 0.5), 3))
        elif form == "incremental_j":
            c.update(natm=_log_int(rng, 10, 60), precision="fp64", out="j", delta=10.0 ** -rng.randint(3, 7))
        else:
            c.update(natm=_log_int(rng, 10, 60), precision="routed")
    elif kind == "batch":
        lo = rng.randint(6, 20)
        c.update(nmol=rng.randint(2, 8 if c["precision"] == "fp64" else 24), lo=lo, hi=rng.randint(lo + 5, 60))
    elif kind == "cluster":
        c.update(units=_log_int(rng, 4, 18 if c["precision"] == "fp64" else 40))
    else:
        c.update(natm=_log_int(rng, 2, 9), spherical=rng.random() < 0.5)
    return c


def jk_noalloc_rows():
    return 65536


# ------------------------------------------------------------------ inputs
def _molecules(case, seed):
    """The molecules of a case with their densities (numpy, FP64)."""
    n_dm = case["ndm"]
    base = 7919 * (seed % 1000003) + 17
    if case["kind"] == "mol":
        if case.get("heavy"):
            mols = [synth.tiny_631gs(base, n_dm)]
        else:
            mols = [synth.batched_molecule(0, base, n_dm, natm=case["natm"])]
    elif case["kind"] == "batch":
        sizes = np.linspace(case["lo"], case["hi"], case["nmol"]).round().astype(int)
        mols = [synth.batched_molecule(i, base, n_dm, natm=int(n)) for i, n in enumerate(sizes)]
    elif case["kind"] == "cluster":
        mols = [synth.water_like_cluster(case["units"], base, n_dm)]
    else:
        rng = np.random.default_rng(base)
        xyz = synth._rejection_box(rng, case["natm"], (case["natm"] / 0.1) ** (1.0 / 3.0), 0.9)
        atom = []
        for _ in range(case["natm"]):
            atom.append([(l, np.sort(np.exp(rng.uniform(math.log(0.2), math.log(20.0 if l == 0 else 2.0), n)))[::-1])
                         for _, l, n in SPDF])
        mols = [synth.custom_basis_molecule(xyz, atom, rng, spherical=case["spherical"], n_dm=n_dm, name="spdf")]
    if case.get("delta"):
        for m in mols:   # a change of the density: symmetric, of low rank, small
            rng = np.random.default_rng(base + 1)
            v = rng.standard_normal((m.D.shape[0], m.nao, 4)) / math.sqrt(m.nao)
            m.D = case["delta"] * np.einsum("kir,r,kjr->kij", v, np.array([1.0, -1.0, 0.5, -0.5]), v)
    return mols


def _blob():
    """Router weights such as a program loads from its disk: a mild network around a negative mean prediction."""
    rng = np.random.default_rng(99)
    theta = np.zeros(ROUTER_N, np.float32)
    theta[:12 * 64] = rng.normal(0, 0.15, 12 * 64)
    theta[1024:1088] = rng.normal(0, 0.05, 64)
    theta[1088:1088 + 4096] = rng.normal(0, 0.1, 4096)
    theta[5184:5248] = rng.normal(0, 0.05, 64)
    theta[5248:5312] = rng.normal(0, 0.1, 64)
    theta[5312] = -0.8
    mu = np.array([0.5, 3.0, 0.5, 3.0, 3.0, 3.0, 4.0, -1.0, -1.0, -0.7, 2.0, 1.0, 0, 0, 0, 0], np.float32)
    isd = np.array([1.0, 0.5, 1.0, 0.5, 0.4, 0.4, 0.4, 1.0, 1.0, 3.0, 0.7, 1.7, 0, 0, 0, 0], np.float32)
    return mu, isd, theta


def _jk_blob():
    mu, isd, theta = _blob()
    b = jk.JkRouterBlob()
    b.magic, b.version, b.margin, b.quantile = jk.ROUTER_MAGIC, 1, 0.2, 0.9
    b.mu[:], b.isd[:], b.theta[:] = mu.tolist(), isd.tolist(), theta.tolist()
    return b


def _router_rows(case, seed):
    """Feature rows and labels with the ranges that logged quartets show."""
    rng = np.random.default_rng(31 * seed + 5)
    mu, isd, _ = _blob()
    X = mu[:12] + rng.standard_normal((case["rows"], 12)) / isd[:12]
    X[:, 10] = rng.integers(0, 5, case["rows"])
    X[:, 11] = rng.uniform(0.0, 2.0, case["rows"])
    y = -0.8 + 0.2 * X[:, 4] - 0.25 * X[:, 6] + 0.4 * rng.standard_normal(case["rows"])
    return X.astype(np.float32), np.minimum(y, 0.0).astype(np.float32)


class State:
    pass


def prepare(case, seed):
    s = State()
    s.case = case
    if case["kind"] == "router":
        X, y = _router_rows(case, seed)
        s.X, s.y = torch.tensor(X, device="cuda"), torch.tensor(y, device="cuda")
        s.blob = _jk_blob()
        return s
    mols = _molecules(case, seed)
    s.eng = jk.JK(mols)
    if case["graph"]:
        s.eng.set_option("use_graph", 1)
        s.eng.set_option("branches", 4)
    if case["omega"]:
        s.eng.set_option("omega", case["omega"])
    if case["kind"] == "spdf":
        s.eng.set_option("tau32", 3e-5)   # the threshold that f shells take
    if case["precision"] == "routed":
        s.eng.load_router(_jk_blob())
    s.D = [torch.tensor(m.D, dtype=torch.float64, device="cuda") for m in mols]
    return s


# --------------------------------------------------------------------- run
def run(state):
    case = state.case
    if case["kind"] == "router":
        f = jk.jk_router_gradient_noalloc if case["noalloc"] else jk.jk_router_gradient
        grad, loss = f(state.blob, state.X, state.y, 0.9)
        return {"grad": grad, "loss": loss}
    wj, wk = "j" in case["out"], "k" in case["out"]
    # a program that captures graphs queues its builds and looks at the error word later
    J, K, _ = state.eng.build(state.D, with_j=wj, with_k=wk, cutoff=CUTOFF, precision=case["precision"],
                              check=not case["graph"])
    out = {}
    if wj:
        out["J"] = J
    if wk:
        out["K"] = K
    return out


# ------------------------------------------------------------- work, tolerance
def _pair_counts(mol):
    """Primitive and contracted pairs per (la, lb): Gaussian estimates of the Schwarz factors, largest first."""
    sh, x = mol.shells, mol.coords
    ex, co, l, at, own = [], [], [], [], []
    for k, (a, li, n, off, _, _) in enumerate(sh):
        for i in range(n):
            ex.append(mol.exps[off + i])
            # size of the primitive where it is largest, in the units of an s function
            co.append(abs(mol.coeffs[off + i]) * (li / (2 * mol.exps[off + i]) / math.e) ** (0.5 * li) if li else abs(mol.coeffs[off + i]))
            l.append(li), at.append(a), own.append(k)
    ex, co, l, at, own = map(np.array, (ex, co, l, at, own))
    i, j = np.tril_indices(len(ex))
    p = ex[i] + ex[j]
    r2 = ((x[at[i]] - x[at[j]]) ** 2).sum(1)
    q = co[i] * co[j] * np.exp(-ex[i] * ex[j] / p * r2) * np.sqrt(2 * math.pi ** 2.5 / np.sqrt(2 * p)) / p
    key = np.maximum(l[i], l[j]) * 8 + np.minimum(l[i], l[j])
    pair = np.maximum(own[i], own[j]).astype(np.int64) * len(sh) + np.minimum(own[i], own[j])
    prim, cont = {}, {}
    for k in np.unique(key):
        m = key == k
        prim[int(k)] = np.sort(q[m])[::-1]
        u, at_ = np.unique(pair[m], return_inverse=True)
        s = np.zeros(len(u))
        np.add.at(s, at_, q[m])
        cont[int(k)] = np.sort(s)[::-1]
    return prim, cont


def _above(a, b, eps):
    """How many pairs of one value of a and one of b (both descending) have a product above eps."""
    return float(len(b) * len(a) - np.searchsorted(b[::-1], eps / np.maximum(a, 1e-300), side="right").sum())


def work(case):
    if case["kind"] == "router":
        n = case["rows"]
        return {"bytes": 4.0 * (13 * n + 2 * ROUTER_N), "flops": 6.0 * n * (12 * 64 + 64 * 64 + 64)}
    nbytes = flops = 0.0
    nc = lambda li: (li + 1) * (li + 2) // 2  # noqa: E731
    for m in _molecules(case, 1):
        ndm, d = case["ndm"], float(np.abs(m.D).max())
        nbytes += 8.0 * ndm * m.nao ** 2 * (1 + len(case["out"]))
        prim, cont = _pair_counts(m)
        keys = sorted(prim)
        for a, b in itertools.combinations_with_replacement(keys, 2):
            la, lb, lc, ld = a // 8, a % 8, b // 8, b % 8
            half = 0.5 if a == b else 1.0
            nq = half * _above(cont[a], cont[b], CUTOFF / d)
            npq = half * _above(prim[a], prim[b], CUTOFF / d)
            nr = (la + lb + lc + ld) // 2 + 1
            ne = nc(la) * nc(lb) * nc(lc) * nc(ld)
            na, ncd = la + lb + 1, lc + ld + 1
            # Rys quadrature: set-up, roots and weights, the 2D tables by recurrence, the products; then the contractions
            tables = 9.0 * na * ncd + 6.0 * ((na * lb) * ncd + (ncd * ld) * (la + 1) * (lb + 1))
            flops += npq * (30 + 40.0 * nr + nr * (tables + 3.0 * ne)) * (2 if case["omega"] < 0 else 1)
            flops += nq * ndm * 2.0 * ne * ((2 if "j" in case["out"] else 0) + (4 if "k" in case["out"] else 0))
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "router":
        return {"rel": 2e-6, "max": 8e-5}     # FP32 sums over the rows in another order
    if case["precision"] == "fp64":
        return {"rel": 2e-12, "max": 4e-11}   # the quartets below the cutoff: up to 5.5e-13 from exact()
    return {"rel": 1e-8, "max": 4e-7}         # the quartets in FP32: up to 2.3e-9 from exact()


# ------------------------------------------------------------------- exact
# McMurchie-Davidson integrals in plain torch, FP64: Hermite expansions of the primitive pairs, Hermite Coulomb integrals
# from the Boys function, contracted to the pairs of functions.
def _cart(l):
    return [(x, y, l - x - y) for x in range(l, -1, -1) for y in range(l - x, -1, -1)]


def _hermites(L):
    return [(t, u, v) for t in range(L + 1) for u in range(L + 1 - t) for v in range(L + 1 - t - u)]


def _boys(mmax, T):
    """F_0 .. F_mmax: the series and downward recursion below T = 40, the limit and upward recursion above."""
    small = T < 40.0
    Ts = torch.where(small, T, torch.zeros_like(T))
    top = float(Ts.max()) if Ts.numel() else 0.0
    eT = torch.exp(-Ts)
    term = torch.full_like(T, 1.0 / (2 * mmax + 1))
    tot = term.clone()
    for i in range(1, 30 + int(4.5 * top)):
        term = term * (2.0 * Ts / (2 * mmax + 2 * i + 1))
        tot = tot + term
        if i > top and i % 16 == 0 and float((term / tot).max()) < 1e-18:
            break
    F = [None] * (mmax + 1)
    F[mmax] = tot * eT
    for m in range(mmax - 1, -1, -1):
        F[m] = (2.0 * Ts * F[m + 1] + eT) / (2 * m + 1)
    Tl = torch.where(small, torch.full_like(T, 40.0), T)
    up, el = 0.5 * torch.sqrt(math.pi / Tl) * torch.erf(torch.sqrt(Tl)), torch.exp(-Tl)
    for m in range(mmax + 1):
        F[m] = torch.where(small, F[m], up)
        up = ((2 * m + 1) * up - el) / (2.0 * Tl)
    return F


def _hermite_coulomb(L, alpha, X, Y, Z, pref, omega):
    """R_tuv for t + u + v <= L (times pref) as a dict; omega < 0: of erfc(|omega| r) / r."""
    def base(a, scale):
        F = _boys(L, a * (X * X + Y * Y + Z * Z))
        return [scale * (-2.0 * a) ** n * F[n] for n in range(L + 1)]
    R = base(alpha, pref)
    if omega:
        w2 = omega * omega
        lr = base(alpha * w2 / (alpha + w2), pref * torch.sqrt(w2 / (alpha + w2)))
        R = [r - q for r, q in zip(R, lr)] if omega < 0 else lr
    level = {n: {(0, 0, 0): R[n]} for n in range(L + 1)}
    for s in range(1, L + 1):
        for n in range(L + 1 - s):
            for t, u, v in _hermites(s):
                if t + u + v != s:
                    continue
                up = level[n + 1]
                if t:
                    r = X * up[t - 1, u, v] + ((t - 1) * up[t - 2, u, v] if t > 1 else 0.0)
                elif u:
                    r = Y * up[t, u - 1, v] + ((u - 1) * up[t, u - 2, v] if u > 1 else 0.0)
                else:
                    r = Z * up[t, u, v - 1] + ((v - 1) * up[t, u, v - 2] if v > 1 else 0.0)
                level[n][t, u, v] = r
    return level[0]


def _hermite_expansion(la, lb, a, b, A, B):
    """E[pair, component of a x component of b, hermite] of primitive pairs with exponents a, b at A, B."""
    p = a + b
    P = (a[:, None] * A + b[:, None] * B) / p[:, None]
    E1 = []
    for ax in range(3):
        PA, PB = P[:, ax] - A[:, ax], P[:, ax] - B[:, ax]
        E = {(0, 0, 0): torch.exp(-a * b / p * (A[:, ax] - B[:, ax]) ** 2)}
        get = lambda i, j, t: E.get((i, j, t), torch.zeros_like(p)) if 0 <= t <= i + j else torch.zeros_like(p)  # noqa: E731
        for i in range(la + 1):
            for j in range(lb + 1):
                if i == j == 0:
                    continue
                for t in range(i + j + 1):
                    if i:
                        E[i, j, t] = get(i - 1, j, t - 1) / (2 * p) + PA * get(i - 1, j, t) + (t + 1) * get(i - 1, j, t + 1)
                    else:
                        E[i, j, t] = get(i, j - 1, t - 1) / (2 * p) + PB * get(i, j - 1, t) + (t + 1) * get(i, j - 1, t + 1)
        E1.append(E)
    zero = torch.zeros_like(p)
    rows = [torch.stack([E1[0].get((ca[0], cb[0], t), zero) * E1[1].get((ca[1], cb[1], u), zero) *
                         E1[2].get((ca[2], cb[2], v), zero) for t, u, v in _hermites(la + lb)], 1)
            for ca in _cart(la) for cb in _cart(lb)]
    return p, P, torch.stack(rows, 1)


def _integrals(mol, omega, dev):
    """(ij|kl) over the Cartesian functions, full array."""
    t64 = lambda v: torch.tensor(np.ascontiguousarray(v), dtype=torch.float64, device=dev)  # noqa: E731
    sh = mol.shells
    off = np.concatenate([[0], np.cumsum([len(_cart(l)) for l in sh[:, 1]])])
    groups, first = {}, 0
    for s1 in range(len(sh)):
        for s2 in range(s1 + 1):
            a, b = (s1, s2) if sh[s1, 1] >= sh[s2, 1] else (s2, s1)
            groups.setdefault((int(sh[a, 1]), int(sh[b, 1])), []).append((a, b))
    G, index = [], []
    for (la, lb), pairs in sorted(groups.items()):
        ex, own = [], []
        for k, (a, b) in enumerate(pairs):
            for i in range(sh[a, 2]):
                for j in range(sh[b, 2]):
                    ea, eb = sh[a, 3] + i, sh[b, 3] + j
                    ex.append((mol.exps[ea], mol.exps[eb], mol.coeffs[ea] * mol.coeffs[eb], sh[a, 0], sh[b, 0]))
                    own.append(k)
        ex = np.array(ex)
        A, B = t64(mol.coords[ex[:, 3].astype(int)]), t64(mol.coords[ex[:, 4].astype(int)])
        p, P, E = _hermite_expansion(la, lb, t64(ex[:, 0]), t64(ex[:, 1]), A, B)
        E = E * t64(ex[:, 2])[:, None, None]
        nf = E.shape[1]
        G.append(dict(L=la + lb, p=p, P=P, E=E, own=torch.tensor(own, device=dev), n=len(pairs), nf=nf, first=first))
        first += len(pairs) * nf
        for a, b in pairs:
            index += [(off[a] + i, off[b] + j) for i in range(len(_cart(la))) for j in range(len(_cart(lb)))]
    V = torch.zeros(first, first, dtype=torch.float64, device=dev)
    for g, h in itertools.combinations_with_replacement(G, 2):
        L, hg, hh = g["L"] + h["L"], _hermites(g["L"]), _hermites(h["L"])
        step = max(1, int(3e7 / (len(h["p"]) * max(len(_hermites(L)), len(hg) * len(hh)))))
        for i0 in range(0, len(g["p"]), step):
            sl = slice(i0, i0 + step)
            p, q = g["p"][sl, None], h["p"][None, :]
            d = g["P"][sl, None, :] - h["P"][None, :, :]
            pref = 2.0 * math.pi ** 2.5 / (p * q * torch.sqrt(p + q))
            R = _hermite_coulomb(L, p * q / (p + q), d[..., 0], d[..., 1], d[..., 2], pref, omega)
            # [ket hermite] contracted to the ket functions, then the bra
            half = []
            for t, u, v in hg:
                K = torch.stack([(-1.0) ** (a + b + c) * R[t + a, u + b, v + c] for a, b, c in hh], 2)
                K = torch.einsum("pqh,qfh->pqf", K, h["E"])
                half.append(torch.zeros(K.shape[0], h["n"], h["nf"], dtype=K.dtype, device=dev).index_add_(1, h["own"], K))
            full = torch.einsum("hpkf,peh->pekf", torch.stack(half), g["E"][sl])
            full = full.reshape(full.shape[0], g["nf"], -1)
            blk = V[g["first"]:g["first"] + g["n"] * g["nf"], h["first"]:h["first"] + h["n"] * h["nf"]]
            acc = torch.zeros(g["n"], g["nf"], h["n"] * h["nf"], dtype=torch.float64, device=dev)
            acc.index_add_(0, g["own"][sl], full)
            blk += acc.reshape(g["n"] * g["nf"], -1)
        if g is not h:
            a, b = (g["first"], g["n"] * g["nf"]), (h["first"], h["n"] * h["nf"])
            V[b[0]:b[0] + b[1], a[0]:a[0] + a[1]] = V[a[0]:a[0] + a[1], b[0]:b[0] + b[1]].T
    n = int(off[-1])
    at = np.zeros((n, n), dtype=np.int64)
    for k, (i, j) in enumerate(index):
        at[i, j] = at[j, i] = k
    at = torch.tensor(at.reshape(-1), device=dev)
    return V[at][:, at].reshape(n, n, n, n)


def _solid_harmonics(l):
    """Cartesian components x (2l+1) real solid harmonics, m = -l .. l (p: x, y, z), each with the norm of x^l."""
    if l < 2:
        return np.eye(2 * l + 1)
    comp = {c: i for i, c in enumerate(_cart(l))}
    f, C = math.factorial, np.zeros((len(comp), 2 * l + 1))
    for m in range(-l, l + 1):
        am, odd = abs(m), int(m < 0)
        N = math.sqrt(2.0 * f(l + am) * f(l - am) / (2.0 if m == 0 else 1.0)) / (2.0 ** am * f(l))
        for t in range((l - am) // 2 + 1):
            for u in range(t + 1):
                for k in range(odd, am + 1, 2):
                    c = (-1.0) ** (t + (k - odd) // 2) * 0.25 ** t * math.comb(l, t) * math.comb(l - t, am + t) * \
                        math.comb(t, u) * math.comb(am, k)
                    C[comp[2 * t + am - 2 * u - k, 2 * u + k, l - 2 * t - am], m + l] += N * c
    return C


def _bf16(v):
    return v.to(torch.bfloat16).to(torch.float64)


def _exact_router(case, seed):
    """Mean pinball loss and its gradient: BF16 weights and layer inputs, everything else in FP64."""
    X, y = (torch.tensor(v) for v in _router_rows(case, seed))
    mu, isd, th = (torch.tensor(v) for v in _blob())
    x = _bf16((X - mu[:12]) * isd[:12])
    w1, w2, w3 = _bf16(th[:768].view(12, 64)), _bf16(th[1088:5184].view(64, 64)), _bf16(th[5248:5312])
    b1, b2, b3 = th[1024:1088].double(), th[5184:5248].double(), th[5312].double()
    a1 = x @ w1 + b1
    h1 = _bf16(torch.relu(a1).float())
    a2 = h1 @ w2 + b2
    h2 = _bf16(torch.relu(a2).float())
    u = y.double() - (h2 @ w3 + b3)
    loss = torch.where(u >= 0, 0.9 * u, -0.1 * u).mean()
    g = ((u < 0).double() - 0.9) / len(u)
    d2 = g[:, None] * w3 * (a2 > 0)
    d1 = (d2 @ w2.T) * (a1 > 0)
    grad = torch.zeros(ROUTER_N, dtype=torch.float64)
    grad[:768], grad[1024:1088] = (x.T @ d1).reshape(-1), d1.sum(0)
    grad[1088:5184], grad[5184:5248] = (h1.T @ d2).reshape(-1), d2.sum(0)
    grad[5248:5312], grad[5312] = h2.T @ g, g.sum()
    return {"grad": grad.numpy(), "loss": float(loss)}


def exact(case, seed):
    if case["kind"] == "router":
        return _exact_router(case, seed)
    mols = _molecules(case, seed)
    if len(mols) > 1 or mols[0].nao_cart > 190:
        return None
    mol, dev = mols[0], "cuda" if torch.cuda.is_available() else "cpu"
    V = _integrals(mol, case["omega"], dev)
    C = torch.tensor(_block_diag([_solid_harmonics(l) if s else np.eye(len(_cart(l)))
                                  for l, s in zip(mol.shells[:, 1], mol.shells[:, 5])]), device=dev)
    J, K = [], []
    for d in torch.tensor(mol.D, device=dev):
        d = C @ d @ C.T
        J.append(C.T @ torch.einsum("ijkl,kl->ij", V, d) @ C)
        K.append(C.T @ torch.einsum("ijkl,jl->ik", V, d) @ C)
    out = {}
    if "j" in case["out"]:
        out["J"] = [torch.stack(J)]
    if "k" in case["out"]:
        out["K"] = [torch.stack(K)]
    return out


def _block_diag(blocks):
    n, m = sum(b.shape[0] for b in blocks), sum(b.shape[1] for b in blocks)
    C, i, j = np.zeros((n, m)), 0, 0
    for b in blocks:
        C[i:i + b.shape[0], j:j + b.shape[1]] = b
        i, j = i + b.shape[0], j + b.shape[1]
    return C
