"""The work that users of this library have it do, as measurable cases.

A case names a batch of shell quartets: its classes (letters of the four angular momenta, or a
mix), its number of quartets, the contraction degrees, the output kind, the path and the form of
the call.  The classes and contraction degrees of a batch follow from the case alone, so that
its work is the same for every seed; centers, exponents and coefficients follow from the seed.
"""
import math

import numpy as np
import torch

from paper_2307_03452_gb300 import lx
from paper_2307_03452_gb300.router import Router

LETTERS = "spdfghik"
MIXED = ["gggg", "hhhh", "iiii", "ghii", "gihh"]


def listed():
    return [
        # the smallest call of earnest use: one class of 64 uncontracted quartets
        {"name": "gggg_64", "form": "batch", "cls": "gggg", "n": 64, "kmin": 1, "kmax": 1, "path": "fp64", "solid": True,
         "cube": 10.0, "emin": 0.1, "emax": 10.0},
        # a handful of quartets left over from a screened list, Cartesian output
        {"name": "few_mixed_cart", "form": "batch", "cls": "mixed", "n": 7, "kmin": 1, "kmax": 2, "path": "fp64",
         "solid": False, "cube": 6.0, "emin": 0.05, "emax": 50.0},
        # low angular momentum, deep contraction: the low end of the class sweep
        {"name": "dddd_contracted", "form": "batch", "cls": "dddd", "n": 8191, "kmin": 1, "kmax": 5, "path": "fp64",
         "solid": True, "cube": 20.0, "emin": 0.05, "emax": 20.0},
        # the headline class on the FP64 path, solid output
        {"name": "iiii_fp64", "form": "batch", "cls": "iiii", "n": 2048, "kmin": 1, "kmax": 1, "path": "fp64",
         "solid": True, "cube": 20.0, "emin": 0.05, "emax": 20.0},
        # the same class in Cartesian functions (28^4 per quartet)
        {"name": "iiii_cart", "form": "batch", "cls": "iiii", "n": 200, "kmin": 1, "kmax": 1, "path": "fp64",
         "solid": False, "cube": 20.0, "emin": 0.05, "emax": 20.0},
        # mixed classes and contraction degrees in one call
        {"name": "mixed_fp64", "form": "batch", "cls": "mixed", "n": 200, "kmin": 1, "kmax": 5, "path": "fp64",
         "solid": True, "cube": 20.0, "emin": 0.05, "emax": 50.0},
        # the headline class on the tensor-core path, at its full size
        {"name": "iiii_split", "form": "batch", "cls": "iiii", "n": 4096, "kmin": 1, "kmax": 1, "path": "split",
         "solid": True, "cube": 20.0, "emin": 0.05, "emax": 20.0},
        # two contracted classes on the tensor-core path
        {"name": "hhhh_iiii_split", "form": "batch", "cls": "hhhh+iiii", "n": 768, "kmin": 1, "kmax": 3, "path": "split",
         "solid": True, "cube": 20.0, "emin": 0.05, "emax": 20.0},
        # l = 4..6, K = 1..5, magnitudes over many decades, each quartet routed by the network
        {"name": "routed", "form": "batch", "cls": "spread", "n": 500, "kmin": 1, "kmax": 5, "path": "routed",
         "solid": True, "cube": 30.0, "emin": 0.05, "emax": 50.0},
        # bra list x ket list, as an integral engine is driven
        {"name": "iiii_pairs_split", "form": "pairs", "cls": "iiii", "n": 4096, "kmin": 1, "kmax": 1, "path": "split",
         "solid": True, "cube": 20.0, "emin": 0.05, "emax": 20.0},
        # Coulomb and exchange matrices of a Fock build from quartets of one shell set
        {"name": "iiii_jk", "form": "jk", "cls": "iiii", "n": 501, "kmin": 1, "kmax": 1, "path": "fp64", "solid": True,
         "cube": 8.0, "emin": 0.05, "emax": 20.0},
        # a batch planned once and replayed as a graph
        {"name": "mixed_graph", "form": "graph", "cls": "mixed", "n": 300, "kmin": 1, "kmax": 3, "path": "split",
         "solid": True, "cube": 20.0, "emin": 0.05, "emax": 50.0},
    ]


def draw(rng):
    """Another case of the same ranges: d to k shells, K = 1..5, every form and path."""
    while True:
        form = rng.choice(["batch", "batch", "batch", "batch", "pairs", "jk", "graph"])
        path = rng.choice(["fp64", "fp64", "fp64", "split", "split4", "split5", "routed"])
        if form == "graph" and path == "routed":  # graphs take one path
            path = "fp64"
        cls = rng.choice(["one", "one", "any", "pair", "mixed", "spread"])
        if form == "pairs" and cls not in ("one", "pair"):
            cls = "pair"
        if cls == "one":
            cls = rng.choice("dfghik") * 4
        elif cls == "pair":
            cls = rng.choice("dfghik") + rng.choice("dfghik") + rng.choice("dfghik") + rng.choice("dfghik")
        kmin = rng.choice([1, 1, 1, 2])
        case = {"form": form, "cls": cls, "n": int(round(math.exp(rng.uniform(math.log(5), math.log(6000))))),
                "kmin": kmin, "kmax": rng.randint(kmin, rng.choice([1, 2, 3, 5]) if kmin == 1 else 5), "path": path,
                "solid": rng.random() < 0.75, "cube": rng.choice([6.0, 10.0, 20.0]), "emin": 0.05,
                "emax": rng.choice([10.0, 20.0, 50.0])}
        w = work(case)
        # no more than the largest listed case: time on the case's path, output kept in memory
        if path == "fp64" and w["flops"] > 4.0e11 or w["flops"] > 8.0e11 or w["bytes"] > 1.0e9:
            continue
        return case


# ------------------------------------------------------------------ shapes and inputs


def _nf(l, solid):
    return 2 * l + 1 if solid else (l + 1) * (l + 2) // 2


def _pyr(n):
    return (n + 1) * (n + 2) * (n + 3) // 6


def _shape(case):
    """(l, K, quartets): per-shell angular momenta and degrees and the quartet list, from the
    case alone.  Pairs: also the two pair lists."""
    r = np.random.default_rng([int(case["n"]), int(case["kmin"]), int(case["kmax"]), sum(map(ord, case["cls"]))])
    n, cls = int(case["n"]), case["cls"]
    if case["form"] == "pairs":
        nb = max(1, int(round(math.sqrt(n))))
        nk = max(1, n // nb)
        l = np.array([LETTERS.index(c) for c in cls[:2] * nb + cls[2:] * nk])
        bra = np.arange(2 * nb, dtype=np.int32).reshape(-1, 2)
        ket = (2 * nb + np.arange(2 * nk, dtype=np.int32)).reshape(-1, 2)
        q = np.concatenate([np.repeat(bra, nk, axis=0), np.tile(ket, (nb, 1))], axis=1)
        k = r.integers(case["kmin"], case["kmax"] + 1, len(l))
        return l, k, q.astype(np.int32), bra, ket
    if case["form"] == "jk":  # quartets over one set of shells, as a Fock build lists them
        if cls in ("mixed", "any", "spread"):
            l = r.integers(2 if cls == "any" else 4, 8 if cls == "any" else 7, 16)
        else:
            one = cls.split("+")[0]
            l = np.array([LETTERS.index(c) for c in one * 4])
        q = r.integers(0, len(l), (n, 4))
        if cls not in ("mixed", "any", "spread"):
            q = 4 * (q // 4) + np.arange(4)[None, :]  # the class's own order of shells
        return l, r.integers(case["kmin"], case["kmax"] + 1, len(l)), q.astype(np.int32), None, None
    if cls == "mixed":
        l = np.array([[LETTERS.index(c) for c in MIXED[i]] for i in r.integers(0, len(MIXED), n)]).reshape(-1)
    elif cls == "spread":
        l = r.integers(4, 7, 4 * n)
    elif cls == "any":
        l = r.integers(2, 8, 4 * n)
    else:
        names = cls.split("+")
        l = np.array([LETTERS.index(c) for i in range(n) for c in names[i % len(names)]])
    k = r.integers(case["kmin"], case["kmax"] + 1, 4 * n)
    return l, k, np.arange(4 * n, dtype=np.int32).reshape(n, 4), None, None


def _inputs(case, seed):
    """(basis, quartets, bra pairs, ket pairs, density): shells of the case with centers and
    exponents of the seed -- uniform in a cube, log-uniform; "spread": the two centers of a pair
    close together, bra and ket up to 30 bohr apart."""
    l, k, q, bra, ket = _shape(case)
    r = np.random.default_rng([seed, 77])
    ns = len(l)
    if case["cls"] == "spread" and case["form"] != "jk":
        n = ns // 4
        base, d = r.uniform(0.0, 20.0, (n, 1, 3)), r.normal(size=(n, 1, 3))
        far = base + d / np.linalg.norm(d, axis=2, keepdims=True) * r.uniform(0.0, case["cube"], (n, 1, 1))
        u = r.normal(size=(n, 4, 3))
        u *= r.uniform(0.0, 3.0, (n, 4, 1)) / np.linalg.norm(u, axis=2, keepdims=True)
        centers = (np.concatenate([base, base, far, far], axis=1) + u).reshape(-1, 3)
    else:
        centers = r.uniform(0.0, case["cube"], (ns, 3))
    off = np.zeros(ns, dtype=np.int32)
    off[1:] = np.cumsum(k)[:-1]
    npr = int(k.sum())
    exps = np.exp(r.uniform(math.log(case["emin"]), math.log(case["emax"]), npr))
    coefs = 1.0 - r.uniform(0.0, 1.0, npr) if case["kmax"] > 1 else np.ones(npr)
    basis = {"l": l.astype(np.int32), "nprim": k.astype(np.int32), "prim_off": off, "center": centers, "exps": exps,
             "coefs": coefs}
    dens = None
    if case["form"] == "jk":
        nbf = int(sum(_nf(int(x), case["solid"]) for x in l))
        dens = r.normal(size=(nbf, nbf))
        dens = dens + dens.T
    return basis, q, bra, ket, dens


def prepare(case, seed):
    basis, q, bra, ket, dens = _inputs(case, seed)
    solid, path = case["solid"], case["path"]
    st = {"form": case["form"]}
    if path == "routed":
        router = Router.load()
        lx.router_set(router.p16, router.tau)
    if case["form"] == "pairs":
        b = lx.PairBatch(basis, bra, ket, solid, path=path)
    elif case["form"] == "jk":
        b = lx.JKBatch(basis, q, solid, path=path)
        st["D"] = torch.tensor(dens, device="cuda")
        st["J"], st["K"] = torch.empty_like(st["D"]), torch.empty_like(st["D"])
    else:
        b = lx.Batch(basis, q, solid, path=path)
    st["b"] = b
    st["ws"] = lx.alloc_workspace(max(min(b.workspace_size(), 48 << 30), b.workspace_min()))
    if case["form"] != "jk":
        st["out"] = torch.empty(b.out_size, dtype=torch.float64, device="cuda")
    if case["form"] == "graph":
        st["graph"] = lx.Graph(b, st["out"], st["ws"])
    return st


def run(state):
    if state["form"] == "jk":
        state["J"].zero_()
        state["K"].zero_()
        state["b"].run_jk(state["D"], state["J"], state["K"], state["ws"])
        return {"J": state["J"], "K": state["K"]}
    if state["form"] == "graph":
        state["graph"].launch()
    else:
        state["b"].run(state["out"], state["ws"])
    return state["out"]


def work(case):
    """Bytes: shells, primitives and quartets read once, integrals (or J, K and D) once.  FLOPs:
    the two transforms in matrix form, 2 N_ab (K_bra N_p) (K_ket N_q) + 2 N_ab (K_ket N_q) N_cd
    per quartet, which is what the framework's FP64-equivalent rates are quoted in."""
    l, k, q, _, _ = _shape(case)
    l, k = l.astype(np.float64), k.astype(np.float64)
    nf = 2 * l + 1 if case["solid"] else (l + 1) * (l + 2) / 2
    pyr = lambda n: (n + 1) * (n + 2) * (n + 3) / 6  # noqa: E731
    a, b, c, d = q.T
    nab, ncd = nf[a] * nf[b], nf[c] * nf[d]
    k1, k2 = k[a] * k[b] * pyr(l[a] + l[b]), k[c] * k[d] * pyr(l[c] + l[d])
    flops = float((2 * nab * k1 * k2 + 2 * nab * k2 * ncd).sum())
    out = 3 * 8 * nf.sum() ** 2 if case["form"] == "jk" else 8 * (nab * ncd).sum()
    return {"bytes": float(out + 40 * len(l) + 16 * k.sum() + 24 * len(q)), "flops": flops}


# ------------------------------------------------------------------ the same numbers, plainly


def _boys(mmax, t):
    """F_0..F_mmax(t) in float64: series and downward recursion up to t = 40, then upward."""
    small = t.clamp(max=40.0)
    term = torch.full_like(t, 1.0 / (2 * mmax + 1))
    s = term.clone()
    for i in range(1, 200):
        term = term * (2.0 * small / (2 * mmax + 2 * i + 1))
        s = s + term
    lo = [None] * (mmax + 1)
    e = torch.exp(-small)
    lo[mmax] = e * s
    for m in range(mmax - 1, -1, -1):
        lo[m] = (2.0 * small * lo[m + 1] + e) / (2 * m + 1)
    big = t.clamp(min=40.0)
    hi = [0.5 * torch.sqrt(math.pi / big) * torch.erf(torch.sqrt(big))]
    eb = torch.exp(-big)
    for m in range(mmax):
        hi.append(((2 * m + 1) * hi[m] - eb) / (2.0 * big))
    return torch.stack([torch.where(t < 40.0, x, y) for x, y in zip(lo, hi)], dim=-1)


def _triplets(lmax):
    return [(n - i, i - v, v) for n in range(lmax + 1) for i in range(n + 1) for v in range(i + 1)]


_solid_cache = {}


def _solid(l):
    """Real solid harmonics (2l+1) x ncart(l) over x^l-normalised Cartesians, by projecting the
    harmonic polynomials Re, Im (x + iy)^m times their even series in z."""
    if l in _solid_cache:
        return _solid_cache[l]
    comps = {(l - i, i - j, j): c for c, (i, j) in enumerate((i, j) for i in range(l + 1) for j in range(i + 1))}
    c = np.zeros((2 * l + 1, len(comps)))
    for m in range(l + 1):
        lead = math.sqrt((2.0 - (m == 0)) * math.factorial(l - m) / math.factorial(l + m)) * math.factorial(l + m) / (
            2.0 ** m * math.factorial(m) * math.factorial(l - m))
        for j in range((l - m) // 2 + 1):
            for p in range(j + 1):  # (x^2 + y^2)^j
                for s in range(m + 1):  # (x + iy)^m
                    w = lead * math.comb(j, p) * math.comb(m, s)
                    key = (m - s + 2 * (j - p), s + 2 * p, l - m - 2 * j)
                    if s % 2 == 0:
                        c[l + m, comps[key]] += w * (-1.0) ** (s // 2)
                    elif m:
                        c[l - m, comps[key]] += w * (-1.0) ** (s // 2)
            if l - m - 2 * j >= 2:
                lead *= -(l - m - 2 * j) * (l - m - 2 * j - 1) / (4.0 * (j + 1) * (j + 1 + m))
    _solid_cache[l] = torch.tensor(c, device="cuda")
    return _solid_cache[l]


def _dfact(l):
    return float(np.prod(np.arange(2 * l - 1, 0, -2))) if l else 1.0


def _hermite(l1, l2, z1, z2, c1, c2, r1, r2, solid, sign):
    """H of shell pairs: z, c (G, K) exponents and normalised coefficients, r (G, 3) centers ->
    H (G, K1 K2, nf nf, pyr), zeta and P of every primitive pair."""
    za, zb = z1[:, :, None].expand(-1, -1, z2.shape[1]).flatten(1), z2[:, None, :].expand(-1, z1.shape[1], -1).flatten(1)
    cc = (c1[:, :, None] * c2[:, None, :]).flatten(1)
    zp = za + zb
    d = r1 - r2
    pre = cc * torch.exp(-za * zb / zp * (d * d).sum(1, keepdim=True))
    p = (za[..., None] * r1[:, None] + zb[..., None] * r2[:, None]) / zp[..., None]
    nt = l1 + l2 + 1
    e = torch.zeros(*za.shape, 3, l1 + 1, l2 + 1, nt + 2, dtype=torch.float64, device=za.device)
    e[..., 0, 0, 1] = 1.0  # the t index is stored one up
    pa, pb = p - r1[:, None], p - r2[:, None]
    tt = torch.arange(1, nt + 1, dtype=torch.float64, device=za.device)

    def up(prev, x):
        return 0.5 / zp[..., None, None] * prev[..., :-2] + x[..., None] * prev[..., 1:-1] + tt * prev[..., 2:]

    for i in range(l1 + 1):
        if i:
            e[..., i, 0, 1:-1] = up(e[..., i - 1, 0, :], pa)
        for j in range(1, l2 + 1):
            e[..., i, j, 1:-1] = up(e[..., i, j - 1, :], pb)
    e = e[..., 1:-1]
    trip = torch.tensor(_triplets(l1 + l2), device=za.device)
    c_a = [(l1 - i, i - j, j) for i in range(l1 + 1) for j in range(i + 1)]
    c_b = [(l2 - i, i - j, j) for i in range(l2 + 1) for j in range(i + 1)]
    ia, ib = torch.tensor(c_a, device=za.device), torch.tensor(c_b, device=za.device)
    h = pre[..., None, None, None]
    for x in range(3):
        h = h * e[:, :, x][:, :, ia[:, x]][:, :, :, ib[:, x]][..., trip[:, x]]
    if solid:
        h = torch.einsum("ma,gkabp->gkmbp", _solid(l1), h)
        h = torch.einsum("nb,gkmbp->gkmnp", _solid(l2), h)
    if sign:
        h = h * (1.0 - 2.0 * (trip.sum(1) % 2).double())
    return h.flatten(2, 3), zp, p


def _norm(l, z, c):
    """Coefficients of unit-normalised contracted shells, z and c (G, K)."""
    n = c * (2.0 * z / math.pi) ** 0.75 * (4.0 * z) ** (0.5 * l) / math.sqrt(_dfact(l))
    s = z[:, :, None] + z[:, None, :]
    ov = _dfact(l) / (2.0 * s) ** l * (math.pi / s) ** 1.5
    return n / torch.sqrt((n[:, :, None] * n[:, None, :] * ov).sum((1, 2)))[:, None]


def _blocks(ls, z, c, r, solid):
    """(ab|cd) blocks (G, nab, ncd) of G quartets of one class and one set of degrees."""
    la, lb, lc, ld = ls
    c = [_norm(ls[i], z[i], c[i]) for i in range(4)]
    hb, zp, p = _hermite(la, lb, z[0], z[1], c[0], c[1], r[0], r[1], solid, False)
    hk, zq, qc = _hermite(lc, ld, z[2], z[3], c[2], c[3], r[2], r[3], solid, True)
    L, dev = sum(ls), zp.device
    trip = _triplets(L)
    pos = {t: i for i, t in enumerate(trip)}
    s1, s2, dr, cf = [0], [0], [0], [0.0]
    for t in trip[1:]:
        x = next(i for i in range(3) if t[i])
        one = tuple(t[i] - (i == x) for i in range(3))
        two = tuple(t[i] - 2 * (i == x) for i in range(3))
        s1.append(pos[one]); s2.append(pos.get(two, 0)); dr.append(x); cf.append(t[x] - 1.0)
    s1, s2, dr = (torch.tensor(v, device=dev) for v in (s1, s2, dr))
    cf = torch.tensor(cf, dtype=torch.float64, device=dev)
    tp, tq = _triplets(la + lb), _triplets(lc + ld)
    idx = torch.tensor([[pos[(a[0] + b[0], a[1] + b[1], a[2] + b[2])] for b in tq] for a in tp], device=dev)
    g, kb, kk = zp.shape[0], zp.shape[1], zq.shape[1]
    a, b = zp[:, :, None].expand(g, kb, kk).reshape(-1), zq[:, None, :].expand(g, kb, kk).reshape(-1)
    pq = (p[:, :, None] - qc[:, None, :]).reshape(-1, 3)
    rho = a * b / (a + b)
    f = _boys(L, rho * (pq * pq).sum(1)) * (2.0 * math.pi ** 2.5 / (a * b * torch.sqrt(a + b)))[:, None]
    f = f * (-2.0 * rho)[:, None] ** torch.arange(L + 1, device=dev)
    cur = f[:, L:L + 1]
    for m in range(L - 1, -1, -1):
        n = _pyr(L - m)
        w = pq[:, dr[:n]] * cur[:, s1[:n].clamp(max=cur.shape[1] - 1)]
        w = w + cf[:n] * cur[:, s2[:n].clamp(max=cur.shape[1] - 1)]
        w[:, 0] = f[:, m]
        cur = w
    cur = cur.view(g, kb, kk, -1)
    hb = hb.transpose(1, 2).flatten(2)  # (G, nab, K_bra N_p)
    out = 0.0
    for j in range(kk):
        r = cur[:, :, j][:, :, idx.reshape(-1)].reshape(g, kb * idx.shape[0], idx.shape[1])
        out = out + (hb @ r) @ hk[:, j].transpose(1, 2)
    return out


def exact(case, seed):
    """The integrals (or J and K) by the plain McMurchie-Davidson sums in float64 torch."""
    if work(case)["flops"] > (1.0e12 if case["solid"] else 3.0e11):
        return None
    basis, q, _, _, dens = _inputs(case, seed)
    solid, l, k = case["solid"], basis["l"], basis["nprim"]
    groups = {}
    for i, s in enumerate(q):
        groups.setdefault((tuple(int(x) for x in l[s]), tuple(int(x) for x in k[s])), []).append(i)
    sizes = np.array([np.prod([_nf(int(x), solid) for x in l[s]]) for s in q], dtype=np.int64)
    off = np.concatenate([[0], np.cumsum(sizes)])
    out = torch.zeros(int(off[-1]), dtype=torch.float64, device="cuda")
    dev = lambda v: torch.tensor(np.asarray(v), dtype=torch.float64, device="cuda")  # noqa: E731
    for (ls, ks), idx in groups.items():
        kb, kk, nb, nk = ks[0] * ks[1], ks[2] * ks[3], _pyr(ls[0] + ls[1]), _pyr(ls[2] + ls[3])
        big = max(kb * _nf(ls[0], False) * _nf(ls[1], False) * nb, kk * _nf(ls[2], False) * _nf(ls[3], False) * nk,
                  kb * nb * nk, kb * kk * _pyr(sum(ls)))
        step = max(1, int(1.0e8 / big))
        for at in range(0, len(idx), step):
            part = np.asarray(idx[at:at + step])
            z = [dev([basis["exps"][basis["prim_off"][s]:basis["prim_off"][s] + kk] for s in q[part, c]]) for c, kk in enumerate(ks)]
            cf = [dev([basis["coefs"][basis["prim_off"][s]:basis["prim_off"][s] + kk] for s in q[part, c]]) for c, kk in enumerate(ks)]
            r = [dev(basis["center"][q[part, c]]) for c in range(4)]
            blk = _blocks(ls, z, cf, r, solid).flatten(1)
            out[torch.tensor(off[part], device="cuda")[:, None] + torch.arange(blk.shape[1], device="cuda")] = blk
    if case["form"] != "jk":
        return out
    nf = np.array([_nf(int(x), solid) for x in l])
    bf = np.concatenate([[0], np.cumsum(nf)])
    D = dev(dens)
    J, K = torch.zeros_like(D), torch.zeros_like(D)
    for i, (a, b, c, d) in enumerate(q):
        v = out[off[i]:off[i + 1]].view(*(int(nf[x]) for x in (a, b, c, d)))
        sl = [slice(int(bf[x]), int(bf[x + 1])) for x in (a, b, c, d)]
        J[sl[0], sl[1]] += torch.einsum("mnls,ls->mn", v, D[sl[2], sl[3]])
        K[sl[0], sl[2]] += torch.einsum("mnls,ns->ml", v, D[sl[1], sl[3]])
    return {"J": J, "K": K}
